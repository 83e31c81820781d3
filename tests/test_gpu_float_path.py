"""Float path: products with what follows them, in both forms (a warp per column, 32 x 32 tiles) and at their edges, over whole steps against the oracle."""
import pytest
import torch

from synth import load_tree
from synth.configs import ModelCfg, HeadCfg
from tests.test_gpu_step import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,head,tree,lens", [
    # widths that are no multiple of a tile (32) or a stage (64 k); rows of 1, 3, 15, 48 and, in a prompt chunk, 192
    ((2, 192, 3, 64, 340, 644), (3, 1, False), "tree15_d3", [70, 1, 33]),
    # two warps a pair of columns (d above 256), tiles in all products of 5 x 64 rows, prefix layer, three-layer heads
    ((2, 512, 4, 128, 1000, 1028), (4, 3, True), "tree63_d4", [70, 20, 64, 9, 65]),
    # draft rows (33 and 30) in tiles, blocks of the gathered rows across their stages
    ((1, 2112, 33, 64, 132, 512), (4, 2, False), "tree63_d4", [5, 9, 20]),
    # Medusa heads
    ((2, 256, 2, 128, 688, 2052), (4, 2, False, True, True), "tree15_d3", [17, 40]),
])
def test_steps_against_the_oracle(model, head, tree, lens):
    st, _ = run(ModelCfg(*model, dtype="fp32"), HeadCfg(*head), load_tree(tree), lens, 3, 83, 160, norm_gain_std=0.1)
    assert st.steps == 3
    # rounded at 24 bits: each product and norm adds about 1e-7, and a layer amplifies what comes in by a small factor (heads: several times a layer)
    assert st.max_hidden_err < 2e-5 and st.max_logit_err < 1e-3 and st.max_hprime_err < 1e-4


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_prompt_pass_is_refused_under_stream_capture(dtype):
    """The float path copies nothing from host memory and waits for nothing, but a prompt pass still belongs to one call."""
    import ctypes as C
    from paper_2402_05109_b200 import Hydra
    from paper_2402_05109_b200.binding import lib, _stream
    from synth import make_prompts, make_weights
    m, h = ModelCfg(2, 256, 2, 128, 512, 1024, dtype=dtype), HeadCfg(3, 1, False)
    g = Hydra(m, h, load_tree("tree15_d3"), {k: v.cuda() for k, v in make_weights(m, h, 7).items()}, 1, 128)
    toks, offs = make_prompts(7, [40], m.vocab)[0].to(torch.int32).cuda(), (C.c_int32 * 2)(0, 40)
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        x += 1
        assert lib.hydra_prefill(g._ctx, 1, toks.data_ptr(), offs, _stream()) != 0
    graph.replay()
    g.prefill([toks])
    assert g.get_buffer("LEN")[0].item() == 40 and x[0].item() == 1
    g.close()
