"""The packed prompt pass of the bfloat16 path (prompts back to back, at most 768 tokens a pass) against the oracle, in lock-step."""
import pytest
import torch

from synth import load_tree, make_prompts, make_weights
from synth.configs import ModelCfg, HeadCfg
from tests.test_gpu_step import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,kv_planes,lens", [
    (128, 2, [512]), (128, 2, [513]), (128, 2, [768]), (128, 2, [769]), (128, 2, [1600]),      # up to one full pass; one row more; several passes
    (128, 2, [700, 67, 1]), (128, 2, [700, 67, 1, 1]), (128, 1, [500, 300, 12, 800]),
    (128, 2, [300, 211, 1, 1, 130, 64]), (128, 1, [500, 12, 1]),         # passes that end inside, at the end of and just after a sequence
    (64, 2, [129, 383, 127]), (64, 1, [1, 511, 2])])
def test_packed_prompt_passes(head_dim, kv_planes, lens):
    m = ModelCfg(2, 256, 256 // head_dim, head_dim, 512, 1024, dtype="bf16", kv_planes=kv_planes)
    st, _ = run(m, HeadCfg(3, 1, True), load_tree("tree15_d3"), lens, 2, 33, max(lens) + 40, kv_layers=(0, 1))
    assert st.steps == 2


@pytest.mark.parametrize("rows", [16, 17, 40, 41, 96, 97])
@pytest.mark.parametrize("d_model", [256, 1280])
def test_row_counts_around_the_norm_clusters(rows, d_model):
    """A pass of few rows shares each row's norm among 8, 4 or 2 CTAs of a cluster, one of many rows does not: the prompt passes at the edges."""
    m = ModelCfg(1, d_model, d_model // 128, 128, 512, 1024, dtype="bf16")
    st, _ = run(m, HeadCfg(1, 1, True), [-1, 0], [rows], 1, 34, rows + 16, kv_layers=(0,))
    assert st.steps == 1


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_offsets_may_begin_anywhere_in_the_token_buffer(dtype):
    """The first offset need not be 0 (prompts inside a larger token buffer): the same root, lengths, hidden rows and caches."""
    import ctypes as C
    from paper_2402_05109_b200 import Hydra
    from paper_2402_05109_b200.binding import lib, _stream
    m = ModelCfg(2, 256, 2, 128, 512, 1024, dtype=dtype)
    w = {k: v.cuda() for k, v in make_weights(m, HeadCfg(2, 1, True), 35).items()}
    prompts = make_prompts(35, [70, 1, 900], m.vocab)
    toks = torch.cat([p.to(torch.int32).flatten() for p in prompts])
    outs = []
    for lead in (0, 5, 777):
        g = Hydra(m, HeadCfg(2, 1, True), [-1, 0, 1], w, 3, 960)
        buf = torch.cat([torch.full((lead,), 1 << 30, dtype=torch.int32), toks]).cuda()       # what lies ahead is no token
        offs = [lead]
        for p in prompts:
            offs.append(offs[-1] + p.numel())
        g.batch = 3
        assert lib.hydra_prefill(g._ctx, 3, buf.data_ptr(), (C.c_int32 * 4)(*offs), _stream()) == 0
        g.poll_status()
        outs.append([g.get_buffer(n).cpu().clone() for n in ("ROOT_TOK", "LEN", "N_NEW", "H_NEW", "KV_BASE", "KV_PREFIX")])
        g.close()
    for other in outs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(outs[0], other))
