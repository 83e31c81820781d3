"""hydra_verify replays a captured graph from the eighth call of a batch on a stream of the caller's own: other candidates, other result buffers, other
prompt lengths and batches give bit for bit what launching kernel by kernel gives."""
import pytest
import torch

from synth import load_tree, make_prompts, make_weights
from synth.configs import ModelCfg, HeadCfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("typical", [False, True])
def test_replay_matches_launches(dtype, typical):
    from paper_2402_05109_b200 import Hydra
    m = ModelCfg(2, 256, 2, 128, 512, 1024, dtype=dtype)
    h = HeadCfg(3, 1, False)
    w = {k: v.cuda() for k, v in make_weights(m, h, 91).items()}
    parent = load_tree("tree15_d3")
    outs = []
    for graph in (False, True):
        g = Hydra(m, h, parent, w, 3, 1100)
        g.set_step_graph(graph)
        if typical:
            g.set_acceptance(1, tau=0.7, eps=0.1, alpha=0.3)
        got = []
        with torch.cuda.stream(torch.cuda.Stream()):
            gen = torch.Generator().manual_seed(5)
            for lens in ([70, 33], [70, 33, 1], [20, 9], [600, 1]):        # the last one needs another attention grid
                g.prefill([p.cuda() for p in make_prompts(91, lens, m.vocab)])
                for want in (True, True, False) * 3:
                    cand = torch.randint(0, m.vocab, (len(lens), len(parent)), dtype=torch.int32, generator=gen).cuda()
                    res = g.verify(cand, want_logits=want)
                    amax = res[0] if want else res
                    got += [r.clone() for r in (res if want else [res])]
                n_acc, _, out = g.accept_compact(cand, amax)
                got += [n_acc.clone(), out.clone(), g.get_buffer("LEN").clone(), g.get_buffer("H_NEW").clone()]
        torch.cuda.synchronize()
        g.poll_status()
        outs.append([t.cpu() for t in got])
        g.close()
    assert all(torch.equal(a, b) for a, b in zip(*outs))


def test_inside_a_capture_of_the_caller():
    from paper_2402_05109_b200 import Hydra
    m = ModelCfg(2, 256, 2, 128, 512, 1024, dtype="bf16")
    h = HeadCfg(3, 1, False)
    g = Hydra(m, h, load_tree("tree15_d3"), {k: v.cuda() for k, v in make_weights(m, h, 92).items()}, 1, 256)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        g.prefill([p.cuda() for p in make_prompts(92, [50], m.vocab)])
        cand = torch.randint(0, m.vocab, (1, 16), dtype=torch.int32, device="cuda")
        want = [g.verify(cand, want_logits=True) for _ in range(3)][-1]
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            amax, logits = g.verify(cand, want_logits=True)
        graph.replay()
    st.synchronize()
    assert torch.equal(amax, want[0]) and torch.equal(logits, want[1])
    graph.reset()
    g.close()
