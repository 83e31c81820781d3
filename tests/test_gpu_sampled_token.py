"""The token after an accepted path, drawn by inverse CDF, at vocabularies whose 256 ranges take several rounds of 32 tokens, end inside a round or
inside the vocabulary, and hold more than 256 tokens: tokens of enough weight are hit exactly, the rest within the float sums' error."""
import pytest
import torch

from synth import load_tree, make_prompts, make_weights
from synth.configs import ModelCfg, HeadCfg

pytestmark = pytest.mark.gpu

# The CDF of float sums against float64: a weight's __expf is within 2 + 1.173 |x| ulp (|x| <= 20 for what weighs anything: 26 x 2^-24 x 2), a range's sum and
# the scan add up to 512 numbers one after the other (2^-24 each at most): 3.1e-6 + 3.1e-5, and as much again where the walk repeats the range's sum.
DELTA = 7e-5


@pytest.mark.parametrize("vocab", [1024, 20608, 32000, 70016])
def test_heavy_tokens_are_hit_and_the_ends_are_kept(vocab):
    from paper_2402_05109_b200 import Hydra
    B, tau, per = 16, 0.15, (vocab + 255) // 256
    m = ModelCfg(1, 256, 2, 128, 512, vocab, dtype="bf16")
    h = HeadCfg(2, 1, False)
    w = make_weights(m, h, 97, device="cuda")
    g = Hydra(m, h, load_tree("tree15_d3")[:3], w, B, 128)
    u = torch.zeros(B, device="cuda")
    gen = torch.Generator().manual_seed(12)
    offsets = set()
    with torch.cuda.stream(torch.cuda.Stream()):
        g.prefill([p.cuda() for p in make_prompts(97, [5 + b for b in range(B)], vocab)])
        g.set_acceptance(1, tau, 1.0, 1e9, u)                # p > 1: no candidate passes, the token follows the root
        cand = torch.randint(0, vocab, (B, 3), dtype=torch.int32, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
        for turn in range(10):
            amax, logits = g.verify(cand, want_logits=True)
            p = torch.softmax(logits[:, 0].double() / tau, dim=-1).cpu()
            cdf = torch.cumsum(p, dim=-1)
            want = [None] * B
            for b in range(B):
                heavy = torch.nonzero(p[b] > 4 * DELTA)[:, 0]
                if turn == 0:
                    u[b] = 0.0
                    want[b] = 0
                elif turn == 1:
                    u[b] = 1.0 - 2.0 ** -24
                elif turn == 2:                              # where a range begins
                    u[b] = float(cdf[b, per * (15 * b + 7) % vocab])
                else:                                        # the middle of a token: the last of its range, the first, late in the vocabulary, any
                    at = heavy % per
                    order = (at, -at, heavy, torch.rand(len(heavy), generator=gen))[turn % 4].argsort(descending=True)
                    t = int(heavy[order[b if turn < 7 else b * 5 % len(heavy)]])
                    u[b] = float(cdf[b, t] - p[b, t] / 2)
                    want[b] = t
                    offsets.add(t % per)
            n, path, out = g.accept_compact(cand, amax)
            g.poll_status()
            assert int(n.max()) == 0
            for b, tok in enumerate(out[:, 0].tolist()):
                if want[b] is not None:
                    assert tok == want[b], (turn, b, tok, want[b])
                lo = float(cdf[b, tok - 1]) if tok else 0.0
                assert lo - DELTA <= float(u[b]) < float(cdf[b, tok]) + DELTA, (turn, b, tok)
            assert g.get_buffer("ROOT_TOK")[:B].tolist() == out[:, 0].tolist()
    assert max(offsets) >= min(per, 257) - 1 and min(offsets) == 0      # ranges' ends and starts, rounds past the first of 32 and of 256
    g.close()
