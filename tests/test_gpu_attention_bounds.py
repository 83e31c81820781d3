"""Float tree attention whose device-side lengths say more than the cache or the call holds: keys end with the cache, rows with the call.  What
lies behind the caches in memory is not a number and would show in every result that read it."""
import pytest
import torch

from oracle.hydra_oracle import masked_attention
from tests.test_gpu_kernels import rnd

pytestmark = pytest.mark.gpu


# few rows and keys (one, two and four rows a CTA), then caches and batches of the kernel whose CTAs share a staged tile
@pytest.mark.parametrize("B,H,tc,S", [(1, 4, 16, 80), (2, 4, 50, 100), (3, 4, 64, 300), (1, 4, 16, 700), (3, 4, 64, 1030), (8, 16, 64, 200)])
@pytest.mark.parametrize("hd", [64, 128])
def test_lengths_past_the_cache(hd, B, H, tc, S):
    from paper_2402_05109_b200 import tree_attention
    pos0 = [S - 3, S + 40, S - tc + 1, S, 0, 2, S - 1, 1 << 30][:B]
    n_rows = [tc, tc, tc, tc - 1, tc + 5, tc, 1 << 30, tc][:B]
    q = rnd((B * tc, H, hd), 84, 3, torch.float32)
    behind = torch.full((256 * hd,), float("nan"))
    caches = []
    for i in (1, 2):
        flat = torch.cat([rnd((B, H, S, hd), 84, i, torch.float32).flatten(), behind]).cuda()
        caches.append(flat[:B * H * S * hd].view(B, H, S, hd))
    mask = torch.tensor([(1 << (i + 1)) - 1 if i < 63 else -1 for i in range(tc)], dtype=torch.int64)      # a chain
    dev = lambda x: torch.tensor(x, dtype=torch.int32).cuda()
    out = tree_attention(q.cuda(), caches[0], caches[1], dev(pos0), dev(n_rows), mask.cuda(), tc).cpu().view(B, tc, H, hd)
    for b in range(B):
        n = min(n_rows[b], tc)
        keys = min(pos0[b] + n, S)
        assert n == tc or float(out[b, n:].abs().max()) == 0.0
        slot = torch.arange(keys)
        allowed = slot[None, :] <= pos0[b] + torch.arange(n)[:, None]
        k, v = (c[b, :, :keys].permute(1, 0, 2).cpu().double() for c in caches)
        ref = masked_attention(q.view(B, tc, H, hd)[b, :n].double(), k, v, allowed)
        # as in the test of the kernels inside their range: float sums of up to 1030 terms, a few ulp (2^-23) each
        assert float((out[b, :n].double() - ref).abs().max()) <= 2e-5
