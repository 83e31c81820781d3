"""Float tree attention of short caches and few rows (the keys of a row shared out over warps): every number of rows a CTA takes, row counts
that end inside a CTA, key counts around the rounds of a warp, empty and ragged sequences."""
import pytest
import torch

from oracle.hydra_oracle import masked_attention
from tests.test_gpu_kernels import rnd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("B,H,tc", [(1, 4, 1), (1, 4, 16), (1, 3, 63), (3, 4, 31), (5, 4, 50), (2, 9, 64), (8, 4, 64)])
@pytest.mark.parametrize("S", [66, 150, 512])
def test_rows_and_keys(hd, B, H, tc, S):
    from paper_2402_05109_b200 import tree_attention
    S = max(S, tc + 2)
    pos0 = [S - tc, 0, 15, 1, 33, 2, 7, 40][:B]
    pos0 = [min(p, S - tc) for p in pos0]
    n_rows = [tc, max(1, tc - 3), tc, 0, 1, tc, tc, 2][:B]
    q, kc, vc = (rnd(s, 83, i, torch.float32) for i, s in ((3, (B * tc, H, hd)), (1, (B, H, S, hd)), (2, (B, H, S, hd))))
    for b in range(B):                                   # slots past the end hold non-finite garbage
        kc[b, :, pos0[b] + n_rows[b]:] = float("nan")
        vc[b, :, pos0[b] + n_rows[b]:] = float("inf")
    par = [max(0, (i - 1) // 2) for i in range(tc)]      # a binary tree
    anc = [[j == i for j in range(tc)] for i in range(tc)]
    for i in range(1, tc):
        anc[i] = [a or b for a, b in zip(anc[i], anc[par[i]])]
    words = [sum(1 << j for j in range(tc) if anc[i][j]) for i in range(tc)]
    mask = torch.tensor([w - (1 << 64) if w >= 1 << 63 else w for w in words], dtype=torch.int64)
    dev = lambda x: torch.tensor(x, dtype=torch.int32).cuda()
    out = tree_attention(q.cuda(), kc.cuda(), vc.cuda(), dev(pos0), dev(n_rows), mask.cuda(), tc).cpu().view(B, tc, H, hd)
    for b in range(B):
        n, L = n_rows[b], pos0[b] + n_rows[b]
        assert n == tc or float(out[b, n:].abs().max()) == 0.0
        if n == 0:
            continue
        allowed = torch.cat([torch.ones(n, pos0[b], dtype=torch.bool), torch.tensor(anc, dtype=torch.bool)[:n, :n]], dim=1)
        ref = masked_attention(q.view(B, tc, H, hd)[b, :n].double(), kc[b, :, :L].permute(1, 0, 2).double(), vc[b, :, :L].permute(1, 0, 2).double(), allowed)
        # float sums of up to 512 terms and expf of scores of size ~10: a few ulp of either (2^-23), with the margin of the test of the general kernel
        assert float((out[b, :n].double() - ref).abs().max()) <= 2e-5
