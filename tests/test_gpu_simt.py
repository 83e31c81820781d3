"""The float path's GEMM at the edges of its dispatch: row groups of 1, 4, 8 and 16, one / two / four warps per column, remainders."""
import pytest
import torch

from synth import normal_

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 3, 4, 5, 8, 9, 16, 17, 64])
@pytest.mark.parametrize("n,k", [(1, 4), (7, 132), (256, 688), (768, 256), (1024, 512), (1376, 260), (3000, 1028)])
def test_simt_gemm(m, n, k):
    from paper_2402_05109_b200 import gemm
    x = normal_(torch.empty(m, k, device="cuda"), 71, m + k, 1.0)
    w = normal_(torch.empty(n, k, device="cuda"), 72, n, 0.02)
    ref = x.double() @ w.double().T
    # float products and sums of k terms: k^0.5 ulp of the terms, on the scale of the largest sum
    assert float((gemm(x, w).double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6
