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


@pytest.mark.parametrize("m,n,k", [(64, 1024, 4096), (512, 4096, 512), (16, 256, 688)])
def test_chained_calls_read_the_first_ones_result(m, n, k):
    """Two calls in a row on one stream through the C entry point, the second with the first one's result as its weights: stream
    order alone has to be enough, and no element may be read before the first call has written it."""
    from paper_2402_05109_b200.binding import lib, _stream
    x = normal_(torch.empty(m, k, device="cuda"), 73, m, 1.0)
    w = normal_(torch.empty(n, k, device="cuda"), 74, n, 0.02)
    x2 = normal_(torch.empty(9, n, device="cuda"), 75, n, 1.0)
    ref = x2.double() @ (x.double() @ w.double().T).T
    for _ in range(20):
        mid, out = torch.full((m, n), float("nan"), device="cuda"), torch.empty(9, m, device="cuda")
        part = torch.empty(max(m * n, 9 * m), device="cuda")
        torch.cuda.synchronize()
        for a, b, c, mm, nn, kk in ((x, w, mid, m, n, k), (x2, mid, out, 9, m, n)):
            assert lib.hydra_gemm(a.data_ptr(), b.data_ptr(), c.data_ptr(), part.data_ptr(), mm, nn, kk, 0, 0, 1, None, _stream()) == 0
        # two float products in a row: k^0.5 and n^0.5 ulp on the scale of the largest sum
        assert float((out.double() - ref).abs().max()) <= 2e-5 * float(ref.abs().max())


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_operands_off_a_boundary_of_four_elements_are_refused(dtype):
    from paper_2402_05109_b200 import HydraError, gemm
    buf = torch.zeros(8 * 64 + 4, dtype=dtype, device="cuda")
    good, off = buf[:8 * 64].view(8, 64), buf[1:1 + 8 * 64].view(8, 64)
    assert gemm(good, good, mode=1).shape == (8, 8)
    for x, w in ((off, good), (good, off)):
        with pytest.raises(HydraError, match="invalid"):
            gemm(x, w, mode=1)
