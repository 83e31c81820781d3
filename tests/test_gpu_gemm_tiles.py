"""Tensor-core GEMM at the edges of its tile choice: row tiles of any multiple of 16 rows, 16 / 17 rows (epilogue paths), 64 / 65, 128 / 129
(one pass, a pass per plane), two row tiles; 128 and 256 weight rows per unit, an output that ends inside its last unit."""
import pytest
import torch

from synth import normal_
from tests.parity import split_hi_lo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 15, 16, 17, 47, 64, 65, 80, 112, 128, 129, 176, 256, 257, 308, 513])
@pytest.mark.parametrize("n,k", [(128, 64), (384, 704), (4096 + 128, 1024), (4096, 4096)])
def test_gemm_tile_edges(m, n, k):
    from paper_2402_05109_b200 import gemm
    x = normal_(torch.empty(m, k, device="cuda"), 61, m + k, 1.0)
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 62, n, 0.02)
    # planes hold 16 bits, products are exact, only the order of the float sums differs: k terms of size ~0.02, a few ulp of the largest sum
    for planes in (split_hi_lo(x), x.to(torch.bfloat16)):
        ref = (planes.double().sum(0) if planes.dim() == 3 else planes.double()) @ w.double().T
        out = gemm(planes, w, mode=0).double()
        assert float((out - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5


@pytest.mark.parametrize("m,n,k", [(1, 128, 64), (1, 256, 256), (11, 2048, 2048), (16, 640, 5632), (16, 1408, 4288), (17, 1408, 4288), (3, 4096, 4096)])
def test_gemm_noalloc_one_and_two_launches(m, n, k):
    """Both sides of the choice between adding the partial sums in the GEMM's own launch and in a second one; several calls in a
    row, because the counters of one call have to be left clean for the next."""
    from paper_2402_05109_b200 import gemm_noalloc
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 63, n, 0.02)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for i in range(4):
        x = normal_(torch.empty(m, k, dtype=torch.bfloat16, device="cuda"), 64 + i, m + k, 1.0)
        out = torch.full((m, n), float("nan"), device="cuda")
        gemm_noalloc(x, w, out, status)
        ref = x.double() @ w.double().T
        assert float((out.double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5
    assert int(status.item()) == 0


@pytest.mark.parametrize("m,n,k", [(1, 128, 64), (11, 2048, 2048), (3, 4096, 4096)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_gemm_noalloc_result_off_a_16_byte_boundary(m, n, k, offset):
    """The result may be any float tensor, a view into a larger buffer included, at sizes on both sides of the one-launch choice."""
    from paper_2402_05109_b200 import gemm_noalloc
    x = normal_(torch.empty(m, k, dtype=torch.bfloat16, device="cuda"), 65, m + k, 1.0)
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 66, n, 0.02)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    buf = torch.full((m * n + 8,), 7.0, device="cuda")
    out = buf[offset:offset + m * n].view(m, n)
    gemm_noalloc(x, w, out, status)
    ref = x.double() @ w.double().T
    assert float((out.double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5
    assert bool((buf[:offset] == 7.0).all()) and bool((buf[offset + m * n:] == 7.0).all()) and int(status.item()) == 0
