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


@pytest.mark.parametrize("m", [96, 97, 112, 128, 129, 160, 161])
@pytest.mark.parametrize("n", [18816, 18944, 19072])
def test_gemm_wide_units_at_97_to_160_rows(m, n):
    """Both sides of the lines in rows and in width, and an output that ends inside its last unit."""
    from paper_2402_05109_b200 import gemm
    k = 320
    x = normal_(torch.empty(m, k, device="cuda"), 79, m, 1.0)
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 80, n, 0.02)
    planes = split_hi_lo(x)
    ref = planes.double().sum(0) @ w.double().T
    # as above
    assert float((gemm(planes, w, mode=0).double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5


@pytest.mark.parametrize("m", [4097, 4360])
@pytest.mark.parametrize("n,k", [(1152, 1024), (4224, 2048)])
def test_gemm_groups_of_row_tiles(m, n, k):
    """More row tiles than walk the weights together: two groups of 9, with 4097 rows one of the 18 places empty."""
    from paper_2402_05109_b200 import gemm
    x = normal_(torch.empty(m, k, device="cuda"), 77, m, 1.0)
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 78, n, 0.02)
    planes = split_hi_lo(x)
    ref = planes.double().sum(0) @ w.double().T
    # as above
    assert float((gemm(planes, w, mode=0).double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5


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


@pytest.mark.parametrize("m,n,k", [(8, 640, 5632), (9, 640, 5632), (9, 256, 4096), (8, 768, 7744), (16, 256, 11008), (64, 8192, 2048), (40, 3072, 1920)])
def test_gemm_noalloc_slots_of_a_tile(m, n, k):
    """Up to 17 or 23 slots a tile in one launch, more in two; in the second one up to twelve in flight together, more in turn."""
    test_gemm_noalloc_one_and_two_launches(m, n, k)


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


@pytest.mark.parametrize("m", [3, 64])
@pytest.mark.parametrize("noalloc", [False, True])
def test_weights_written_by_the_preceding_kernel(m, noalloc):
    """The weights of a stand-alone call may be the result of the kernel before it on the stream (here the library's attention, which
    lets its successor start early): stream order alone has to be enough."""
    from paper_2402_05109_b200 import tree_attention
    from paper_2402_05109_b200.binding import lib, _stream
    B, tc, H, hd, S = 2, 64, 8, 128, 2048
    n, k = B * tc, H * hd
    half = lambda shape, i: normal_(torch.empty(shape, dtype=torch.float16, device="cuda"), 81, i, 1.0)
    q, kc, vc = half((n, H, hd), 1), half((B, H, S, hd), 2), half((B, H, S, hd), 3)
    pos0 = torch.tensor([S - tc, S - 2 * tc], dtype=torch.int32, device="cuda")
    x = normal_(torch.empty(m, k, dtype=torch.bfloat16, device="cuda"), 82, m, 1.0)
    w = tree_attention(q, kc, vc, pos0, None, None, tc)
    ref = x.double() @ w.double().T
    part = torch.empty(lib.hydra_gemm_partial_floats(m, n, k, 1, 0), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(20):
        w.fill_(float("nan"))
        out = torch.empty(m, n, device="cuda")
        torch.cuda.synchronize()
        assert lib.hydra_tree_attention(q.data_ptr(), kc.data_ptr(), vc.data_ptr(), pos0.data_ptr(), None, None, w.data_ptr(), None,
                                        B, tc, H, hd, S, 1, 1, 1, status.data_ptr(), _stream()) == 0
        if noalloc:
            assert lib.hydra_gemm_noalloc(x.data_ptr(), w.data_ptr(), out.data_ptr(), m, n, k, status.data_ptr(), _stream()) == 0
        else:
            assert lib.hydra_gemm(x.data_ptr(), w.data_ptr(), out.data_ptr(), part.data_ptr(), m, n, k, 1, 0, 1, status.data_ptr(), _stream()) == 0
        assert float((out.double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5
    assert int(status.item()) == 0


def _noalloc_counters():
    """The counters of hydra_gemm_noalloc's one-launch form as an int64 tensor."""
    import ctypes as C
    from paper_2402_05109_b200.binding import lib
    ptr, part, cnt = C.c_void_p(), C.c_size_t(), C.c_size_t()
    assert lib.hydra_gemm_noalloc_scratch(C.byref(ptr), C.byref(part), C.byref(cnt)) == 0 and part.value == 8 << 20

    class View:
        __cuda_array_interface__ = dict(shape=(cnt.value // 8,), typestr="<i8", data=(ptr.value + part.value, False), version=2)
    return torch.as_tensor(View(), device="cuda")


@pytest.mark.parametrize("m,n,k", [(1, 128, 64), (11, 2048, 2048), (16, 640, 5632)])
def test_gemm_noalloc_after_a_call_that_left_its_counters(m, n, k):
    """A call that timed out, or that another one overlapped, leaves tiles counted in part.  Later calls, and replays of a
    captured one, must not see it: every counter set to a small count of the first call before each of them."""
    from paper_2402_05109_b200 import gemm_noalloc
    counters = _noalloc_counters()
    x = normal_(torch.empty(m, k, dtype=torch.bfloat16, device="cuda"), 67, m + k, 1.0)
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 68, n, 0.02)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = x.double() @ w.double().T
    tol = 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5
    out = torch.empty(m, n, device="cuda")
    gemm_noalloc(x, w, out, status)
    assert n // 128 <= counters.numel() and int(counters[: n // 128].abs().max()) == 0
    graph, replayed = torch.cuda.CUDAGraph(), torch.empty(m, n, device="cuda")
    with torch.cuda.graph(graph):
        gemm_noalloc(x, w, replayed, status)
    for left in range(1, 9):
        for again, call in ((out, lambda: gemm_noalloc(x, w, out, status)), (replayed, graph.replay)):
            counters.fill_((1 << 16) + left)
            again.fill_(float("nan"))
            call()
            torch.cuda.synchronize()
            assert float((again.double() - ref).abs().max()) <= tol
    counters.zero_()
    assert int(status.item()) == 0


@pytest.mark.parametrize("m,n,k", [(64, 11008, 4096), (128, 8192, 2048), (100, 12800, 1024)])
def test_gemm_noalloc_takes_fewer_ctas_where_the_sums_would_not_fit(m, n, k):
    """Results that fit the built-in scratch although the partial sums of the usual plan do not: fewer CTAs share the work."""
    from paper_2402_05109_b200 import gemm_noalloc
    from paper_2402_05109_b200.binding import lib
    assert m * n * 4 <= 8 << 20 < 4 * lib.hydra_gemm_partial_floats(m, n, k, 1, 0)
    x = normal_(torch.empty(m, k, dtype=torch.bfloat16, device="cuda"), 69, m + k, 1.0)
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 70, n, 0.02)
    status, out = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((m, n), float("nan"), device="cuda")
    gemm_noalloc(x, w, out, status)
    ref = x.double() @ w.double().T
    assert float((out.double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5
    assert int(status.item()) == 0


@pytest.mark.parametrize("m", [64, 65, 80, 112, 144, 160, 208, 224, 240, 288, 320])
@pytest.mark.parametrize("n", [512, 22016])
def test_gemm_ring_above_64_rows(m, n):
    """Row tiles whose stages fill more than 200 KB, and their neighbours; more blocks of k than stages, units of one and of two weight tiles."""
    from paper_2402_05109_b200 import gemm
    k = 1088
    x = normal_(torch.empty(m, k, device="cuda"), 81, m, 1.0)
    w = normal_(torch.empty(n, k, dtype=torch.bfloat16, device="cuda"), 82, n, 0.02)
    # as above
    for planes in (split_hi_lo(x), x.to(torch.bfloat16)):
        ref = (planes.double().sum(0) if planes.dim() == 3 else planes.double()) @ w.double().T
        assert float((gemm(planes, w, mode=0).double() - ref).abs().max()) <= 1e-5 * float(ref.abs().max()) + 1e-6 * k ** 0.5
