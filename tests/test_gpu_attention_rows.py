"""Float16 attention of one and two rows a sequence: lengths around the lane groups' rounds (32 or 64 keys a round of a CTA, four rounds in flight) and the chunks' cuts, empty
sequences and rows, with and without a mask.  What lies behind a sequence's keys in its cache is not a number and would show in every result that read it
(in the zeros of rows past the call's, too: a sum that is no number stays none)."""
import pytest
import torch

from oracle.hydra_oracle import masked_attention
from tests.test_gpu_kernels import rnd, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,planes", [(128, 2), (128, 1), (64, 2), (64, 1)])
@pytest.mark.parametrize("tc,masked", [(1, True), (1, False), (2, True), (2, False)])
@pytest.mark.parametrize("H,S,pos0", [(1, 96, [0, 1, 31, 33, 63]), (5, 300, [64, 127, 128, 129, 297]), (60, 700, [255, 257, 511, 0, 690])])
def test_few_rows(H, S, pos0, tc, masked, hd, planes):
    from paper_2402_05109_b200 import tree_attention
    B, n_rows = len(pos0), [tc, tc, tc - 1, tc, tc]
    src = torch.float32 if planes == 2 else torch.float16
    (q_d, q), (k_d, kc), (v_d, vc) = (_dev(rnd(shape, 91, i, src), planes) for i, shape in ((3, (B * tc, H, hd)), (1, (B, H, S, hd)), (2, (B, H, S, hd))))
    for b in range(B):
        for cache in (k_d, v_d):
            cache[..., b, :, pos0[b] + n_rows[b]:, :] = float("nan")
    bits = [1, 2]                                         # two siblings: the second does not see the first
    dev = lambda x, t=torch.int32: torch.tensor(x, dtype=t).cuda()
    out = tree_attention(q_d, k_d, v_d, dev(pos0), dev(n_rows), dev(bits[:tc], torch.int64) if masked else None, tc, out_planes=2).float().cpu().sum(0).view(B, tc, H, hd)
    for b in range(B):
        n, L = n_rows[b], pos0[b] + n_rows[b]
        assert n == tc or float(out[b, n:].abs().max()) == 0.0
        if n == 0:
            continue
        new = torch.eye(n, dtype=torch.bool) if masked else torch.tril(torch.ones(n, n, dtype=torch.bool))
        allowed = torch.cat([torch.ones(n, pos0[b], dtype=torch.bool), new], dim=1)
        ref = masked_attention(q.view(B, tc, H, hd)[b, :n].double(), kc[b, :, :L].permute(1, 0, 2).double(), vc[b, :, :L].permute(1, 0, 2).double(), allowed)
        # weights and sums are float; the result is rounded to two bfloat16 planes (2^-17 of at most 4)
        assert float((out[b, :n].double() - ref).abs().max()) <= 1e-4


def test_lengths_past_the_cache_give_zeros():
    from paper_2402_05109_b200 import tree_attention
    H, S, hd = 3, 80, 128
    q, k, v = (rnd(s, 92, i, torch.float16).cuda() for i, s in ((3, (5, H, hd)), (1, (5, H, S, hd)), (2, (5, H, S, hd))))
    out = tree_attention(q, k, v, torch.tensor([S, -1, 1 << 30, 2147483647, S - 1], dtype=torch.int32).cuda(), None, None, 1, out_planes=2).float().sum(0).view(5, H, hd)
    assert float(out[:4].abs().max()) == 0.0 and float(out[4].abs().min(-1).values.max()) > 0.0


@pytest.mark.parametrize("planes", [1, 2])
@pytest.mark.parametrize("tc", [1, 2])
@pytest.mark.parametrize("H,B,length", [(4, 2, 20), (4, 2, 700), (50, 3, 70)])      # one round, several chunks, one chunk
def test_what_is_not_a_number_shows(H, B, length, tc, planes):
    """A key, a value or a score that is not finite reaches every row that sees it, as on the tensor cores (three rows), and no other sequence, head or row."""
    from paper_2402_05109_b200 import tree_attention
    hd, S, b0, h0, bad = 128, length + 8, B - 1, H - 2, float("nan")
    base = [rnd(shape, 93, i, torch.float16) for i, shape in ((3, (B, 3, H, hd)), (1, (B, H, S, hd)), (2, (B, H, S, hd)))]
    pos0, bits = torch.full((B,), length, dtype=torch.int32).cuda(), [1, 2, 4]

    def call(rows, poison):
        q, k, v = (torch.stack([t, torch.zeros_like(t)]) if planes == 2 else t[None].clone() for t in base)
        poison(q, k, v)
        q = q[:, :, :rows].reshape(planes, B * rows, H, hd)
        q, k, v = (t.contiguous().cuda() if planes == 2 else t[0].contiguous().cuda() for t in (q, k, v))
        out = tree_attention(q, k, v, pos0, None, torch.tensor(bits[:rows], dtype=torch.int64).cuda(), rows, out_planes=2)
        return out.float().sum(0).view(B, rows, H, hd)[:, :tc].cpu()

    def key_nan(q, k, v): k[:, b0, h0, length // 2, 5] = bad

    def key_inf(q, k, v):                                  # a value past float16: hi is inf, lo what is left of it
        k[0, b0, h0, length // 3, :] = float("inf")
        if planes == 2: k[1, b0, h0, length // 3, :] = -float("inf")
    def score_inf(q, k, v): q[0, b0, :, h0, 7] = 1.0; k[0, b0, h0, 3, 7] = float("inf")
    def value_nan(q, k, v): v[:, b0, h0, length - 1, :] = bad
    def faint_value_nan(q, k, v): q[0, b0, :, h0, :] = 8.0; k[0, b0, h0, :length] = 8.0; k[0, b0, h0, 0] = -8.0; v[:, b0, h0, 0, :] = bad      # a weight of zero
    where = torch.zeros(B, tc, H, hd, dtype=torch.bool)
    where[b0, :, h0] = True
    for poison in (key_nan, key_inf, score_inf, value_nan, faint_value_nan):
        got = call(tc, poison)
        assert torch.equal(got.isnan(), where), poison.__name__
        assert torch.equal(call(3, poison).isnan(), where), poison.__name__
    # the query of the last row, and the key of the last row, which only that one sees
    def query_nan(q, k, v): q[:, b0, tc - 1, h0, 9] = bad
    def own_nan(q, k, v): k[:, b0, h0, length + tc - 1] = bad; v[:, b0, h0, length + tc - 1] = bad
    where[b0, :tc - 1, h0] = False
    for poison in (query_nan, own_nan):
        assert torch.equal(call(tc, poison).isnan(), where), poison.__name__
    if planes == 1:                                        # every visible score -inf: no weight at all, and zeros as on the tensor cores
        def no_weight(q, k, v): q[0, b0, :, h0] = 1.0; k[0, b0, h0, :length + tc] = -float("inf")
        assert float(call(tc, no_weight)[b0, :, h0].abs().max()) == 0.0


@pytest.mark.parametrize("hd,planes", [(128, 2), (64, 1)])
@pytest.mark.parametrize("tc", [1, 2])
@pytest.mark.parametrize("H,S,pos0", [(1, 440, [0, 1, 200, 300, 437]), (2, 700, [0, 63, 100, 640, 697]),      # six to eight chunks
                                      (32, 800, [0, 127, 400, 766, 798]), (32, 767, [0, 63, 384, 700, 765]), (41, 768, [1, 63, 384, 700, 766]),      # two for a short last wave
                                      (7, 1024, [0, 64, 600, 1000, 1022])])
def test_chunks(H, S, pos0, tc, hd, planes):
    test_few_rows(H, S, pos0, tc, True, hd, planes)


@pytest.mark.parametrize("hd", [64, 128])
def test_two_rows_past_the_line(hd):
    """The tensor cores' side of 1024 keys; two planes leave the same error."""
    test_few_rows(7, 1025, [0, 64, 600, 1000, 1023], 2, True, hd, 2)
