"""Tree attention over every way of cutting the keys: one chunk per (head, sequence) pair (rows normalised and written out of
tensor memory) up to eight (rows merged across the cluster), with sequences that are empty, shorter
than the chunk count in tiles, and ragged in their row counts."""
import pytest
import torch

from oracle.hydra_oracle import masked_attention
from tests.test_gpu_kernels import rnd, _dev

pytestmark = pytest.mark.gpu

# with 148 SMs and nine 64-key tiles the pair counts below are cut into up to eight chunks down to one
PAIRS = [(4, 1), (4, 5), (4, 7), (4, 9), (4, 17), (4, 40)]


@pytest.mark.parametrize("hd,planes,tc", [(128, 2, 64), (128, 2, 128), (128, 1, 33), (64, 2, 40), (64, 1, 128)])
@pytest.mark.parametrize("B,H", PAIRS)
def test_chunk_counts(B, H, hd, planes, tc):
    from paper_2402_05109_b200 import tree_attention
    S = 576
    pos0, n_rows = [S - tc, 0, 70, 200], [tc, min(tc, 31), 0, tc - 1]
    src = torch.float32 if planes == 2 else torch.float16
    (q_d, q), (k_d, kc), (v_d, vc) = (_dev(rnd(shape, 29, i, src), planes)
                                      for i, shape in ((3, (B * tc, H, hd)), (1, (B, H, S, hd)), (2, (B, H, S, hd))))
    dev = lambda x, t=torch.int32: torch.tensor(x, dtype=t).cuda()
    out = tree_attention(q_d, k_d, v_d, dev(pos0), dev(n_rows), None, tc, out_planes=2).float().cpu().sum(0).view(B, tc, H, hd)
    for b in range(B):
        n, L = n_rows[b], pos0[b] + n_rows[b]
        assert n == tc or float(out[b, n:].abs().max()) == 0.0
        if n == 0:
            continue
        allowed = torch.cat([torch.ones(n, pos0[b], dtype=torch.bool), torch.tril(torch.ones(n, n, dtype=torch.bool))], dim=1)
        ref = masked_attention(q.view(B, tc, H, hd)[b, :n].double(), kc[b, :, :L].permute(1, 0, 2).double(),
                               vc[b, :, :L].permute(1, 0, 2).double(), allowed)
        # one plane: softmax weights rounded to float16 (2^-12 relative); two: the hi/lo rounding of the result (2^-17)
        assert float((out[b, :n].double() - ref).abs().max()) <= (1.5e-3 if planes == 1 else 1e-4)


def test_result_buffer_off_a_16_byte_boundary():
    """The result only has to lie on an 8-byte boundary; with one chunk per pair the launch then merges two."""
    from paper_2402_05109_b200 import tree_attention, lib
    B, H, hd, S, tc = 4, 40, 128, 192, 16
    q, kc, vc = (rnd(s, 31, i, torch.float16).cuda() for i, s in ((3, (B * tc, H, hd)), (1, (B, H, S, hd)), (2, (B, H, S, hd))))
    pos0 = torch.tensor([100, 0, 64, 170], dtype=torch.int32).cuda()
    want = tree_attention(q, kc, vc, pos0, None, None, tc, out_planes=1)
    buf = torch.zeros(B * tc * H * hd + 8, dtype=torch.bfloat16, device="cuda")
    out, status = buf[4:4 + B * tc * H * hd], torch.zeros(1, dtype=torch.int32, device="cuda")
    assert lib.hydra_tree_attention(q.data_ptr(), kc.data_ptr(), vc.data_ptr(), pos0.data_ptr(), None, None, out.data_ptr(), None,
                                    B, tc, H, hd, S, 1, 1, 1, status.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    got = out.view_as(want).float()
    # both round the same float result to bfloat16, summed in a different order: at most one bfloat16 step (2^-8) apart
    assert float((got - want.float()).abs().max()) <= float(want.float().abs().max()) * 2.0 ** -8
    assert int(status) == 0 and float(buf[:4].abs().max()) == 0.0 and float(buf[-4:].abs().max()) == 0.0


@pytest.mark.parametrize("hd,S,tc", [(64, 96, 16), (128, 96, 64), (64, 400, 64), (128, 300, 5)])      # one chunk of keys and several
@pytest.mark.parametrize("which", ["q", "k", "v"])
def test_float_operands_off_a_16_byte_boundary(hd, S, tc, which):
    """Float q, K and V may be any float tensors, views into larger buffers included: bit for bit the result of aligned ones."""
    from paper_2402_05109_b200 import tree_attention
    B, H = 2, 3
    ops = {n: rnd(s, 37, i, torch.float32).cuda() for i, (n, s) in enumerate({"q": (B * tc, H, hd), "k": (B, H, S, hd), "v": (B, H, S, hd)}.items())}
    pos0, n_rows = (torch.tensor(x, dtype=torch.int32).cuda() for x in ([S - tc, 7], [tc, tc - 1]))
    mask = torch.tensor([(1 << (i + 1)) - 1 if i < 63 else -1 for i in range(tc)], dtype=torch.int64).cuda()
    want = tree_attention(ops["q"], ops["k"], ops["v"], pos0, n_rows, mask, tc)
    for off in (1, 2, 3):
        t = ops[which]
        buf = torch.empty(t.numel() + 4, device="cuda")
        view = buf[off:off + t.numel()].view(t.shape)
        view.copy_(t)
        moved = dict(ops, **{which: view})
        assert torch.equal(tree_attention(moved["q"], moved["k"], moved["v"], pos0, n_rows, mask, tc), want)
