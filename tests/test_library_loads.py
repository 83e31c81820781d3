"""The C-ABI library builds for sm_100a, loads without a GPU and exports every symbol the header declares."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_exports_every_declared_symbol():
    from paper_2402_05109_b200.build import build
    build()
    import paper_2402_05109_b200 as pkg
    hdr = open(os.path.join(ROOT, "include", "hydra.h")).read()
    names = sorted(set(re.findall(r"\b(hydra_[a-z_0-9]+)\s*\(", hdr)))
    assert len(names) >= 18
    for n in names:
        assert hasattr(pkg.lib, n), n
    assert pkg.lib.hydra_status_str(3).decode() == "call out of order"


def test_workspace_bytes_and_invalid_configs_without_gpu():
    import ctypes as C
    from paper_2402_05109_b200.binding import lib, ModelCfgC, HeadCfgC, TreeCfgC
    mc = ModelCfgC(2, 256, 4, 64, 688, 1024, 1e-6, 1e4, 0, 1, 128)
    hc = HeadCfgC(3, 1, 0, 1)
    par = (C.c_int32 * 4)(-1, 0, 0, 1)
    n = lib.hydra_workspace_bytes(C.byref(mc), C.byref(hc), C.byref(TreeCfgC(4, par)))
    assert n > 2 * 2 * 4 * 128 * 64 * 4 and n % 256 == 0
    bad = (C.c_int32 * 4)(-1, 0, 1, 0)                       # rows not ordered by (depth, rank path)
    assert lib.hydra_workspace_bytes(C.byref(mc), C.byref(hc), C.byref(TreeCfgC(4, bad))) == 0
    deep = (C.c_int32 * 5)(-1, 0, 1, 2, 3)                   # deeper than the number of heads
    assert lib.hydra_workspace_bytes(C.byref(mc), C.byref(hc), C.byref(TreeCfgC(5, deep))) == 0
    mc.n_heads = 3                                           # n_heads * head_dim != d_model
    assert lib.hydra_workspace_bytes(C.byref(mc), C.byref(hc), C.byref(TreeCfgC(4, par))) == 0


def test_current_stream_without_the_private_torch_function(monkeypatch):
    """The raw-stream shortcut is not a public name of torch: the binding works where it is absent."""
    from types import SimpleNamespace
    import torch
    from paper_2402_05109_b200 import binding
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=7))
    monkeypatch.setattr(binding, "_raw_stream", lambda device: 100 + device)
    assert binding._stream() == 103
    monkeypatch.setattr(binding, "_raw_stream", None)
    assert binding._stream() == 7


def test_weights_off_a_boundary_of_four_elements_are_refused():
    """The checks come before anything touches the device: made-up addresses do on a machine without a GPU."""
    import ctypes as C
    import pytest
    import torch
    from paper_2402_05109_b200.binding import lib, HeadCfgC, ModelCfgC, TreeCfgC, WeightsC, _PP
    if torch.cuda.is_available():
        pytest.skip("with a GPU the good call would go on to the device")
    L, K = 2, 1
    mc, hc = ModelCfgC(L, 256, 4, 64, 688, 1024, 1e-6, 1e4, 0, 1, 128), HeadCfgC(K, 1, 1, 0)
    tc = TreeCfgC(2, (C.c_int32 * 2)(-1, 0))
    arrays = ("attn_norm", "wqkv", "wo", "ffn_norm", "w_gate_up", "w_down", "head_w1", "head_b1", "head_wr", "head_br")

    def create(name=None, off=0):
        w, keep = WeightsC(), []
        for f, _ in WeightsC._fields_:
            at = 0x10000 + (off if f == name else 0)
            if f in arrays:
                keep.append((C.c_void_p * L)(0x10000, at))
                setattr(w, f, C.cast(keep[-1], _PP))
            else:
                setattr(w, f, at)
        ctx = C.c_void_p()
        return lib.hydra_create(C.byref(ctx), C.byref(mc), C.byref(hc), C.byref(tc), C.byref(w), 0x100000, 1 << 40)

    assert create() == 5 and create("head_b1", 4) == 5                    # past the checks, as far as the missing device
    for name in ("embed", "final_norm", "attn_norm", "ffn_norm", "pfx_attn_norm", "pfx_ffn_norm"):
        assert create(name, 4) == 1, name


def test_workspace_of_a_float_model_holds_what_its_kernels_use():
    """The float model's products leave their sums where they are wanted: no normed rows, no gathered head inputs, and partial sums for vocabulary projections only.
    Sizes grow accordingly (256-byte steps aside; 64 sequences, so no row count is rounded up)."""
    import ctypes as C
    from paper_2402_05109_b200.binding import lib, HeadCfgC, ModelCfgC, TreeCfgC
    B, S, V, T = 64, 64, 128, 2

    def size(d=256, ffn=512, K=3):
        n = lib.hydra_workspace_bytes(C.byref(ModelCfgC(1, d, d // 64, 64, ffn, V, 1e-6, 1e4, 0, B, S)), C.byref(HeadCfgC(K, 1, 0, 1)),
                                      C.byref(TreeCfgC(T, (C.c_int32 * T)(-1, 0))))
        assert n > 0
        return n
    R, RH, slack, base = 64 * B, B, 64 * 256, size()       # rows of a prompt pass and of a draft level
    # activations after SiLU
    assert size(ffn=4096) - base <= 4 * R * (4096 - 512) + slack
    # hidden rows of the last step (and the tree's path table)
    assert size(K=60) - base <= 4 * 57 * (B * 256 + T) + slack
    # K and V; residual rows, q, hidden rows and attention output; last step's rows, h' and the heads' two row buffers; attention's partial rows
    att = lib.hydra_attention_scratch_bytes(B, 64, 8, 64, S) - lib.hydra_attention_scratch_bytes(B, 64, 4, 64, S)
    assert size(d=512) - base <= 4 * 256 * (2 * B * S + 4 * R + B * 4 + B + 2 * RH) + att + slack
