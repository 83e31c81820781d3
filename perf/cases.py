"""Performance cases: what a program that serves a decoder with libhydra has the library do.

Four kinds of pass:
  generate   one request (or one batch of requests): the prompt pass, then a fixed number of decode steps (draft the tree,
             verify it, accept, compact the cache), the emitted tokens collected after every step;
  prompt     the prompt pass alone (time to first token, prefix caching, scoring);
  verify     one verification of candidates that the caller brings (its own drafter), with the logits of every row;
  gemm       the stand-alone allocation-free GEMM, the smallest call of the library.

Models are random, with one structure planted into embedding, vocabulary projection and draft heads so that tokens are chosen
with the clear margins of a trained model and part of the drafts is accepted (see `weights`).  Shapes are those of the
benchmark configurations: the tiny float decoder, the 7B and the 13B shape at full depth, the 33B shape at 20 of its 60 layers
(so that several states fit one GPU), plus generic widths in `draw`.
"""
import math
from types import SimpleNamespace

import torch

from paper_2402_05109_b200 import Hydra, gemm_noalloc
from paper_2402_05109_b200.tree_search import grow_trees, to_parent_list

_TINY = dict(dtype="fp32", layers=2, d=256, heads=4, ffn=688, vocab=1024, planes=1)
_7B = dict(dtype="bf16", layers=32, d=4096, heads=32, ffn=11008, vocab=32000, planes=2)
_13B = dict(dtype="bf16", layers=40, d=5120, heads=40, ffn=13824, vocab=32000, planes=2)
_33B = dict(dtype="bf16", layers=20, d=6656, heads=52, ffn=17920, vocab=32000, planes=2)
# Draft models: Hydra++ (four-layer heads behind the prefix layer), plain Hydra and Medusa (independent) heads
_HYDRAPP = dict(K=4, mlp=4, prefix=True, medusa=False)
_HYDRA = dict(K=4, mlp=1, prefix=False, medusa=False)
_MEDUSA = dict(K=4, mlp=1, prefix=False, medusa=True)


def _generate(name, model, draft, **kw):
    return dict(name=name, kind="generate", **model, **draft, **dict(dict(buffers="kept", typical=False), **kw))


def listed():
    return [
        # a toy model in float: every call is launch latency; the tokens are kept as the step returns them
        _generate("tiny_fp32", _TINY, dict(_HYDRA, K=3), batch=1, lo=32, hi=32, tree=15, steps=8, buffers="fresh"),
        # one chat request at the quoted configuration
        _generate("7b_chat", _7B, _HYDRAPP, batch=1, lo=512, hi=512, tree=63, steps=32),
        # plain autoregressive decoding (root-only tree): the baseline that speculation is compared with
        _generate("7b_autoregressive", _7B, _HYDRA, batch=1, lo=129, hi=129, tree=0, steps=32, buffers="fresh"),
        # Medusa heads, the other baseline, on a mid-size tree
        _generate("7b_medusa", _7B, _MEDUSA, batch=1, lo=77, hi=77, tree=31, steps=16),
        # sampling from a small batch with the typical criterion
        _generate("7b_typical_b2", _7B, _HYDRAPP, batch=2, lo=128, hi=1024, tree=63, steps=12, typical=True),
        # batched serving with the small tree that suits a batch, single-plane cache
        _generate("7b_b4_small_tree", dict(_7B, planes=1), _HYDRAPP, batch=4, lo=128, hi=1024, tree=7, steps=16),
        # batched serving with the full tree: ragged prompts
        _generate("7b_b8_ragged", _7B, _HYDRAPP, batch=8, lo=128, hi=1024, tree=63, steps=8),
        # a long prompt on the 13B shape
        _generate("13b_long", _13B, _HYDRAPP, batch=1, lo=2048, hi=2048, tree=63, steps=16),
        # the widest model, four long prompts
        _generate("33b_b4", _33B, _HYDRAPP, batch=4, lo=1024, hi=1024, tree=63, steps=6),
        # first token of a short ragged batch: the prompt pass alone
        dict(name="7b_prompt_b3", kind="prompt", **_7B, **_HYDRAPP, batch=3, lo=50, hi=400, tree=63),
        # candidates from the caller's own drafter, scored with logits
        dict(name="7b_verify_47", kind="verify", **_7B, **_HYDRA, batch=1, lo=700, hi=700, tree=46),
        # a projection of a few rows inside a plugin that may not allocate
        dict(name="gemm_noalloc", kind="gemm", m=11, n=4096, k=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["generate"] * 7 + ["prompt", "verify", "gemm"])
    if kind == "gemm":
        # the partial sums of the call have to fit the library's 8 MiB
        k = 64 * _log(rng, 4, 172)
        m = _log(rng, 1, 64)
        n = 128 * _log(rng, 2, max(2, min(86, (8 << 20) // (m * 512 * 12))))
        return dict(kind="gemm", m=m, n=n, k=k)
    if rng.random() < 0.15:
        model = dict(_TINY, layers=rng.randint(1, 4))
    else:
        # a benchmark width or any other, with enough layers for at most 7 billion parameters
        model = dict(rng.choice([_7B, _7B, _13B, _33B]))
        if rng.random() < 0.4:
            d = 128 * _log(rng, 6, 52)
            hd = rng.choice([128, 128, 64])
            model.update(d=d, heads=d // hd, ffn=64 * int(d * rng.uniform(2.5, 3.5) / 64), vocab=128 * _log(rng, 16, 400))
        per_layer = 4 * model["d"] ** 2 + 3 * model["d"] * model["ffn"]
        model.update(layers=_log(rng, 2, max(2, min(40, int(7e9 / per_layer)))), planes=rng.choice([2, 2, 1]))
    draft = dict(rng.choice([_HYDRAPP, _HYDRAPP, _HYDRA, _MEDUSA]))
    draft.update(K=rng.randint(2, 5), mlp=rng.randint(1, 4))
    batch = rng.choice([1, 1, 2, 3, 4, 5, 6, 8])
    hi = _log(rng, 24, 2500 if batch == 1 else 1100)
    lo = hi if rng.random() < 0.5 else max(8, hi // 4)
    case = dict(kind=kind, **model, **draft, batch=batch, lo=lo, hi=hi, tree=rng.choice([0, 3, 7, 15, 31, 47, 63, rng.randint(1, 63)]))
    if kind == "generate":
        case.update(steps=rng.randint(4, 10), buffers=rng.choice(["kept", "fresh"]), typical=rng.random() < 0.25)
    return case


def _lens(case):
    """Prompt lengths of the sequences: spread over [lo, hi], the first the longest."""
    b, lo, hi = case["batch"], case["lo"], case["hi"]
    return [hi - (hi - lo) * i // max(1, b - 1) - (i * 37) % max(1, min(64, (hi - lo) // 8)) for i in range(b)]


def _rank_prob(depth, rank):
    return (0.70, 0.55, 0.45, 0.38, 0.33)[depth - 1] * 0.55 * 0.45 ** rank


def _tree(case):
    return [-1] if case["tree"] == 0 else to_parent_list(grow_trees(case["tree"], case["K"], _rank_prob)[-1])


def weights(case, gen):
    """Random weights on the GPU.  Linear layers are N(0, 0.02); the two projections back into the residual stream are scaled
    so that all layers together weigh about as much as the token itself.  The planted structure: every token v has a successor
    next(v); its embedding is [a(v) ; b(v)] with a random code a(v) and b(v) = a(next(v)), for 30 % of the tokens a wrong code
    instead; the vocabulary row of next(v) points along a(v), so the base model continues v with next(v); the heads read the b
    half of the token before the last, so a draft is right after the 70 % of tokens whose b is."""
    d, f, V, L, K = case["d"], case["ffn"], case["vocab"], case["layers"], case["K"]
    dt = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    half = d // 2

    def normal(*shape, std=0.02):
        return torch.empty(*shape, dtype=dt, device="cuda").normal_(0.0, std, generator=gen)

    one = torch.ones(d, dtype=dt, device="cuda")
    s = 0.02 * math.sqrt(d)                                  # size of a normed row's projection
    back_o = 1.0 / (math.sqrt(2 * L * d) * s * 0.5)          # (more would let the averages over the context drown the tokens)
    back_f = 1.0 / (math.sqrt(2 * L * f) * 0.55 * s * s)

    def layer(p):
        return {p + "attn_norm": one, p + "wqkv": normal(3 * d, d), p + "wo": normal(d, d, std=back_o),
                p + "ffn_norm": one, p + "w_gate_up": normal(2 * f, d), p + "w_down": normal(d, f, std=back_f)}

    code = normal(V, half, std=1.0)
    nxt = torch.randperm(V, generator=gen, device="cuda")
    hint = torch.where(torch.rand(V, generator=gen, device="cuda") < 0.3, torch.randperm(V, generator=gen, device="cuda"), nxt)
    lm = normal(V, d)
    lm[nxt, :half] += code * (20.0 / min(half, 2048))
    w = {"embed": torch.cat([code, code[hint]], 1).contiguous(), "lm_head": lm, "final_norm": one}
    for i in range(L):
        w.update(layer("L%d." % i))
    if case["prefix"]:
        w.update(layer("P."))
    eye = 4.0 * torch.eye(half, dtype=dt, device="cuda")
    for i in range(1, K + 1):
        w1 = normal(d, d if case["medusa"] else (i + 1) * d)
        if not case["medusa"] or i == 1:
            at = 0 if case["medusa"] else (i - 1) * d
            w1[:half, at + half:at + d] += eye               # the token before the last on the path (for head 1: the hidden state)
        w["H%d.w1" % i] = w1
        w["H%d.b1" % i] = normal(d)
        if case["mlp"] > 1:
            w["H%d.wr" % i] = normal(case["mlp"] - 1, d, d, std=0.01)
            w["H%d.br" % i] = normal(case["mlp"] - 1, d)
    return w


_stream = None


def _serving_stream():
    """The stream of the serving loop: steps are replayed as graphs only on a stream of the caller's own."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        x = torch.empty(m, k, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
        w = torch.empty(n, k, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=gen)
        return SimpleNamespace(case=case, x=x, w=w, out=torch.empty(m, n, device="cuda"),
                               status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    parent = _tree(case)
    T, K, B = len(parent), case["K"], case["batch"]
    lens = _lens(case)
    model = SimpleNamespace(n_layers=case["layers"], d_model=case["d"], n_heads=case["heads"], head_dim=case["d"] // case["heads"],
                            d_ffn=case["ffn"], vocab=case["vocab"], rms_eps=1e-6, rope_theta=1e4, dtype=case["dtype"], kv_planes=case["planes"])
    head = SimpleNamespace(n_heads=K, n_mlp_layers=case["mlp"], prefix_attn=case["prefix"], has_bias=True, medusa=case["medusa"])
    max_seq = max(lens) + case.get("steps", 1) * (K + 1) + T
    s = SimpleNamespace(case=case, T=T, K=K)
    s.h = Hydra(model, head, parent, weights(case, gen), B, max_seq)
    s.prompts = [torch.randint(0, case["vocab"], (n,), dtype=torch.int32, device="cuda", generator=gen) for n in lens]
    s.stream = _serving_stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s.stream):
        if case["kind"] == "generate":
            s.n_acc = torch.empty(B, dtype=torch.int32, device="cuda")
            s.out = torch.empty(B, K + 1, dtype=torch.int32, device="cuda")
            if case["typical"]:
                s.u = torch.empty(B, device="cuda")
                s.draws = torch.rand(case["steps"], B, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed + 1))
                s.h.set_acceptance(1, tau=0.7, eps=0.15, alpha=math.sqrt(0.15), u=s.u)
        if case["kind"] == "verify":
            s.h.prefill(s.prompts)
            s.candidates = torch.randint(0, case["vocab"], (B, T), dtype=torch.int32, device="cuda", generator=gen)
    return s


def run(s):
    case = s.case
    if case["kind"] == "gemm":
        gemm_noalloc(s.x, s.w, s.out, s.status)
        return s.out
    h = s.h
    with torch.cuda.stream(s.stream):
        if case["kind"] == "verify":
            amax, logits = h.verify(s.candidates, want_logits=True)
            return logits
        h.prefill(s.prompts)
        if case["kind"] == "prompt":
            out = dict(root=h.get_buffer("ROOT_TOK"), length=h.get_buffer("LEN"), hidden=h.get_buffer("H_NEW"))
            if case["prefix"]:
                out["prefix_cache"] = h.get_buffer("KV_PREFIX")
            return out
        tokens, accepted = [], []
        for i in range(case["steps"]):
            if case["typical"]:
                s.u.copy_(s.draws[i])
            if case["buffers"] == "fresh":
                n_acc, out = h.step()
                tokens.append(out)
                accepted.append(n_acc)
            else:
                h.step(s.n_acc, s.out)
                tokens.append(s.out.clone())
                accepted.append(s.n_acc.clone())
        return dict(tokens=torch.stack(tokens), accepted=torch.stack(accepted), length=h.get_buffer("LEN"),
                    root=h.get_buffer("ROOT_TOK"), hidden=h.get_buffer("H_NEW"), new=h.get_buffer("N_NEW"))


def work(case):
    """Weights once per sequential pass over them (the prompt pass; every draft and every verification), every live cache row
    read once and every new one written; two operations per weight and row that has to go through it."""
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=2.0 * (m * k + n * k) + 4.0 * m * n, flops=2.0 * m * n * k)
    d, f, V, L, K, B = case["d"], case["ffn"], case["vocab"], case["layers"], case["K"], case["batch"]
    es = 4 if case["dtype"] == "fp32" else 2
    parent, lens = _tree(case), _lens(case)
    T = len(parent)
    row = 2.0 * es * case["planes"] * d                      # K and V of one position and layer
    layer = 4.0 * d * d + 3.0 * d * f
    pfx = layer if case["prefix"] else 0.0
    base, head = L * layer, V * d
    tokens = float(sum(lens))
    attn = lambda rows, n: 4.0 * d * rows * n                # scores and weighted sum of `rows` query rows over n keys
    prompt = dict(bytes=es * (base + pfx + head) + tokens * row * (L + (case["prefix"] and 1)),
                  flops=2.0 * tokens * (base + pfx) + 2.0 * B * head + sum((L + (case["prefix"] and 1)) * attn(n, n / 2) for n in lens))
    verify = dict(bytes=es * (base + head) + L * row * (tokens + 2.0 * B * T), flops=2.0 * B * T * (base + head) + L * sum(attn(T, n + T) for n in lens))
    if case["kind"] == "prompt":
        return prompt
    if case["kind"] == "verify":
        verify["bytes"] += 4.0 * B * T * V
        return verify
    depth = [0] * T
    for i in range(1, T):
        depth[i] = depth[parent[i]] + 1
    draft = dict(bytes=es * pfx, flops=2.0 * B * 2 * pfx)
    if case["prefix"]:
        draft["bytes"] += tokens * row
        draft["flops"] += sum(attn(2, n) for n in lens)
    for lvl in range(1, max(depth) + 1):
        parents = len({parent[i] for i in range(T) if depth[i] == lvl})
        mlp = ((1 if case["medusa"] else lvl + 1) + case["mlp"] - 1.0) * d * d + head
        draft["bytes"] += es * mlp
        draft["flops"] += 2.0 * B * (1 if case["medusa"] else parents) * mlp
    return {k: prompt[k] + case["steps"] * (draft[k] + verify[k]) for k in ("bytes", "flops")}


def tolerance(case):
    """Whole tokens are decided with wide margins (see `weights`).  Floats: 32-bit sums in the float model and in the stand-alone
    GEMM (other split counts of the sums: 3e-7); in the bfloat16 models activations are rounded to two bfloat16 planes (16 bits)
    between the layers: other split counts moved the results by up to 1e-4 (two cache planes) and 5e-4 (one)."""
    if case["kind"] == "gemm" or case["dtype"] == "fp32":
        return dict(rel=1e-5, max=1e-3, differ=0.005)
    return dict(rel=5e-4 if case["planes"] == 2 else 2e-3, max=0.03, differ=0.005)
