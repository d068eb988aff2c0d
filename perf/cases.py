"""What this library's users have it do, as measurable cases.

A cache that keeps its keys and values as sparse codes calls the codec in a few ways: whole
prompts are encoded layer by layer (prefill), a decoding step encodes the handful of rows it
adds and attends to the coded cache, codes are turned back into rows (on the device, or from
host memory), and a layer's dictionary is trained on batches of rows.  `listed()` holds one or
two cases of each at sizes of `workloads.py` / `bench_configs.py` or odd ones beside them;
`draw()` gives more of the same ranges.  Every case goes through the public entry points of
`paper_2412_11741_b200`.
"""
from __future__ import annotations

import math
import weakref

import torch

import paper_2412_11741_b200 as csr

_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
_MODES = {"fast": csr.CSR_MODE_BF16_FAST, "exact": csr.CSR_MODE_FP32_EXACT}
_MAX_FLOPS = 2.0 * (1 << 21) * 8192 * 128 * 16           # the largest listed case


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------

def listed():
    return [
        # one layer's decoding step of one sequence with 8 KV heads and 4 query heads per KV head: the 8 new
        # K rows and 8 new V rows are encoded into their places in the cache, then attention
        # over everything cached so far; the smallest calls, where latency counts
        dict(name="decode_layer", kind="decode", B=8, H=4, T=4099, N=8192, d=128, s=16, q="bf16", encode=True),
        # attention of one layer over a long batch (8 sequences x 8 KV heads x 16384 tokens)
        dict(name="attention_long", kind="decode", B=64, H=4, T=16384, N=8192, d=128, s=16, q="f32", encode=False),
        # a short prompt in fp32 against a small dictionary that has no handle (the tiny configuration)
        dict(name="tiny_f32", kind="encode", mode="fast", M=4160, N=1024, d=128, s=8, x="f32", coef="f16", handle=False),
        # one layer's prefill: 32 heads x 4096 tokens x {K, V}
        dict(name="prefill_layer", kind="encode", mode="fast", M=262144, N=4096, d=128, s=8, x="bf16", coef="f16", handle=True),
        # the long-context batch of the benchmark, encoded and restored; the largest case
        dict(name="gqa_long_roundtrip", kind="roundtrip", M=1 << 21, N=8192, d=128, s=16, x="bf16"),
        # 64-channel heads (or half-head chunks) at sparsity 6, an odd number of rows, a dictionary with online
        # atoms appended (odd size, rebuilt for each prompt, so no handle), fp16 rows
        dict(name="head64_ragged", kind="encode", mode="fast", M=100003, N=5001, d=64, s=6, x="f16", coef="f16", handle=False),
        # prefill in the exact mode, fp32 rows and coefficients (calibration, verification)
        dict(name="exact_prefill", kind="encode", mode="exact", M=100000, N=4096, d=128, s=8, x="f32", coef="f32", handle=False),
        # the rows one decoding step of 8 sequences adds, in the exact mode
        dict(name="exact_decode", kind="encode", mode="exact", M=128, N=8192, d=128, s=16, x="bf16", coef="f16", handle=False),
        # codes back into rows: a million vectors from a prepared dictionary
        dict(name="restore", kind="restore", M=1 << 20, N=8192, d=128, s=8, out="bf16", coef="f16", handle=True),
        # the same for a ragged prompt and a dictionary with online atoms (fp32 atoms, no handle), fp16 rows out
        dict(name="restore_ragged", kind="restore", M=77777, N=5001, d=128, s=6, out="f16", coef="f16", handle=False),
        # one step of dictionary training in its default (exact) mode
        dict(name="train_step", kind="train", mode="exact", M=65536, N=8192, d=128, s=8, x="bf16"),
        # a cache offloaded to host memory: rows encoded from pinned host buffers, codes restored into them
        dict(name="host_roundtrip", kind="host", M=200003, N=4096, d=128, s=8, x="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "encode", "encode", "exact", "exact", "restore", "restore", "roundtrip", "train", "host"])
    d = rng.choice([128, 128, 64])
    s = rng.choice([4, 6, 8, 8, 12, 16, 16, 24, 32])
    N = _log_int(rng, 512, 16384)
    handle = rng.random() < 0.6
    x = rng.choice(["bf16", "bf16", "f16", "f32"])
    if kind == "decode":
        B, H = rng.choice([4, 8, 8, 16, 32, 64]), rng.choice([1, 2, 4, 4, 8])
        s = rng.choice([4, 6, 8, 16])
        T = min(_log_int(rng, 300, 40000), (1 << 24) // (B * s))
        return dict(kind="decode", B=B, H=H, T=T, N=min(N, 8192), d=d, s=s, q=rng.choice(["bf16", "f32"]), encode=rng.random() < 0.5)
    if kind in ("encode", "exact"):
        exact = kind == "exact"
        M = _log_int(rng, 16, (1 << 18) if exact else (1 << 20))
        M = max(16, min(M, int((0.2 if exact else 1.0) * _MAX_FLOPS / (2.0 * N * d * s))))
        return dict(kind="encode", mode="exact" if exact else "fast", M=M, N=N, d=d, s=s, x=x,
                    coef=rng.choice(["f16", "f16", "f32"]), handle=handle and not exact)
    if kind == "restore":
        return dict(kind="restore", M=_log_int(rng, 1000, 1 << 20), N=N, d=d, s=s, out=x, coef=rng.choice(["f16", "f16", "f32"]), handle=handle)
    if kind == "roundtrip":
        M = max(4096, min(_log_int(rng, 4096, 1 << 20), int(_MAX_FLOPS / (2.0 * N * d * s))))
        return dict(kind="roundtrip", M=M, N=N, d=d, s=s, x=x)
    if kind == "train":
        return dict(kind="train", mode=rng.choice(["exact", "fast"]), M=_log_int(rng, 2000, 131072), N=min(N, 8192), d=d,
                    s=rng.choice([4, 8]), x=rng.choice(["bf16", "f32"]))
    return dict(kind="host", M=_log_int(rng, 4096, 1 << 19), N=min(N, 8192), d=d, s=rng.choice([4, 8, 16]), x=rng.choice(["bf16", "f16"]))


# ---------------------------------------------------------------------------------------
# inputs: Gaussian stand-ins of key and value rows, as in workloads.py
# ---------------------------------------------------------------------------------------

def _channels(g, d, heads=8):
    """Four outlier channels for each of `heads` heads, as the columns of a 0/1 mask."""
    return torch.zeros(heads, d, device="cuda").scatter_(1, torch.rand(heads, d, device="cuda", generator=g).argsort(1)[:, :4], 1.0)


def _rows(g, M, d, mask, keys):
    """M rows: the first `keys` key-like (outlier channels times 10, head by head), the rest N(0, 1)."""
    X = torch.randn(M, d, device="cuda", generator=g)
    if keys:
        per_head = -(-keys // mask.shape[0])
        for h in range(mask.shape[0]):
            X[h * per_head:min(keys, (h + 1) * per_head)] *= 1.0 + 9.0 * mask[h]
    return X


def _dictionary(g, N, d, mask, keys):
    return torch.nn.functional.normalize(_rows(g, N, d, mask, keys), dim=1).contiguous()


def _codes(g, rows, N, s, coef_dtype):
    """Codes as an encoder leaves them: atoms of uneven popularity, coefficients that fall with the iteration."""
    order = torch.randperm(N, device="cuda", generator=g).to(torch.int32)
    pick = (torch.rand(rows, s, device="cuda", generator=g).pow_(1.5) * N).to(torch.int64).clamp_(max=N - 1)
    idx = order[pick].to(torch.int16).view(torch.uint16)
    coef = torch.randn(rows, s, device="cuda", generator=g).mul_(0.15)
    coef = (coef + torch.where(torch.rand(rows, s, device="cuda", generator=g) < 0.5, -1.0, 1.0)) * 4.2
    coef *= 0.93 ** torch.arange(s, device="cuda", dtype=torch.float32)
    return idx, coef.to(coef_dtype).contiguous()


class _Dict:
    """A dictionary's prepared handle, freed with the object."""

    def __init__(self, D):
        self.handle = csr.csr_dict_create(D)
        weakref.finalize(self, csr.csr_dict_destroy, self.handle)


def _handle(st):
    return st["dict"].handle if st["dict"] is not None else None


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind, N, d, s = case["kind"], case["N"], case["d"], case["s"]
    mask = _channels(g, d)
    st = {"case": case, "dict": None}
    if kind == "decode":
        B, H, T = case["B"], case["H"], case["T"]
        st["Dk"], st["Dv"] = _dictionary(g, N, d, mask, N), _dictionary(g, N, d, mask, 0)
        for side in ("k", "v"):
            idx, coef = _codes(g, B * T, N, s, torch.float16)
            st[side + "_idx"], st[side + "_coef"] = idx.view(B, T, s), coef.view(B, T, s)
        st["Q"] = torch.randn(B, H, d, device="cuda", generator=g).to(_DTYPES[case["q"]])
        st["weights"] = torch.empty(B, H, T, device="cuda")
        st["out"] = torch.empty(B, H, d, device="cuda")
        if case["encode"]:
            st["k_new"] = _rows(g, B, d, mask, B).to(torch.bfloat16)
            st["v_new"] = _rows(g, B, d, mask, 0).to(torch.bfloat16)
            st["dict_k"], st["dict_v"] = _Dict(st["Dk"]), _Dict(st["Dv"])
        return st
    M = case["M"]
    st["D"] = _dictionary(g, N, d, mask, N // 2)
    if kind == "restore":
        st["idx"], st["coef"] = _codes(g, M, N, s, _DTYPES[case["coef"]])
        st["X_hat"] = torch.empty(M, d, dtype=_DTYPES[case["out"]], device="cuda")
        if case["handle"]:
            st["dict"] = _Dict(st["D"])
        return st
    st["X"] = _rows(g, M, d, mask, M // 2).to(_DTYPES[case["x"]])
    if kind == "train":
        st["losses"] = torch.empty(2, dtype=torch.float64, device="cuda")
        return st
    if kind == "encode":
        st["idx"] = torch.empty(M, s, dtype=torch.uint16, device="cuda")
        st["coef"] = torch.empty(M, s, dtype=_DTYPES[case["coef"]], device="cuda")
        if case["handle"]:
            st["dict"] = _Dict(st["D"])
        return st
    st["dict"] = _Dict(st["D"])
    where = dict(device="cuda") if kind == "roundtrip" else dict(pin_memory=True)
    st["idx"] = torch.empty(M, s, dtype=torch.uint16, **where)
    st["coef"] = torch.empty(M, s, dtype=torch.float16, **where)
    st["X_hat"] = torch.empty(M, d, dtype=st["X"].dtype, **where)
    if kind == "host":
        X = torch.empty(M, d, dtype=st["X"].dtype, pin_memory=True)
        st["X"] = X.copy_(st["X"])
    return st


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------

def _bits(t):
    """Indices with a signed element type of the same bits: few torch operations take uint16."""
    return t.view(torch.int16) if t.dtype == torch.uint16 else t


def run(st):
    case = st["case"]
    kind, s = case["kind"], case["s"]
    if kind == "decode":
        if case["encode"]:
            # the new rows' codes go to the last token of every stream
            new = [(st[k + "_idx"][:, -1], st[k + "_coef"][:, -1]) for k in ("k", "v")]
            csr.csr_encode_grouped([(st["Dk"], st["k_new"], s, *new[0], st["dict_k"].handle),
                                    (st["Dv"], st["v_new"], s, *new[1], st["dict_v"].handle)])
        out, weights = csr.csr_decode_attention(st["Dk"], st["Dv"], st["Q"], st["k_idx"], st["k_coef"], st["v_idx"], st["v_coef"],
                                                1.0 / math.sqrt(case["d"]), weights=st["weights"], out=st["out"])
        return (out, weights, *[_bits(t) for t in new[0] + new[1]]) if case["encode"] else (out, weights)
    if kind == "encode":
        idx, coef = csr.csr_encode_ex(st["D"], st["X"], s, mode=_MODES[case["mode"]], out_idx=st["idx"], out_coef=st["coef"], dict=_handle(st))
        return _bits(idx), coef
    if kind == "restore":
        return csr.csr_reconstruct_ex(st["D"], st["idx"], st["coef"], X_hat=st["X_hat"], dict=_handle(st))
    if kind == "roundtrip":
        csr.csr_encode_ex(st["D"], st["X"], s, out_idx=st["idx"], out_coef=st["coef"], dict=_handle(st))
        csr.csr_reconstruct_ex(st["D"], st["idx"], st["coef"], X_hat=st["X_hat"], dict=_handle(st))
        return _bits(st["idx"]), st["coef"], st["X_hat"]
    if kind == "host":
        csr.csr_encode_host(st["D"], st["X"], s, st["idx"], st["coef"], dict=_handle(st))
        csr.csr_reconstruct_host(st["D"], st["idx"], st["coef"], st["X_hat"], dict=_handle(st))
        return _bits(st["idx"]), st["coef"], st["X_hat"]
    if kind == "train":
        csr.csr_dict_train_step(st["D"], st["X"], s, 1e-5, 0.1, mode=_MODES[case["mode"]], losses=st["losses"])
        return st["D"], st["losses"]
    raise ValueError(kind)


# ---------------------------------------------------------------------------------------
# what a pass cannot do without, and how close two correct results are
# ---------------------------------------------------------------------------------------

def work(case):
    kind, N, d, s = case["kind"], case["N"], case["d"], case["s"]
    size = {"f32": 4, "bf16": 2, "f16": 2}
    if kind == "decode":
        B, H, T = case["B"], case["H"], case["T"]
        nbytes = 2 * B * T * s * 4 + B * H * T * 4 + B * H * d * (size[case["q"]] + 4) + 2 * N * d * 4
        flops = 2.0 * B * H * (2 * T * s + 2 * N * d)
        if case["encode"]:
            nbytes += 2 * B * d * 2
            flops += 2 * 2.0 * B * N * d * s
        return {"bytes": nbytes, "flops": flops}
    M = case["M"]
    pursuit = 2.0 * M * N * d * s                        # every correlation of every iteration
    if kind == "encode":
        return {"bytes": M * d * size[case["x"]] + M * s * (2 + size[case["coef"]]) + N * d * (2 if case["handle"] else 4), "flops": pursuit}
    if kind == "restore":
        return {"bytes": M * s * (2 + size[case["coef"]]) + M * d * size[case["out"]] + N * d * (2 if case["handle"] else 4), "flops": 2.0 * M * s * d}
    if kind in ("roundtrip", "host"):
        return {"bytes": 2 * M * d * size[case["x"]] + 2 * M * s * 4 + 2 * N * d * 2, "flops": pursuit + 2.0 * M * s * d}
    # training: the pursuit, the loss gradient of the picked atoms, the two N x N products of the diversity term
    return {"bytes": M * d * size[case["x"]] + 2 * N * d * 4 + 16, "flops": pursuit + 4.0 * M * s * d + 4.0 * N * N * d}


def tolerance(case):
    kind = case["kind"]
    if kind == "decode":
        # Measured against fp64: weights 3e-7, outputs 6e-5 (the value sums are kept on a fixed-point grid).
        return {"rel": 2.5e-4, "max": 1e-3, "differ": 0.003}
    if kind == "restore":
        # The atoms' values are given (fp32, or the handle's fp16), so only the order of at most 32 fp32
        # additions is free: measured against fp64 sums 4e-6 of fp16 results (one-ulp roundings).
        return {"f32": {"rel": 1e-6, "max": 2e-5}, "f16": {"rel": 2e-5, "max": 2e-3}, "bf16": {"rel": 1e-4, "max": 1.6e-2}}[case["out"]]
    if kind == "train":
        # D and both losses; atomic fp32 sums differ by 3e-8 from run to run, L_div by 1e-6.
        return {"rel": 1e-5, "max": 1e-3}
    if kind == "encode" and case["mode"] == "exact":
        # fp64 arithmetic behind every pick: two encoders of this library return the same codes.
        return {"rel": 1e-6, "max": 1e-3, "differ": 1e-5}
    # The fast mode may resolve correlations that agree to 2^-15 either way: the library's own arg-max
    # variants differ in up to 0.08 % of the indices (every later pick of such a row among them).
    return {"rel": 0.03, "max": 0.99, "differ": 0.003}


# ---------------------------------------------------------------------------------------
# the same results from 64-bit sums in plain torch
# ---------------------------------------------------------------------------------------

def _pursuit64(D, X, s):
    """Matching pursuit of the rows of X over the atoms of D, all in 64 bits."""
    D, idx, coef = D.double(), [], []
    for x in X.split(max(64, (1 << 26) // D.shape[0])):
        R, picks, cs = x.double(), [], []
        for _ in range(s):
            corr = R @ D.T
            n = corr.abs().argmax(dim=1)
            c = corr.gather(1, n[:, None])
            R = R - c * D[n]
            picks.append(n)
            cs.append(c)
        idx.append(torch.stack(picks, 1))
        coef.append(torch.cat(cs, 1))
    return torch.cat(idx), torch.cat(coef)


def _rows64(D, idx, coef, group=1 << 16):
    """The rows that codes stand for."""
    return torch.cat([(c.double()[:, :, None] * D[i]).sum(1) for i, c in zip(idx.split(group), coef.split(group))])


def _ints(idx):
    return idx.view(torch.int16).long() & 0xFFFF


def exact(case, seed):
    """run()'s outputs in 64 bits.  None where they hang on the fast mode's picks: it resolves near-ties
    in 16 bits, either way, and every later number of such a row follows from its picks."""
    kind, s = case["kind"], case["s"]
    if kind in ("roundtrip", "host") or case.get("encode") is True or (kind in ("encode", "train") and case["mode"] == "fast"):
        return None
    st = prepare(case, seed)
    if kind == "decode":
        B, T, d = case["B"], case["T"], case["d"]
        Dk, Dv, Q = st["Dk"].double(), st["Dv"].double(), st["Q"].double()
        out, weights = [], []
        for b in range(B):
            K = _rows64(Dk, _ints(st["k_idx"][b]), st["k_coef"][b], 1 << 14)
            w = torch.softmax(Q[b] @ K.T / math.sqrt(d), dim=-1)
            weights.append(w)
            out.append(w @ _rows64(Dv, _ints(st["v_idx"][b]), st["v_coef"][b], 1 << 14))
        return torch.stack(out), torch.stack(weights)
    if kind == "restore":
        D = st["D"].half().double() if case["handle"] else st["D"].double()
        return _rows64(D, _ints(st["idx"]), st["coef"], 1 << 14)
    idx, coef = _pursuit64(st["D"], st["X"], s)
    if kind == "encode":
        return idx, coef
    # one step of gradient descent on ||X - X_hat||^2 + beta ||D D^T - I||^2 / N^2, then unit atoms
    D, N = st["D"].double(), case["N"]
    grad, loss = torch.zeros_like(D), 0.0
    for x, i, c in zip(st["X"].split(1 << 14), idx.split(1 << 14), coef.split(1 << 14)):
        e = x.double() - _rows64(D, i, c)
        loss = loss + (e * e).sum()
        grad.index_add_(0, i.reshape(-1), (-2.0 * c[:, :, None] * e[:, None, :]).reshape(-1, D.shape[1]))
    G = D @ D.T - torch.eye(N, dtype=D.dtype, device=D.device)
    W = D - 1e-5 * (grad + 0.1 * 4.0 / N ** 2 * (G @ D))
    return torch.nn.functional.normalize(W, dim=1), torch.stack([loss, (G * G).sum() / N ** 2])
