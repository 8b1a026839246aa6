"""The calls a user of the library makes, as cases that can be timed and compared.

A serving process runs three kinds of work through `paper_2503_18893_b200.xkv`:

  prefill   `factorize`  xkv_clf_factorize of one cache of one window (Eq. 1), once per prompt, cache and window
            `landmarks`  xkv_build_landmarks with the static outlier chunks (Algorithm 1), once per prompt and window
            `quantize`   xkv_quantize_rtn / xkv_dequantize_rtn: the token bases of a window to 4- or 3-bit codes, the
                         small reconstruction matrices to codes and back (the handle takes them as bf16)
  decode    `decode`     xkv_sr_select, then xkv_sr_reconstruct_attend (with an uncompressed tail of generated tokens:
                         ..._attend_tail), per window or, as a model has to, layer after layer; per token
  dense     `dense`      xkv_dense_attend over an uncompressed cache: the attention of a window that is not compressed

Sizes are those of the benchmark configurations (`synth.config`), of the stress sweep around them, and of real prompts,
which are ragged.  A case is a dict of plain values; `prepare` makes what the program has in hand, `run` is one pass.
"""
from __future__ import annotations

import math

import torch

from paper_2503_18893_b200 import xkv

LLAMA = dict(G=4, H_kv=8, H_q=32, d_h=128)
QWEN = dict(G=4, H_kv=4, H_q=28, d_h=128)
TINY = dict(G=2, H_kv=2, H_q=8, d_h=64)


def _decode(name, heads, T, r_k, r_v, k, batch=1, calls="window", tail=0, bits=16, outliers=0, decay=1.0, select="handle"):
    c = dict(op="decode", T=T, r_k=r_k, r_v=r_v, k=k, batch=batch, calls=calls, tail=tail, bits=bits, outliers=outliers,
             decay=decay, select=select, **heads)
    return dict(name=name, **c) if name else c


def _prefill(name, op, **sizes):
    c = dict(op=op, **sizes)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest model and context: everything is latency and launches
        _decode("decode_tiny_2k", TINY, 2048, 64, 64, 256, decay=0.0),
        # a model's own loop: the queries of layer l+1 exist only after layer l, so every layer is a call of its own
        _decode("decode_32k_by_layer", LLAMA, 32768, 512, 512, 2048, calls="layer"),
        # the headline: one window of an 8B model at 128K, one sequence
        _decode("decode_128k", LLAMA, 131072, 512, 512, 4096),
        # the same with four sequences in the batch
        _decode("decode_128k_batch4", LLAMA, 131072, 512, 512, 4096, batch=4),
        # seven query heads per KV head, eight sequences
        _decode("decode_qwen_64k_batch8", QWEN, 65536, 256, 256, 2048, batch=8, decay=0.8),
        # generation under way on a ragged prompt: ranks 384 / 576 (1 : 1.5), outlier chunks, an uncompressed tail, by layer
        _decode("decode_122k_tail_by_layer", LLAMA, 121873, 384, 576, 2048, calls="layer", tail=1500, outliers=48),
        # bases kept as 4-bit codes
        _decode("decode_128k_4bit", LLAMA, 131072, 512, 512, 4096, bits=4),
        # a large budget over long bases: the reconstruction dominates
        _decode("decode_64k_budget16k", LLAMA, 65536, 1024, 1024, 16384),
        # prefill of one window
        _prefill("landmarks_128k", "landmarks", T=131072, batch=1, G=4, H_kv=8, d_h=128, outliers=48),
        _prefill("factorize_128k", "factorize", T=131072, G=4, d=1024, r=512),
        _prefill("quantize_64k_4bit", "quantize", T=65536, batch=1, r_k=384, r_v=576, G=4, d=1024, bits=4),
        # a window left uncompressed, two sequences of different length
        _prefill("dense_64k_batch2", "dense", T=65536, batch=2, G=4, H_kv=8, H_q=32, d_h=128),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["decode"] * 6 + ["landmarks", "factorize", "quantize", "dense"])
    if op == "decode":
        heads = rng.choice([LLAMA, LLAMA, QWEN, TINY])
        T = _logint(rng, 2048, 131072)
        batch = min(rng.choice([1, 1, 2, 3, 4, 8]), max(1, 524288 // T))
        bits = rng.choice([16, 16, 16, 4, 3])
        step = rng.choice([8, 64]) if bits == 16 else 32
        r_k = max(64, _logint(rng, 64, 128 if heads is TINY else 1024) // step * step)
        r_v = min(1024, r_k * rng.choice([2, 3]) // 2 // step * step)
        k = min(_logint(rng, 256, 16384), T // 2)
        tail = rng.choice([0, 0, _logint(rng, 1, 8192)])
        outliers = rng.choice([0, 0, 48])
        select = "static" if not outliers and batch * T <= 131072 and rng.random() < 0.15 else "handle"
        return _decode(None, heads, T, r_k, r_v, k, batch=batch, calls=rng.choice(["window", "layer"]), tail=tail, bits=bits,
                       outliers=outliers, decay=rng.choice([0.8, 1.0]), select=select)
    if op == "landmarks":
        return _prefill(None, op, T=_logint(rng, 2048, 131072), batch=1, G=rng.choice([2, 4]), H_kv=rng.choice([2, 4, 8]),
                        d_h=rng.choice([64, 128]), outliers=rng.choice([0, 48]))
    if op == "factorize":
        G, d, r = rng.choice([(2, 1024, 256), (4, 1024, 384), (4, 1024, 512), (4, 512, 256), (4, 1024, 576)])
        return _prefill(None, op, T=_logint(rng, 4096, 110000), G=G, d=d, r=r)
    if op == "quantize":
        r_k = 32 * rng.randint(4, 24)
        return _prefill(None, op, T=_logint(rng, 2048, 131072), batch=1, r_k=r_k, r_v=r_k + 32 * rng.randint(0, 8), G=4, d=1024,
                        bits=rng.choice([3, 4]))
    heads = rng.choice([LLAMA, QWEN])
    T = _logint(rng, 2048, 131072)
    return _prefill(None, op, T=T, batch=1 if T > 65536 else rng.choice([1, 2]), **heads)


# ---------------------------------------------------------------------------------------------------------------------
# inputs


def _spectrum(r, rho, decay, Gd, T, noise=0.01):
    """Standard deviation of every column of A = U Sigma: i^-decay over the signal, a flat noise floor behind it, scaled
    so that the keys A B have unit rms."""
    i = torch.arange(r, device="cuda", dtype=torch.float32)
    sig = (i + 1.0) ** (-decay)
    srms2 = float((sig[:rho] ** 2).sum()) / rho
    floor = noise * math.sqrt(srms2) * (1.0 + math.sqrt(Gd / T))
    a = torch.where(i < rho, sig * math.sqrt(Gd / rho), torch.full_like(sig, floor))
    return a * math.sqrt(Gd / float((a ** 2).sum()))


def _randn(shape, g, dtype=torch.bfloat16):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).to(dtype)


def _factors(c, r, g):
    Gd = c["G"] * c["H_kv"] * c["d_h"]
    a = _spectrum(r, max(1, r // 2), c["decay"], Gd, c["T"])
    A = torch.empty((c["batch"], c["T"], r), dtype=torch.bfloat16, device="cuda")
    for b in range(c["batch"]):
        A[b] = (torch.randn((c["T"], r), generator=g, device="cuda") * a).to(torch.bfloat16)
    # rows of B_cat: Gaussian, nearly orthonormal
    B = _randn((c["batch"], c["G"], r, c["H_kv"] * c["d_h"]), g, torch.float32) / math.sqrt(Gd)
    return A, B.to(torch.bfloat16)


def _prepare_decode(c, g):
    G, batch, T, H_kv, H_q, d_h = (c[n] for n in ("G", "batch", "T", "H_kv", "H_q", "d_h"))
    A_k, B_k = _factors(c, c["r_k"], g)
    A_v, B_v = _factors(c, c["r_v"], g)
    n_c = -(-T // 8)
    lm = torch.empty((batch, G, H_kv, n_c, d_h), dtype=torch.bfloat16, device="cuda")
    n_out = c["outliers"]
    out_ids = torch.empty((G, batch, H_kv, n_out), dtype=torch.int32, device="cuda") if n_out else None
    for b in range(batch):
        keys = torch.stack([A_k[b] @ B_k[b, l] for l in range(G)]).unsqueeze(0)
        ids = torch.empty((G, 1, H_kv, n_out), dtype=torch.int32, device="cuda") if n_out else None
        mc = torch.empty((G, 1, H_kv, n_c), dtype=torch.float32, device="cuda") if n_out else None
        xkv.xkv_build_landmarks(keys, lm[b:b + 1], G=G, batch=1, T=T, H_kv=H_kv, d_h=d_h, min_cos=mc, n_outliers=n_out,
                                outliers=ids)
        if n_out:
            out_ids[:, b:b + 1] = ids
        del keys
    grp = xkv.create_from_tensors(A_k, A_v, B_k, B_v, lm, H_kv=H_kv, H_q=H_q, k_max=c["k"])
    if n_out:
        xkv.xkv_group_set_outliers(grp, out_ids, n_out)
    if c["bits"] != 16:
        ck, mk = xkv.xkv_quantize_rtn(A_k, c["bits"])
        cv, mv = xkv.xkv_quantize_rtn(A_v, c["bits"])
        xkv.xkv_group_set_quantized_bases(grp, ck, mk, cv, mv, c["bits"])
    k_cap = (-(-c["k"] // 8) + n_out) * 8
    s = dict(case=c, grp=grp, k_cap=k_cap, lm=lm, q=_randn((G, batch, H_q, d_h), g),
             sel_idx=torch.empty((G, batch, H_kv, k_cap), dtype=torch.int32, device="cuda"),
             sel_cnt=torch.empty((G, batch, H_kv), dtype=torch.int32, device="cuda"),
             out=torch.empty((G, batch, H_q, d_h), dtype=torch.bfloat16, device="cuda"),
             lse=torch.empty((G, batch, H_q), dtype=torch.float32, device="cuda"))
    if c["tail"]:
        cap = c["tail"]
        s["tail_k"] = _randn((G, batch, H_kv, cap, d_h), g)
        s["tail_v"] = _randn((G, batch, H_kv, cap, d_h), g)
        # the sequences of a batch have generated different numbers of tokens
        s["tail_len"] = torch.tensor([max(1, cap - 37 * b) for b in range(batch)], dtype=torch.int32, device="cuda")
        s["ws"] = torch.empty(xkv.xkv_tail_workspace_bytes(grp, cap), dtype=torch.uint8, device="cuda")
    return s


def _run_decode(s):
    c, grp, k_cap = s["case"], s["grp"], s["k_cap"]
    G = c["G"]
    ranges = [(l, l + 1) for l in range(G)] if c["calls"] == "layer" else [(0, G)]
    for lo, hi in ranges:
        if c["select"] == "static":
            xkv.xkv_sr_select_static(G=G, batch=c["batch"], T=c["T"], H_kv=c["H_kv"], H_q=c["H_q"], d_h=c["d_h"],
                                     landmarks=s["lm"], layer_begin=lo, layer_end=hi, q=s["q"], k=c["k"],
                                     sel_idx=s["sel_idx"], sel_cnt=s["sel_cnt"])
        else:
            xkv.xkv_sr_select(grp, lo, hi, s["q"], c["k"], s["sel_idx"], s["sel_cnt"])
        if c["tail"]:
            xkv.xkv_sr_reconstruct_attend_tail(grp, lo, hi, s["q"], s["sel_idx"], s["sel_cnt"], k_cap, s["tail_k"],
                                               s["tail_v"], s["tail_len"], c["tail"], s["ws"], s["out"], s["lse"])
        else:
            xkv.xkv_sr_reconstruct_attend(grp, lo, hi, s["q"], s["sel_idx"], s["sel_cnt"], k_cap, s["out"], s["lse"])
    return {"sel_idx": s["sel_idx"], "sel_cnt": s["sel_cnt"], "out": s["out"], "lse": s["lse"]}


def _cache(T, Gd, r, g):
    """A cache with a token subspace of r/2 directions shared by the layers, spectrum i^-1, and 1 % noise."""
    rho = max(1, r // 2)
    s = torch.arange(1, rho + 1, device="cuda", dtype=torch.float32).rsqrt() ** 2
    Z = (torch.randn((T, rho), generator=g, device="cuda") * s).to(torch.bfloat16)
    M = (torch.randn((rho, Gd), generator=g, device="cuda") / math.sqrt(rho)).to(torch.bfloat16)
    rms = math.sqrt(float((s ** 2).sum()) / rho)
    X = torch.empty((T, Gd), dtype=torch.bfloat16, device="cuda")
    for t in range(0, T, 32768):
        n = min(32768, T - t)
        X[t:t + n] = ((Z[t:t + n] @ M).float() / rms + 0.01 * torch.randn((n, Gd), generator=g, device="cuda")).to(torch.bfloat16)
    return X


def _prepare_factorize(c, g):
    T, Gd, r = c["T"], c["G"] * c["d"], c["r"]
    cfg = xkv.make_clf_config(T=T, G=c["G"], d=c["d"], r=r)
    return dict(case=c, cfg=cfg, X=_cache(T, Gd, r, g), omega=_randn((Gd, xkv.xkv_clf_rank_l(cfg)), g),
                ws=torch.empty(xkv.xkv_clf_workspace_bytes(cfg), dtype=torch.uint8, device="cuda"),
                A=torch.empty((T, r), dtype=torch.bfloat16, device="cuda"),
                B=torch.empty((c["G"], r, c["d"]), dtype=torch.bfloat16, device="cuda"),
                sigma=torch.empty((r,), dtype=torch.float32, device="cuda"))


def _run_factorize(s):
    xkv.xkv_clf_factorize(s["cfg"], s["X"], s["omega"], s["ws"], s["A"], s["B"], s["sigma"])
    # The factors are unique only up to signs and to rotations inside (nearly) equal singular values; what a program
    # relies on is the cache they stand for, so that is handed back, whole, beside the singular values.
    r = s["case"]["r"]
    return {"x_hat": s["A"] @ s["B"].permute(1, 0, 2).reshape(r, -1), "sigma": s["sigma"]}


def _prepare_landmarks(c, g):
    G, batch, T, H_kv, d_h, n_out = (c[n] for n in ("G", "batch", "T", "H_kv", "d_h", "outliers"))
    n_c = -(-T // 8)
    # neighbouring tokens' keys resemble one another: a chunk's common part and each row's own
    keys = torch.empty((batch, G, T, H_kv * d_h), dtype=torch.bfloat16, device="cuda")
    for b in range(batch):
        for l in range(G):
            common = torch.randn((n_c, H_kv * d_h), generator=g, device="cuda").repeat_interleave(8, 0)[:T]
            keys[b, l] = (common + 0.5 * torch.randn((T, H_kv * d_h), generator=g, device="cuda")).to(torch.bfloat16)
    return dict(case=c, keys=keys, lm=torch.empty((batch, G, H_kv, n_c, d_h), dtype=torch.bfloat16, device="cuda"),
                min_cos=torch.empty((G, batch, H_kv, n_c), dtype=torch.float32, device="cuda") if n_out else None,
                ids=torch.empty((G, batch, H_kv, n_out), dtype=torch.int32, device="cuda") if n_out else None)


def _run_landmarks(s):
    c = s["case"]
    xkv.xkv_build_landmarks(s["keys"], s["lm"], G=c["G"], batch=c["batch"], T=c["T"], H_kv=c["H_kv"], d_h=c["d_h"],
                            min_cos=s["min_cos"], n_outliers=c["outliers"], outliers=s["ids"])
    return {"landmarks": s["lm"], "min_cos": s["min_cos"], "outliers": s["ids"]}


def _prepare_quantize(c, g):
    T, batch = c["T"], c["batch"]
    Gd = c["G"] * c["d"]
    s = dict(case=c)
    for n in ("k", "v"):
        r = c["r_" + n]
        a = _spectrum(r, r // 2, 1.0, Gd, T)
        s["A_" + n] = (torch.randn((batch, T, r), generator=g, device="cuda") * a).to(torch.bfloat16)
        s["B_" + n] = (torch.randn((batch, c["G"], r, c["d"]), generator=g, device="cuda") / math.sqrt(Gd)).to(torch.bfloat16)
    return s


def _run_quantize(s):
    bits = s["case"]["bits"]
    out = {}
    for n in ("k", "v"):
        out["codes_" + n], out["meta_" + n] = xkv.xkv_quantize_rtn(s["A_" + n], bits)
        codes, meta = xkv.xkv_quantize_rtn(s["B_" + n], bits)
        out["B_" + n] = xkv.xkv_dequantize_rtn(codes, meta, bits)
    return out


def _prepare_dense(c, g):
    G, batch, T, H_kv, H_q, d_h = (c[n] for n in ("G", "batch", "T", "H_kv", "H_q", "d_h"))
    # the handle of an uncompressed window carries shapes only
    A, B = _randn((batch, 8, 8), g), _randn((batch, G, 8, H_kv * d_h), g)
    grp = xkv.create_from_tensors(A, A, B, B, None, H_kv=H_kv, H_q=H_q, k_max=8)
    K = torch.empty((G, batch, H_kv, T, d_h), dtype=torch.bfloat16, device="cuda")
    V = torch.empty_like(K)
    for l in range(G):
        K[l] = _randn(K[l].shape, g)
        V[l] = _randn(V[l].shape, g)
    return dict(case=c, grp=grp, K=K, V=V, q=_randn((G, batch, H_q, d_h), g),
                len=torch.tensor([T - 1003 * b for b in range(batch)], dtype=torch.int32, device="cuda"),
                ws=torch.empty(xkv.xkv_dense_workspace_bytes(grp, T), dtype=torch.uint8, device="cuda"),
                out=torch.empty((G, batch, H_q, d_h), dtype=torch.bfloat16, device="cuda"),
                lse=torch.empty((G, batch, H_q), dtype=torch.float32, device="cuda"))


def _run_dense(s):
    c = s["case"]
    xkv.xkv_dense_attend(s["grp"], 0, c["G"], s["q"], s["K"], s["V"], s["len"], c["T"], s["ws"], s["out"], s["lse"])
    return {"out": s["out"], "lse": s["lse"]}


_PREPARE = {"decode": _prepare_decode, "factorize": _prepare_factorize, "landmarks": _prepare_landmarks,
            "quantize": _prepare_quantize, "dense": _prepare_dense}
_RUN = {"decode": _run_decode, "factorize": _run_factorize, "landmarks": _run_landmarks, "quantize": _run_quantize,
        "dense": _run_dense}


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return _PREPARE[case["op"]](case, g)


def run(state):
    return _RUN[state["case"]["op"]](state)


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without


def work(case):
    c = case
    op = c["op"]
    if op == "decode":
        d, n_rep = c["H_kv"] * c["d_h"], c["H_q"] // c["H_kv"]
        problems, n_c = c["G"] * c["batch"] * c["H_kv"], -(-c["T"] // 8)
        M = min((-(-c["k"] // 8) + c["outliers"]) * 8, c["T"])
        # distinct rows of a sequence: half of what independent selections of its (layer, head) problems would touch
        # (measured on these inputs, whose selections overlap), at least one selection
        uniq = max(M, 0.5 * c["T"] * (1.0 - (1.0 - M / c["T"]) ** (c["G"] * c["H_kv"])))
        per = 2.0 if c["bits"] == 16 else (c["bits"] + 1) / 8.0
        r = c["r_k"] + c["r_v"]
        tail = 2 * problems * c["tail"] * c["d_h"] * 2
        small = 2 * 2 * c["G"] * c["batch"] * c["H_q"] * c["d_h"] + problems * (M + 1) * 4
        nbytes = problems * n_c * c["d_h"] * 2 + c["batch"] * uniq * r * per + c["batch"] * c["G"] * r * d * 2 + tail + small
        flops = problems * (2 * n_c * c["d_h"] * n_rep + 2 * M * c["d_h"] * c["r_k"] + 2 * M * n_rep * (c["d_h"] + c["r_v"])
                            + 2 * c["r_v"] * c["d_h"] * n_rep + 4 * c["tail"] * c["d_h"] * n_rep)
        return {"bytes": nbytes, "flops": flops}
    if op == "factorize":
        N, T, r = c["G"] * c["d"], c["T"], c["r"]
        l = (r + 32 + 63) // 64 * 64
        # X once; three subspace iterations of two products, the factor A, and the reconstruction handed back
        return {"bytes": 2 * T * N * 2 + 2 * 2 * (T * r + N * r) + 2 * N * l, "flops": 2.0 * T * N * (6 * l + 2 * r)}
    if op == "landmarks":
        keys = c["batch"] * c["G"] * c["T"] * c["H_kv"] * c["d_h"]
        return {"bytes": keys * 2 + keys // 8 * 2 + (keys // c["d_h"] // 8 * 4 if c["outliers"] else 0), "flops": 10.0 * keys}
    if op == "quantize":
        r = c["r_k"] + c["r_v"]
        a, b = c["batch"] * c["T"] * r, c["batch"] * c["G"] * r * c["d"]
        code = (c["bits"] + 1) / 8.0
        return {"bytes": a * (2 + code) + b * (4 + 2 * code), "flops": 4.0 * (a + b)}
    rows = sum(c["T"] - 1003 * b for b in range(c["batch"])) * c["G"] * c["H_kv"]
    return {"bytes": rows * c["d_h"] * 4 + 4 * c["G"] * c["batch"] * c["H_q"] * c["d_h"],
            "flops": 4.0 * rows * c["d_h"] * (c["H_q"] // c["H_kv"])}


def tolerance(case):
    op = case["op"]
    if op == "quantize":
        return "exact"
    if op == "factorize":
        # bf16 factors; the directions beyond the signal are fitted to 1 % noise
        return {"rel": 1e-2, "max": 0.1}
    if op == "landmarks":
        # bf16 landmarks; outlier ids may differ where two cosines agree to the last bits of fp32
        return {"rel": 5e-3, "max": 0.02, "differ": 0.002}
    # index sets are exact; attention weights and outputs are bf16
    return {"rel": 1e-2, "max": 0.1}
