"""What this library is used for, as cases that can be timed: linear layers with INT8 and MXFP4 weights from one token to a
prefill of thousands, mixture-of-experts layers, and decode attention over INT8 caches (contiguous, paged, several query
tokens, latent).

`listed()` names the cases, `draw()` gives more of the same ranges, `prepare()` makes what a serving program holds before the
call (weights, prepared scales, caches, workspaces, output buffers), `run()` is one pass through the entry points of
`paper_2605_13915_b200.binding`.  Inputs follow the distributions of `paper_2605_13915_b200.inputs`, drawn on the GPU.
"""
import torch

from paper_2605_13915_b200 import binding as msd


def listed():
    return [
        # One attention output projection at 16 tokens, FP32 result: the smallest call, a chain of latencies.
        {"name": "w8_square_m16", "kind": "w8", "M": 16, "N": 4096, "K": 4096, "fp32": True},
        # The MLP of a layer (up, then down projection of its result) while a single sequence decodes.
        {"name": "w8_mlp_m1", "kind": "w8_mlp", "M": 1, "d": 4096, "ff": 14336},
        # The same MLP under a batch of sequences, a ragged number of them.
        {"name": "w8_mlp_m61", "kind": "w8_mlp", "M": 61, "d": 4096, "ff": 14336},
        # The same MLP on a chunk of a prompt.
        {"name": "w8_mlp_m1000", "kind": "w8_mlp", "M": 1000, "d": 4096, "ff": 14336},
        # The MLP with MXFP4 weights (scales prepared when the weights were loaded), 16 sequences decoding.
        {"name": "w4_mlp_m16", "kind": "w4_mlp", "M": 16, "d": 4096, "ff": 14336},
        # A long prompt through one MXFP4 layer.
        {"name": "w4_m4096", "kind": "w4", "M": 4096, "N": 8192, "K": 8192, "fp32": False},
        # Mixture of experts: 32 experts, about 16 tokens each, routed unevenly; INT8 and MXFP4 weights.
        {"name": "w8_moe_e32", "kind": "w8_moe", "E": 32, "tokens": 512, "N": 2048, "K": 7168},
        {"name": "w4_moe_e32", "kind": "w4_moe", "E": 32, "tokens": 512, "N": 2048, "K": 7168},
        # Decode attention of a grouped-query model, a batch of sequences of mixed lengths in a contiguous cache.
        {"name": "attn_gqa_b32", "kind": "attn", "B": 32, "Hq": 32, "Hkv": 8, "D": 128, "lo": 2048, "hi": 8192},
        # The same from a paged cache with the small pages that serving engines default to, 8 query heads to a KV head.
        {"name": "attn_paged16_b24", "kind": "attn_paged", "B": 24, "Hq": 64, "Hkv": 8, "D": 128, "lo": 512, "hi": 4096, "page": 16},
        # Speculative decoding: four query tokens a sequence.
        {"name": "attn_spec4_b16", "kind": "attn_spec", "B": 16, "Hq": 32, "Hkv": 8, "D": 128, "lo": 1024, "hi": 8192, "q_len": 4},
        # Decode attention on a latent cache (one KV head of 576, values are its first 512), long contexts.
        {"name": "attn_mla_b64", "kind": "attn_mla", "B": 64, "Hq": 64, "D": 576, "Dv": 512, "lo": 16384, "hi": 16384},
    ]


def _log(rng, lo, hi, multiple=1):
    """A size between lo and hi, spread over its logarithm, rounded to a multiple."""
    v = lo * (hi / lo) ** rng.random()
    return min(hi, max(lo, int(round(v / multiple)) * multiple))


def draw(rng):
    kind = rng.choice(["w8", "w8_mlp", "w8_mlp_prefill", "w4_mlp", "w4", "w8_moe", "w4_moe", "attn", "attn_paged", "attn_spec",
                       "attn_mla"])
    if kind == "w8":
        step = rng.choice([64, 64, 16])
        return {"kind": "w8", "M": _log(rng, 1, 128), "N": _log(rng, 1024, 16384, step), "K": _log(rng, 1024, 16384, step),
                "fp32": rng.random() < 0.3}
    if kind == "w8_mlp":
        d = _log(rng, 2048, 6144, 64)
        return {"kind": "w8_mlp", "M": _log(rng, 1, 128), "d": d, "ff": min(16384, int(d * rng.uniform(2.5, 4.0)) // 64 * 64)}
    if kind == "w8_mlp_prefill":
        d = _log(rng, 2048, 6144, 64)
        ff = min(16384, int(d * rng.uniform(2.5, 4.0)) // 64 * 64)
        return {"kind": "w8_mlp", "M": _log(rng, 129, max(130, min(4096, int(58e9 / (d * ff)))), 1), "d": d, "ff": ff}
    if kind == "w4_mlp":
        d = _log(rng, 2048, 6144, 128)
        return {"kind": "w4_mlp", "M": _log(rng, 1, 128), "d": d, "ff": min(16384, int(d * rng.uniform(2.5, 4.0)) // 128 * 128)}
    if kind == "w4":
        N, K = _log(rng, 2048, 8192, 64), _log(rng, 2048, 8192, 128)
        return {"kind": "w4", "M": _log(rng, 129, 4096), "N": N, "K": K, "fp32": rng.random() < 0.2}
    if kind in ("w8_moe", "w4_moe"):
        E = _log(rng, 8, 64)
        K = _log(rng, 1024, 7168, 128)
        N = _log(rng, 1024, max(1024, min(7168, int(4.6e8 / (E * K)))), 64)
        return {"kind": kind, "E": E, "tokens": E * _log(rng, 2, 48) + rng.randrange(E), "N": N, "K": K}
    if kind == "attn_mla":
        B = _log(rng, 1, 64)
        hi = _log(rng, 1024, 16384)
        return {"kind": kind, "B": B, "Hq": rng.choice([16, 32, 64]), "D": 576, "Dv": 512, "lo": max(1, int(hi * rng.choice([0.25, 0.5, 1.0]))),
                "hi": hi}
    B = _log(rng, 1, 64)
    hi = _log(rng, 256, min(32768, 160000 // B))
    case = {"kind": kind, "B": B, "Hq": rng.choice([8, 16, 24, 32, 40, 64]), "Hkv": 8, "D": 128,
            "lo": max(16, int(hi * rng.choice([0.1, 0.25, 0.5, 1.0]))), "hi": hi}
    if kind == "attn_paged":
        case["page"] = rng.choice([16, 32, 64, 128])
    if kind == "attn_spec":
        case["q_len"] = rng.choice([2, 3, 4])
        case["Hq"] = rng.choice([8, 16, 32])
    return case


# ---- inputs, on the GPU ----------------------------------------------------------------------------------------------------
def _activations(g, M, K):
    """N(0,1), one channel in a hundred 50 times larger, BF16."""
    x = torch.randn((M, K), generator=g, device="cuda")
    x[:, torch.randperm(K, generator=g, device="cuda")[:K // 100]] *= 50.0
    return x.to(torch.bfloat16).contiguous()


def _weights_int8(g, N, K):
    """N(0, 0.02), symmetric INT8 with one scale per output channel."""
    q = torch.empty((N, K), dtype=torch.int8, device="cuda")
    s = torch.empty(N, device="cuda")
    rows = max(1, (1 << 27) // K)
    for r in range(0, N, rows):
        w = torch.randn((min(rows, N - r), K), generator=g, device="cuda").mul_(0.02)
        sc = w.abs().amax(1) / 127.0
        s[r:r + rows] = sc
        q[r:r + rows] = torch.round(w / sc[:, None]).clamp_(-127, 127).to(torch.int8)
    return q, s


def _weights_mxfp4(g, N, K):
    """N(0, 0.02) as E2M1 values with one power-of-two scale per 32 elements of K; element 2i in the low nibble."""
    q = torch.empty((N, K // 2), dtype=torch.uint8, device="cuda")
    e = torch.empty((N, K // 32), dtype=torch.uint8, device="cuda")
    mids = torch.tensor([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0], device="cuda")
    rows = max(1, (1 << 26) // K)
    for r in range(0, N, rows):
        w = torch.randn((min(rows, N - r), K), generator=g, device="cuda").mul_(0.02)
        blk = w.view(w.shape[0], K // 32, 32)
        ex = torch.floor(torch.log2(blk.abs().amax(2).clamp_min(2.0 ** -120))) - 2.0
        v = blk / torch.exp2(ex)[:, :, None]
        code = torch.bucketize(v.abs().clamp_max(6.0), mids, out_int32=True).to(torch.uint8) | ((v < 0).to(torch.uint8) << 3)
        code = code.view(w.shape[0], K // 2, 2)
        q[r:r + rows] = code[:, :, 0] | (code[:, :, 1] << 4)
        e[r:r + rows] = (ex + 127.0).to(torch.uint8)
    return q, e


def _cache_int8(g, T, H, D):
    """N(0,1) rounded to BF16, then INT8 with one scale per token and KV head."""
    k = torch.empty((T, H, D), dtype=torch.int8, device="cuda")
    s = torch.empty((T, H), device="cuda")
    rows = max(1, (1 << 27) // (H * D))
    for t in range(0, T, rows):
        x = torch.randn((min(rows, T - t), H, D), generator=g, device="cuda").to(torch.bfloat16).float()
        sc = x.abs().amax(2) / 127.0
        s[t:t + rows] = sc
        k[t:t + rows] = torch.round(x / sc[:, :, None]).clamp_(-127, 127).to(torch.int8)
    return k, s


def _group_sizes(case, seed):
    """Tokens per expert: every token goes to an expert of its own choice, at most 128 to one (some experts may get none)."""
    g = torch.Generator()
    g.manual_seed(seed)
    load = torch.rand(case["E"], generator=g) + 0.5
    pick = torch.multinomial(load, case["tokens"], replacement=True, generator=g)
    return torch.bincount(pick, minlength=case["E"]).clamp_max_(128).tolist()


def _lengths(case, seed):
    g = torch.Generator()
    g.manual_seed(seed)
    return torch.randint(case["lo"], case["hi"] + 1, (case["B"],), generator=g, dtype=torch.int32)


def _out_dtype(case):
    return torch.float32 if case.get("fp32") else torch.bfloat16


# ---- the pass --------------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    st = {"kind": kind}
    if kind in ("w8", "w8_mlp", "w4", "w4_mlp"):
        M = case["M"]
        layers = [(case["N"], case["K"])] if kind in ("w8", "w4") else [(case["ff"], case["d"]), (case["d"], case["ff"])]
        st["x"] = _activations(g, M, layers[0][1])
        st["layers"] = []
        for N, K in layers:
            y = torch.empty((M, N), dtype=_out_dtype(case), device="cuda")
            if kind.startswith("w8"):
                w, s = _weights_int8(g, N, K)
                ws = msd.workspace(msd.gemm_w8a16_workspace_bytes(M, N, K))
            else:
                w, e = _weights_mxfp4(g, N, K)
                s = msd.prepare_w4a16_scales(e)
                ws = msd.workspace(msd.gemm_w4a16_workspace_bytes(M, N, K))
            st["layers"].append((w, s, ws, y))
    elif kind in ("w8_moe", "w4_moe"):
        E, N, K = case["E"], case["N"], case["K"]
        sizes = _group_sizes(case, seed)
        M = sum(sizes)
        st["x"], st["sizes"] = _activations(g, M, K), sizes
        st["y"] = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        if kind == "w8_moe":
            w, s = _weights_int8(g, E * N, K)
            st["w"], st["s"] = w.view(E, N, K), s.view(E, N)
            st["ws"] = msd.workspace(msd.lib().msd_grouped_gemm_w8a16_workspace_bytes(M, max(sizes), E, N, K))
        else:
            w, e = _weights_mxfp4(g, E * N, K)
            st["w"], st["s"] = w.view(E, N, K // 2), msd.prepare_w4a16_scales(e.view(E, N, K // 32))
            st["ws"] = msd.workspace(msd.lib().msd_grouped_gemm_w4a16_workspace_bytes(E, N, K))
    else:
        B, Hq, D = case["B"], case["Hq"], case["D"]
        Hkv, Dv, q_len = case.get("Hkv", 1), case.get("Dv", D), case.get("q_len", 1)
        lengths = _lengths(case, seed)
        st["max_seqlen"] = int(lengths.max())
        st["scale"] = D ** -0.5
        st["dv"] = Dv
        if kind == "attn_paged":
            page = case["page"]
            blocks = (lengths + page - 1) // page
            order = torch.randperm(int(blocks.sum()), generator=torch.Generator().manual_seed(seed)).to(torch.int32)
            table = torch.full((B, int(blocks.max())), -1, dtype=torch.int32)
            at = 0
            for b, n in enumerate(blocks.tolist()):
                table[b, :n] = order[at:at + n]
                at += n
            st["table"], st["lengths"], st["page"] = table.cuda(), lengths.cuda(), page
            T = at * page
        else:
            cu = torch.zeros(B + 1, dtype=torch.int32)
            cu[1:] = torch.cumsum(lengths, 0)
            st["cu"] = cu.cuda()
            T = int(cu[-1])
        st["q"] = torch.randn((B, Hq, D) if q_len == 1 else (B, q_len, Hq, D), generator=g, device="cuda").to(torch.bfloat16)
        st["k"], st["ks"] = _cache_int8(g, T, Hkv, D)
        st["v"], st["vs"] = (None, None) if kind == "attn_mla" else _cache_int8(g, T, Hkv, Dv)
        st["ws"] = msd.workspace(msd.attn_decode_int8kv_workspace_bytes(B, Hq * q_len, Hkv, D, Dv, st["max_seqlen"]))
        st["y"] = torch.empty((B, Hq, Dv), dtype=torch.bfloat16, device="cuda")
    return st


def run(st):
    kind = st["kind"]
    if kind in ("w8", "w8_mlp"):
        x, outs = st["x"], []
        for w, s, ws, y in st["layers"]:
            x = msd.gemm_w8a16(x, w, s, ws=ws, out=y)
            outs.append(x)
        return outs
    if kind in ("w4", "w4_mlp"):
        x, outs = st["x"], []
        for w, s, ws, y in st["layers"]:
            x = msd.gemm_w4a16(x, w, None, ws=ws, out=y, prepared=s)
            outs.append(x)
        return outs
    if kind == "w8_moe":
        return msd.grouped_gemm_w8a16(st["x"], st["w"], st["s"], st["sizes"], ws=st["ws"], out=st["y"])
    if kind == "w4_moe":
        return msd.grouped_gemm_w4a16(st["x"], st["w"], None, st["sizes"], ws=st["ws"], out=st["y"], prepared=st["s"])
    if kind == "attn_paged":
        return msd.attn_decode_int8kv_paged(st["q"], st["k"], st["v"], st["ks"], st["vs"], st["table"], st["lengths"], st["page"],
                                            st["max_seqlen"], st["scale"], ws=st["ws"], out=st["y"])
    if kind == "attn_spec":
        return msd.attn_decode_int8kv_spec(st["q"], st["k"], st["v"], st["ks"], st["vs"], st["cu"], st["max_seqlen"], st["scale"],
                                           ws=st["ws"])
    return msd.attn_decode_int8kv(st["q"], st["k"], st["v"], st["ks"], st["vs"], st["cu"], st["max_seqlen"], st["scale"], dv=st["dv"],
                                  ws=st["ws"], out=st["y"])


def work(case):
    """Weights or cache with their scales once, activations in, results out; two multiply-accumulates per weight and
    component (the method multiplies both components)."""
    kind = case["kind"]
    if kind in ("w8", "w8_mlp", "w4", "w4_mlp"):
        M = case["M"]
        layers = [(case["N"], case["K"])] if kind in ("w8", "w4") else [(case["ff"], case["d"]), (case["d"], case["ff"])]
        out = 4 if case.get("fp32") else 2
        per = [(N * K + 4 * N if kind.startswith("w8") else N * K // 2 + N * K // 32) + M * (2 * K + out * N) for N, K in layers]
        return {"bytes": sum(per), "flops": sum(4 * M * N * K for N, K in layers)}
    if kind in ("w8_moe", "w4_moe"):
        E, N, K, M = case["E"], case["N"], case["K"], case["tokens"]
        w = N * K + 4 * N if kind == "w8_moe" else N * K // 2 + N * K // 32
        return {"bytes": E * w + M * 2 * (K + N), "flops": 4 * M * N * K}
    B, Hq, D, q_len = case["B"], case["Hq"], case["D"], case.get("q_len", 1)
    Hkv, Dv = case.get("Hkv", 1), case.get("Dv", D)
    T = B * (case["lo"] + case["hi"]) // 2
    cache = T * Hkv * (D + 4 + (0 if kind == "attn_mla" else Dv + 4))
    return {"bytes": cache + B * q_len * Hq * 2 * (D + Dv), "flops": 4 * T * q_len * Hq * (D + Dv)}


def tolerance(case):
    """Four times the differences measured on the listed cases.  Linear layers against FP64 sums of the same components
    (rounded once): 4e-8 relative for an FP32 result, at most 1.0e-4 and one BF16 unit in the last place (0.0078) for a
    BF16 one, the second layer's input rounding included.  Attention with the context split at other places: 1.6e-3 and
    0.015 (the probabilities are then quantized against other running maxima); against an FP64 softmax 1.7e-3."""
    if case["kind"].startswith("attn"):
        return {"rel": 6.5e-3, "max": 0.06}
    if case.get("fp32"):
        return {"rel": 1e-6, "max": 1e-5}
    return {"rel": 5e-4, "max": 0.032}
