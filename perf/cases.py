"""The work whose speed this repository is measured by, through its public entry points.

Eight kinds of call sequence, each as a quantization program issues it:

* ``hessian``       h = diag(X^T X) over calibration tokens streamed in chunks (Sec. 3.2, Eq. 4);
* ``quantize``      a linear layer's NVFP4 codes: the global scale, then the scale search with
                    packing (Algorithm 1, or Algorithm 2 with the 4over6 start);
* ``rtn``           the plain round-to-nearest baseline: global scale, RTN codes, packing;
* ``output_error``  the layer-output evaluation ||X dW^T||^2 of a quantization (Eq. 3);
* ``hessian_full``  H = X^T X for GPTQ, one call over the tokens;
* ``factor``        GPTQ's damped inverse-Cholesky factor of H;
* ``gptq``          Algorithm 3's block loop with H-Scale as its local quantizer;
* ``gptq_layer``    all of Algorithm 3 for one small layer: H, factor, global scale, block loop.

``exact`` restates each in plain torch at 64 bits.
"""
from __future__ import annotations

import torch

import paper_2608_28113_gb300 as hs
from paper_2608_28113_gb300 import workloads as wl

BF16, F32, F64, U8 = torch.bfloat16, torch.float32, torch.float64, torch.uint8


def listed():
    return [
        # one calibration chunk of the smallest layer: a call whose cost is latency
        {"name": "hessian_small", "kind": "hessian", "tokens": 2048, "n": 1024, "chunk": 2048, "ready": False},
        # an attention input space streamed from device memory, eight 8192-token chunks
        {"name": "hessian_stream", "kind": "hessian", "tokens": 65536, "n": 4096, "chunk": 8192, "ready": True},
        # the smallest layer of the configurations: launches and latency
        {"name": "quantize_small", "kind": "quantize", "m": 512, "n": 1024, "down": 4, "up": 4, "start": "rtn",
         "weighted": True, "layout": "whole", "shared": False},
        # an attention projection under the paper's default window of 16 candidates
        {"name": "quantize_attention", "kind": "quantize", "m": 4096, "n": 4096, "down": 9, "up": 6, "start": "rtn",
         "weighted": True, "layout": "whole", "shared": False},
        # the widest MLP matrix of the configurations, with the work-sharing workspace
        {"name": "quantize_wide", "kind": "quantize", "m": 28672, "n": 8192, "down": 4, "up": 4, "start": "rtn",
         "weighted": True, "layout": "whole", "shared": True},
        # Algorithm 2 on a layer whose rows are not whole 512-column chunks
        {"name": "quantize_4over6_ragged", "kind": "quantize", "m": 3001, "n": 3216, "down": 4, "up": 4,
         "start": "4over6", "weighted": True, "layout": "whole", "shared": False},
        # the RTN baseline of an MLP projection
        {"name": "rtn_pack", "kind": "rtn", "m": 14336, "n": 4096},
        # layer-output error of a quantized attention projection over one calibration chunk
        {"name": "output_error", "kind": "output_error", "tokens": 8192, "m": 4096, "n": 4096},
        # GPTQ's full Hessian of a 4096-wide input space
        {"name": "hessian_full", "kind": "hessian_full", "tokens": 16384, "n": 4096},
        # its factor, once per input space
        {"name": "gptq_factor", "kind": "factor", "n": 4096},
        # Algorithm 3's block loop over an attention projection
        {"name": "gptq_attention", "kind": "gptq", "m": 4096, "n": 4096, "block": 128, "down": 4, "up": 4},
        # Algorithm 3 from the activations to the packed weights on the smallest layer
        {"name": "gptq_layer_small", "kind": "gptq_layer", "tokens": 2048, "m": 512, "n": 1024, "block": 128,
         "down": 4, "up": 4},
    ]


def _log(rng, lo, hi, step=1):
    """A whole number spread over the logarithm of [lo, hi], a multiple of step."""
    v = lo * (hi / lo) ** rng.random()
    return max(step, min(hi // step * step, int(v / step + 0.5) * step))


def draw(rng):
    kind = rng.choice(["hessian", "quantize", "quantize", "rtn", "output_error", "hessian_full", "factor", "gptq",
                       "gptq_layer"])
    window = rng.choice([(1, 1), (2, 2), (4, 4), (8, 8), (9, 6), (16, 16)])
    if kind == "hessian":
        n = _log(rng, 256, 28672, 8)
        tokens = _log(rng, 256, min(131072, (1 << 29) // n))
        return {"kind": kind, "tokens": tokens, "n": n, "chunk": min(tokens, rng.choice([2048, 4096, 5000, 8192])),
                "ready": rng.random() < 0.5}
    if kind == "quantize":
        n = _log(rng, 256, 28672, rng.choice([16, 512, 1024]))
        most = 28672 * 8192 * 9 // (9 + sum(window)) // n
        return {"kind": kind, "m": _log(rng, 16, min(28672, most)), "n": n, "down": window[0], "up": window[1],
                "start": rng.choice(["rtn", "rtn", "given", "4over6"]), "weighted": rng.random() < 0.8,
                "layout": rng.choice(["whole", "whole", "columns"]), "shared": rng.random() < 0.3}
    if kind == "rtn":
        n = _log(rng, 256, 28672, 16)
        return {"kind": kind, "m": _log(rng, 16, min(28672, 28672 * 4096 // n)), "n": n}
    if kind == "output_error":
        n = _log(rng, 256, 14336, 16)
        m = _log(rng, 64, 14336)
        return {"kind": kind, "tokens": _log(rng, 128, max(128, min(8192, 8192 * 4096 * 4096 // (n * m)))), "m": m,
                "n": n}
    if kind == "hessian_full":
        n = _log(rng, 256, 8192, rng.choice([8, 8, 64, 1]))
        return {"kind": kind, "tokens": _log(rng, 512, min(65536, 16384 * 4096 * 4096 // (n * n))), "n": n}
    if kind == "factor":
        return {"kind": kind, "n": _log(rng, 128, 4096)}
    block = rng.choice([32, 64, 128, 128, 256])
    if kind == "gptq":
        n = _log(rng, 512, 4096, block)
        return {"kind": kind, "m": _log(rng, 64, min(14336, 4096 ** 3 // (n * n))), "n": n, "block": block,
                "down": window[0], "up": window[1]}
    return {"kind": kind, "tokens": _log(rng, 1024, 8192), "m": _log(rng, 64, 2048), "n": _log(rng, 256, 2048, block),
            "block": block, "down": window[0], "up": window[1]}


# ---------------------------------------------------------------- inputs
def _dev():
    return torch.device("cuda", 0)


def _weights(case, seed):
    return wl.weight(case["m"], case["n"], 0.02, seed, _dev())


def _magnitudes(n, seed):
    return wl.channel_magnitudes(n, 1.0, max(1, n // 512), 50.0, seed, _dev())


def _activations(tokens, n, seed):
    """bf16 [tokens, n] with the workloads' channel magnitudes and correlated channels (64 shared
    directions with a third of the energy), as real activations have."""
    g = torch.Generator(device=_dev())
    g.manual_seed(wl.chunk_seed(seed, "cases", n))
    a = _magnitudes(n, seed)
    mix = torch.randn(64, n, generator=g, device=_dev())
    x = torch.randn(tokens, n, generator=g, device=_dev())
    x.addmm_(torch.randn(tokens, 64, generator=g, device=_dev()), mix, alpha=0.5 ** 0.5 / 8.0)
    return x.mul_(a).to(BF16)


def _h(n, seed):
    """The diagonal proxy of a layer whose calibration is done: sums of 4096 squares."""
    g = torch.Generator(device=_dev())
    g.manual_seed(wl.chunk_seed(seed, "cases-h", n))
    a = _magnitudes(n, seed)
    return (a * a * 4096.0 * (1.0 + 0.02 * torch.randn(n, generator=g, device=_dev()))).contiguous()


def _hessian64(x):
    n = x.shape[1]
    H = torch.zeros(n, n, dtype=F64, device=x.device)
    for t in range(0, x.shape[0], 8192):
        xt = x[t:t + 8192].to(F64)
        H.addmm_(xt.T, xt)
    return H


def _hessian_input(n, seed):
    """A layer's H in fp32 (2 n tokens or more, so that it has full rank)."""
    x = _activations(max(1024, 2 * n), n, seed).to(F32)
    return (x.T @ x).contiguous()


def _factor64(H, damp=0.01):
    """U upper with U^T U = (H + damp mean(diag H) I)^-1 at 64 bits."""
    A = torch.triu(H.to(F64))
    A = A + torch.triu(A, 1).T
    d = torch.diagonal(A)
    d += damp * d.mean()
    L = torch.linalg.cholesky(torch.flip(A, (0, 1)))
    Z = torch.linalg.solve_triangular(L, torch.eye(L.shape[0], dtype=F64, device=L.device), upper=False)
    return torch.flip(Z, (0, 1))


def _outputs(m, n):
    return (torch.empty(m, n // 16, dtype=U8, device=_dev()), torch.empty(m, n // 2, dtype=U8, device=_dev()))


def prepare(case, seed):
    kind, dev = case["kind"], _dev()
    s = {"case": case}
    if kind == "hessian":
        a = _magnitudes(case["n"], seed)
        s["x"] = [wl.activation_chunk(min(case["chunk"], case["tokens"] - t), a, seed, i)
                  for i, t in enumerate(range(0, case["tokens"], case["chunk"]))]
        s["h"] = torch.zeros(case["n"], dtype=F32, device=dev)
        return s
    if kind in ("hessian_full", "gptq_layer"):
        n = case["n"]
        s["x"] = _activations(case["tokens"], n, seed)
        s["H"] = torch.zeros(n, n, dtype=F32, device=dev)
        s["H_ws"] = None
        if n % 8:  # rows that are not 16-byte aligned: the call needs its workspace
            nbytes = hs.hscale_hessian_full_workspace_bytes(case["tokens"], n)
            s["H_ws"] = torch.empty(nbytes, dtype=U8, device=dev)
        if kind == "hessian_full":
            return s
    if kind == "factor":
        s["H"] = _hessian_input(case["n"], seed)
    if kind in ("factor", "gptq_layer"):
        n = case["n"]
        s["U"] = torch.zeros(n, n, dtype=F32, device=dev)
        s["dead"] = torch.zeros(n, dtype=U8, device=dev)
        s["info"] = torch.zeros(3, dtype=torch.int32, device=dev)
        s["U_ws"] = torch.empty(hs.hscale_gptq_factor_workspace_bytes(n), dtype=U8, device=dev)
        if kind == "factor":
            return s
    m, n = case["m"], case["n"]
    s["w"] = _weights(case, seed)
    s["sg"] = torch.zeros(1, dtype=F32, device=dev)
    s["ws"] = torch.empty(hs.hscale_rtn_workspace_bytes(), dtype=U8, device=dev)
    s["codes"], s["packed"] = _outputs(m, n)
    if kind in ("quantize", "gptq"):
        s["h"] = _h(n, seed) if case.get("weighted", True) else None
    if kind == "quantize":
        s["init"] = _outputs(m, n)[0] if case["start"] == "given" else None
        s["share"] = torch.empty(hs.hscale_refine_workspace_bytes(), dtype=U8, device=dev) if case["shared"] else None
    if kind == "gptq":
        H = _hessian_input(n, seed)
        s["h"] = torch.diagonal(H).clone()
        s["U"] = _factor64(H).to(F32).contiguous()
        s["dead"] = torch.zeros(n, dtype=U8, device=dev)
    if kind in ("gptq", "gptq_layer"):
        s["loop_ws"] = torch.empty(hs.hscale_gptq_workspace_bytes(m, n, case["block"]), dtype=U8, device=dev)
    if kind == "gptq":
        hs.hscale_rtn_scales(s["w"], s["sg"], None, s["ws"])
    if kind == "output_error":
        s["x"] = _activations(case["tokens"], n, seed)
        hs.hscale_rtn_scales(s["w"], s["sg"], s["codes"], s["ws"])
        hs.hscale_pack_nvfp4(s["w"], s["sg"], s["codes"], s["packed"])
        s["dw2"] = torch.zeros(m, hs.residual_ld(n), dtype=BF16, device=dev)
        s["sum"] = torch.zeros(1, dtype=F64, device=dev)
        s["e_ws"] = torch.empty(hs.hscale_output_error_workspace_bytes(case["tokens"], m), dtype=U8, device=dev)
    return s


# ---------------------------------------------------------------- one pass
def _search(s):
    case, w, h = s["case"], s["w"], s["h"]
    down, up, four = case["down"], case["up"], case["start"] == "4over6"
    if case["layout"] == "columns":
        n = case["n"]
        cut = (n // 32 + 1) * 16 if n >= 64 else n
        for c0, c1 in ((0, cut), (cut, n)):
            init = None if s["init"] is None else s["init"][:, c0 // 16:c1 // 16]
            hs.hscale_refine_scales_strided(w[:, c0:c1], None if h is None else h[c0:c1], s["sg"], init, four, down,
                                            up, s["codes"][:, c0 // 16:c1 // 16], s["packed"][:, c0 // 2:c1 // 2])
    elif s["share"] is not None:
        hs.hscale_refine_scales_ws(w, h, s["sg"], s["init"], int(four), down, up, s["codes"], s["packed"], 0,
                                   s["share"])
    elif four:
        hs.hscale_refine_scales_4over6(w, h, s["sg"], down, up, s["codes"], s["packed"])
    else:
        hs.hscale_refine_scales(w, h, s["sg"], s["init"], down, up, s["codes"], s["packed"])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "hessian":
        flags = hs.HSCALE_HESSIAN_X_READY if case["ready"] else 0
        s["h"].zero_()
        for x in s["x"]:
            hs.hscale_hessian_diag_accumulate_ex(x, s["h"], flags)
        return {"h": s["h"]}
    if kind == "quantize":
        hs.hscale_rtn_scales(s["w"], s["sg"], s["init"], s["ws"])
        _search(s)
        return {"global_scale": s["sg"], "codes": s["codes"], "packed": s["packed"]}
    if kind == "rtn":
        hs.hscale_rtn_scales(s["w"], s["sg"], s["codes"], s["ws"])
        hs.hscale_pack_nvfp4(s["w"], s["sg"], s["codes"], s["packed"])
        return {"global_scale": s["sg"], "codes": s["codes"], "packed": s["packed"]}
    if kind == "output_error":
        s["sum"].zero_()
        hs.hscale_dequant_residual(s["w"], s["sg"], s["codes"], s["packed"], s["dw2"])
        hs.hscale_output_error(s["x"], s["dw2"], case["m"], s["sum"], s["e_ws"])
        return {"residual": s["dw2"], "error": s["sum"]}
    if kind == "hessian_full":
        s["H"].zero_()
        hs.hscale_hessian_full_accumulate(s["x"], s["H"], s["H_ws"])
        return {"H": s["H"]}
    if kind == "factor":
        hs.hscale_gptq_factor(s["H"], 0.01, s["U"], s["dead"], s["info"], s["U_ws"])
        return {"U": s["U"], "dead": s["dead"], "info": s["info"]}
    if kind == "gptq":
        hs.hscale_gptq_hscale(s["w"], s["U"], s["h"], s["sg"], s["dead"], case["block"], case["down"], case["up"],
                              s["codes"], s["packed"], s["loop_ws"])
        return {"codes": s["codes"], "packed": s["packed"]}
    # gptq_layer
    s["H"].zero_()
    hs.hscale_hessian_full_accumulate(s["x"], s["H"], s["H_ws"])
    h = torch.diagonal(s["H"]).clone()
    hs.hscale_gptq_factor(s["H"], 0.01, s["U"], s["dead"], s["info"], s["U_ws"])
    hs.hscale_rtn_scales(s["w"], s["sg"], None, s["ws"])
    hs.hscale_gptq_hscale(s["w"], s["U"], h, s["sg"], s["dead"], case["block"], case["down"], case["up"], s["codes"],
                          s["packed"], s["loop_ws"])
    return {"H": s["H"], "U": s["U"], "global_scale": s["sg"], "codes": s["codes"], "packed": s["packed"]}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    n = case["n"]
    m, t = case.get("m", 0), case.get("tokens", 0)
    quantized = m * n // 16 + m * n // 2
    if kind == "hessian":
        return {"bytes": 2 * t * n + 4 * n, "flops": 2 * t * n}
    if kind == "quantize":  # five operations per element and candidate
        candidates = case["down"] + case["up"] + 1
        return {"bytes": 2 * m * n + quantized + (4 * n if case["weighted"] else 0), "flops": 5 * candidates * m * n}
    if kind == "rtn":
        return {"bytes": 2 * m * n + quantized, "flops": 2 * m * n}
    if kind == "output_error":
        return {"bytes": 2 * t * n + 2 * m * n + quantized + 4 * m * n, "flops": 2 * t * m * n}
    upper = n * (n + 1) // 2
    if kind == "hessian_full":
        return {"bytes": 2 * t * n + 4 * n * n, "flops": 2 * t * upper}
    if kind == "factor":  # a Cholesky factor and its triangular inverse
        return {"bytes": 4 * upper + 4 * n * n, "flops": 2 * n ** 3 // 3}
    candidates = case["down"] + case["up"] + 1
    loop = {"bytes": 2 * m * n + 4 * upper + quantized,
            "flops": m * n * (n - case["block"]) + 5 * candidates * m * n}
    if kind == "gptq":
        return loop
    return {"bytes": 2 * t * n + 4 * n * n + 2 * m * n + quantized,
            "flops": 2 * t * upper + 2 * n ** 3 // 3 + loop["flops"]}


def tolerance(case):
    """About four times what run() is measured to be off exact() over the listed and drawn cases."""
    kind = case["kind"]
    if kind == "hessian":       # fp32 sums on the tensor cores: 2.5e-6
        return {"rel": 1e-5, "max": 1e-5}
    if kind == "quantize":      # near-ties of fp32 error sums: 1.5e-5 of the codes
        return {"rel": 0.0, "differ": 6e-5}
    if kind == "rtn":           # decided exactly
        return "exact"
    if kind == "output_error":  # 8e-6
        return {"rel": 3e-5, "max": 3e-5}
    if kind == "hessian_full":  # 5.8e-6
        return {"rel": 2.5e-5, "max": 2.5e-5}
    if kind == "factor":        # 9e-7, 1.2e-5 at the worst entry
        return {"rel": 4e-6, "max": 5e-5}
    # a weight near a rounding midpoint changes the errors propagated along the rest of its row:
    # 2.3e-4 of the bytes over many rows, a good part of one row where there are few
    differ = min(0.01, 1e-3 + 0.5 / case["m"])
    if kind == "gptq":
        return {"rel": 0.0, "differ": differ}
    return {"rel": 2.5e-5, "max": 7e-5, "differ": differ}


# ---------------------------------------------------------------- the same at 64 bits
_GRID = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)
_MIDS = (0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0)


def _e4m3(c):
    """Value of the E4M3 codes c (a tensor of 0..126) at 64 bits."""
    e, f = c // 8, (c % 8).to(F64)
    return torch.where(e == 0, f * 2.0 ** -9, (1 + f / 8) * torch.pow(2.0, e.to(F64) - 7))


def _e2m1(a, s):
    """E2M1 magnitude codes of |a| / s, ties to the even code; the midpoints times s are exact."""
    k = torch.zeros(a.shape, dtype=torch.int64, device=a.device)
    for i, mid in enumerate(_MIDS):
        t = mid * s
        k += (a >= t) if i % 2 else (a > t)
    return k


def _anchored(amax, s_g, c):
    """max(1, RNE_E4M3(amax / (c s_g)))."""
    codes = torch.arange(1, 127, device=amax.device)
    lo, hi = _e4m3(codes - 1), _e4m3(codes)
    mid = (lo + hi) / 2 * c * s_g           # exact
    even = codes % 2 == 0
    n_ge = torch.searchsorted(mid, amax.contiguous(), right=True)   # midpoints <= amax
    tie = (n_ge > 0) & (mid[(n_ge - 1).clamp(min=0)] == amax) & ~even[(n_ge - 1).clamp(min=0)]
    return (n_ge - tie.long()).clamp(min=1)


def _errors(a, hg, s):
    q = torch.tensor(_GRID, dtype=F64, device=a.device)[_e2m1(a, s)]
    return (hg * (a - q * s) ** 2).sum(-1)


def _search64(w, h, s_g, start, down, up):
    """(codes, magnitude codes) of rows w (64 bits) under Algorithm 1 or 2."""
    m, n = w.shape
    a = w.abs().view(m, n // 16, 16)
    hg = h.view(1, n // 16, 16)
    c0 = _anchored(a.amax(-1), s_g, 6.0)
    if start == "4over6":
        c4 = _anchored(a.amax(-1), s_g, 4.0)
        one = torch.ones_like(hg)
        c0 = torch.where(_errors(a, one, (_e4m3(c0) * s_g)[..., None]) < _errors(a, one, (_e4m3(c4) * s_g)[..., None]),
                         c0, c4)
    best, be = c0.clone(), torch.full(c0.shape, float("inf"), dtype=F64, device=w.device)
    shifts = sorted(range(-down, up + 1), key=lambda d: (abs(d), d))
    for d in shifts:
        c = c0 + d
        ok = (c >= 1) & (c <= 126)
        c = c.clamp(1, 126)
        e = _errors(a, hg, (_e4m3(c) * s_g)[..., None])
        take = ok & (e < be)
        be, best = torch.where(take, e, be), torch.where(take, c, best)
    return best, _e2m1(a, (_e4m3(best) * s_g)[..., None])


def _pack(w, k):
    nib = (k.view(w.shape) + 8 * torch.signbit(w).long()).to(U8)
    return nib[:, 0::2] | (nib[:, 1::2] << 4)


def _rows(m, n):
    step = max(1, (1 << 24) // n)
    return [(r, min(m, r + step)) for r in range(0, m, step)]


def _gptq64(w, U, h, s_g, block, down, up):
    """Algorithm 3's block loop on the running weights at 64 bits."""
    m, n = w.shape
    W, U = w.to(F64), U.to(F64)
    codes, packed = _outputs(m, n)
    for c in range(0, n, block):
        cs = slice(c, c + block)
        wb = W[:, cs].contiguous()
        best, k = _search64(wb, h[cs], s_g, "rtn", down, up)
        codes[:, c // 16:(c + block) // 16] = best.to(U8)
        packed[:, c // 2:(c + block) // 2] = _pack(wb, k)
        grid = torch.tensor(_GRID, dtype=F64, device=w.device)
        what = (grid[k] * (_e4m3(best) * s_g)[..., None]).view(m, block)
        E = (wb - torch.where(torch.signbit(wb), -what, what)) / torch.diagonal(U)[cs]
        W[:, c + block:] -= E @ U[cs, c + block:]
    return codes, packed


def exact(case, seed):
    kind = case["kind"]
    s = prepare(case, seed)
    if kind == "hessian":
        return {"h": sum(x.to(F64).square().sum(0) for x in s["x"])}
    if kind in ("quantize", "rtn"):
        w = s["w"]
        m, n = w.shape
        amax = w.abs().amax().to(F64)
        sg64 = amax / 2688.0
        s_g = float(sg64.to(F32))
        codes, packed = _outputs(m, n)
        h = s.get("h")
        h = torch.ones(n, dtype=F64, device=w.device) if h is None else h.to(F64)
        for r0, r1 in _rows(m, n):
            wr = w[r0:r1].to(F64)
            best, k = _search64(wr, h, s_g, case.get("start", "rtn"), case.get("down", 0), case.get("up", 0))
            codes[r0:r1], packed[r0:r1] = best.to(U8), _pack(wr, k)
        return {"global_scale": sg64.view(1), "codes": codes, "packed": packed}
    if kind == "output_error":
        w, n = s["w"].to(F64), case["n"]
        nib = torch.stack([s["packed"] & 15, s["packed"] >> 4], -1).view(w.shape).long()
        q = torch.tensor(_GRID, dtype=F64, device=w.device)[nib & 7] * (1 - 2 * (nib >> 3))
        scale = _e4m3(s["codes"].long()) * s["sg"].to(F64)
        dw = w - q * scale.repeat_interleave(16, 1)
        total = torch.zeros(1, dtype=F64, device=w.device)
        for t in range(0, case["tokens"], 2048):
            total += (s["x"][t:t + 2048].to(F64) @ dw.T).square().sum()
        return {"residual": None, "error": total}
    if kind == "factor":
        return {"U": _factor64(s["H"]), "dead": s["dead"], "info": s["info"]}
    if kind == "gptq":
        c, p = _gptq64(s["w"], s["U"], s["h"].to(F64), float(s["sg"]), case["block"], case["down"], case["up"])
        return {"codes": c, "packed": p}
    H = _hessian64(s["x"])
    # tiles of 128 x 256 wholly below the diagonal are not written by the accumulation
    n = case["n"]
    i, j = torch.arange(n, device=H.device), torch.arange(n, device=H.device)
    written = (j[None, :] // 256 + 1) * 256 > (i[:, None] // 128) * 128
    H_out = torch.where(written, H, torch.zeros((), dtype=F64, device=H.device))
    if kind == "hessian_full":
        return {"H": H_out}
    U = _factor64(H)
    sg64 = s["w"].abs().amax().to(F64) / 2688.0
    c, p = _gptq64(s["w"], U, torch.diagonal(H), float(sg64.to(F32)), case["block"], case["down"], case["up"])
    return {"H": H_out, "U": U, "global_scale": sg64.view(1), "codes": c, "packed": p}
