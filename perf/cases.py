"""Performance cases of the loop-program library, through its Python binding.

A case is one kind of call with its sizes; `prepare` makes what a user's program holds before
the call (the program handle with its device arena, host frames and operands, device matrices),
`run` is one pass of it.  Programs whose INIT loop makes the operands take the seed, the others
get host or device inputs drawn from it.

Kinds:
  six       the six-loop matrix program (init, C = 1.5 AB + 0.5 C, D = C + 2A, E = D^T, row sums,
            norm), every loop on the GPU
  gemm      init and GEMM alone (rectangular, optionally with power-of-two row factors on A)
  twelve    the twelve-loop program on an m x m result with inner dimension k
  host_gemm the GEMM on operands in pinned host memory, result back in pinned host memory
  image     the edge-detection program on a frame its INIT loop makes
  frame     the same program on a frame from pinned host memory
  residual  the binary64 residual check of a GEMM on device matrices
  colmax    column maxima of a device matrix without allocation
  batch     one gene over a suite of six-loop programs of mixed sizes
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_1806_01430_gb300 as gao

DEV = "cuda"
ALPHA, BETA = 1.5, 0.5
PREC = {"fp32": gao.FP32_SIMT, "bf16": gao.BF16, "bf16x3": gao.BF16X3, "bf16x6": gao.BF16X6, "fp8": gao.FP8}


def listed():
    return [
        # column maxima of one 1080p frame, the allocation-free call of a latency-critical loop
        {"name": "colmax_1080x1920", "kind": "colmax", "rows": 1080, "cols": 1920},
        # the smallest program of the benchmark set, default options, outputs read on the host
        {"name": "six_256_fp32", "kind": "six", "n": 256, "prec": "fp32", "fuse": 0, "read": "host"},
        # the matrix size of the paper's evaluation in the default precision
        {"name": "six_2048_fp32", "kind": "six", "n": 2048, "prec": "fp32", "fuse": 0, "read": "device"},
        # the six-loop benchmark: split bfloat16 with the loop chain in the GEMM's epilogue
        {"name": "six_4096_bf16x6_fused", "kind": "six", "n": 4096, "prec": "bf16x6", "fuse": 1, "read": "device"},
        # the headline GEMM program
        {"name": "gemm_8192_bf16x6", "kind": "gemm", "m": 8192, "n": 8192, "k": 8192, "prec": "bf16x6", "rowscale": 0},
        # a ragged block-scaled FP8 product (odd row length of B and C)
        {"name": "gemm_3000x5003x4100_fp8", "kind": "gemm", "m": 3000, "n": 5003, "k": 4100, "prec": "fp8", "rowscale": 0},
        # the twelve-loop program (element-wise chain and reductions after the GEMM chain)
        {"name": "twelve_6000x1500_bf16x3", "kind": "twelve", "m": 6000, "k": 1500, "prec": "bf16x3", "fuse": 1},
        # a product of operands that live on the host, result wanted there
        {"name": "host_gemm_4096_bf16x6", "kind": "host_gemm", "m": 4096, "n": 4096, "k": 4096, "prec": "bf16x6"},
        # the edge-detection benchmark frame, edge energy and column maxima in one pass
        {"name": "image_8192_fused", "kind": "image", "h": 8192, "w": 8192, "fuse": 1, "maps": 0},
        # a 4K camera frame from the host, the edge map wanted back
        {"name": "frame_2160x3840", "kind": "frame", "h": 2160, "w": 3840, "fuse": 1, "maps": 1},
        # verifying a product on the device
        {"name": "residual_4096", "kind": "residual", "m": 4096, "n": 4096, "k": 4096},
        # a generation's all-GPU individual over a suite of mixed sizes
        {"name": "batch_16_bf16x3", "kind": "batch", "programs": 16, "lo": 128, "hi": 2048, "sizes": 2000,
         "prec": "bf16x3", "fuse": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """Log-uniform; about half the sizes odd or ragged, the others multiples of 64 or 4."""
    n = _log(rng, lo, hi)
    pick = rng.random()
    if pick < 0.3:
        n = max(64, n // 64 * 64)
    elif pick < 0.5:
        n = max(4, n // 4 * 4)
    return n


def draw(rng):
    kind = rng.choice(["six", "six", "six", "gemm", "gemm", "twelve", "host_gemm", "image", "image", "frame", "residual",
                       "colmax", "batch"])
    if kind == "six":
        prec = rng.choice(["fp32", "fp32", "bf16x6", "bf16x3", "bf16", "fp8"])
        n = _size(rng, 128, 3000 if prec == "fp32" else 5000)
        return {"kind": kind, "n": n, "prec": prec, "fuse": rng.randint(0, 1), "read": rng.choice(["host", "device"])}
    if kind == "gemm":
        return {"kind": kind, "m": _size(rng, 256, 7000), "n": _size(rng, 256, 7000), "k": _size(rng, 128, 7000),
                "prec": rng.choice(["bf16x6", "bf16x3", "bf16", "fp8"]), "rowscale": int(rng.random() < 0.25)}
    if kind == "twelve":
        return {"kind": kind, "m": _size(rng, 500, 6000), "k": _size(rng, 128, 2000),
                "prec": rng.choice(["fp32", "bf16x3", "bf16x6"]) if rng.random() < 0.7 else "bf16", "fuse": rng.randint(0, 1)}
    if kind == "host_gemm":
        return {"kind": kind, "m": _size(rng, 256, 4096), "n": _size(rng, 256, 4096), "k": _size(rng, 256, 4096),
                "prec": rng.choice(["bf16x6", "bf16x3", "bf16"])}
    if kind == "image":
        return {"kind": kind, "h": _size(rng, 240, 8000), "w": _size(rng, 320, 8000), "fuse": rng.randint(0, 1),
                "maps": rng.randint(0, 1)}
    if kind == "frame":
        return {"kind": kind, "h": _size(rng, 240, 4500), "w": _size(rng, 320, 8000), "fuse": rng.randint(0, 1),
                "maps": rng.randint(0, 1)}
    if kind == "residual":
        return {"kind": kind, "m": _size(rng, 256, 6000), "n": _size(rng, 256, 6000), "k": _size(rng, 256, 6000)}
    if kind == "colmax":
        return {"kind": kind, "rows": _size(rng, 64, 8192), "cols": _size(rng, 64, 8192)}
    return {"kind": kind, "programs": rng.randint(6, 20), "lo": 128, "hi": rng.choice([512, 1024, 2048]),
            "sizes": rng.randint(0, 9999), "prec": rng.choice(["bf16x3", "bf16x6"]), "fuse": rng.randint(0, 1)}


# ---- programs ------------------------------------------------------------------------------


def _buf(rows, cols, role=gao.TEMP, dtype=gao.F32):
    return SimpleNamespace(rows=rows, cols=cols, role=role, dtype=dtype)


def _loop(kind, ins, outs, alpha=0.0, beta=0.0, flags=0):
    return SimpleNamespace(kind=kind, ins=ins, outs=outs, alpha=alpha, beta=beta, flags=flags)


def _six(n):
    o = gao.OUTPUT
    bufs = [_buf(n, n), _buf(n, n), _buf(n, n, o), _buf(n, n), _buf(n, n), _buf(n, 1, o), _buf(1, 1, o, gao.F64)]
    A, B, C, D, E, r, f = range(7)
    loops = [_loop(gao.INIT, [], [A, B, C]), _loop(gao.GEMM, [A, B, C], [C], ALPHA, BETA),
             _loop(gao.AXPY, [C, A], [D], 2.0), _loop(gao.TRANSPOSE, [D], [E]), _loop(gao.ROWSUM, [E], [r]),
             _loop(gao.FROBENIUS, [E], [f])]
    return bufs, loops, {"C": C, "r": r, "f": f}


def _gemm(m, n, k, rowscale):
    bufs = [_buf(m, k), _buf(k, n), _buf(m, n), _buf(m, n, gao.OUTPUT)]
    loops = [_loop(gao.INIT, [], [0, 1, 2], flags=1 if rowscale else 0), _loop(gao.GEMM, [0, 1, 2], [3], ALPHA, BETA)]
    return bufs, loops, {"C": 3}


def _host_gemm(m, n, k):
    i = gao.INPUT
    bufs = [_buf(m, k, i), _buf(k, n, i), _buf(m, n, i), _buf(m, n, gao.OUTPUT)]
    return bufs, [_loop(gao.GEMM, [0, 1, 2], [3], ALPHA, BETA)], {"C": 3}


def _twelve(m, k):
    o = gao.OUTPUT
    A, B, C, S, D, E, r, f, F, G, H, P, q, s = range(14)
    bufs = [_buf(m, k), _buf(k, m), _buf(m, m, o)] + [_buf(m, m) for _ in range(3)]
    bufs += [_buf(m, 1, o), _buf(1, 1, o, gao.F64)] + [_buf(m, m) for _ in range(4)]
    bufs += [_buf(1, m, o), _buf(1, 1, o, gao.F64)]
    loops = [_loop(gao.INIT, [], [A, B, C, S]), _loop(gao.GEMM, [A, B, C], [C], ALPHA, BETA),
             _loop(gao.AXPY, [C, S], [D], 2.0), _loop(gao.TRANSPOSE, [D], [E]), _loop(gao.ROWSUM, [E], [r]),
             _loop(gao.FROBENIUS, [E], [f]), _loop(gao.RELU, [E], [F]), _loop(gao.AXPY, [E, F], [G], -0.5),
             _loop(gao.SQUARE, [G], [H]), _loop(gao.AXPY, [H, D], [P], 0.25), _loop(gao.COLMAX, [P], [q]),
             _loop(gao.SUM, [P], [s])]
    return bufs, loops, {"C": C, "r": r, "f": f, "q": q, "s": s}


def _image(h, w, host, maps):
    X, B, gx, gy, sx, sy, M2, e, q = range(9)
    bufs = [_buf(h, w) for _ in range(7)] + [_buf(1, 1, gao.OUTPUT, gao.F64), _buf(1, w, gao.OUTPUT)]
    if host:
        bufs[X].role = gao.INPUT
    if maps:
        bufs[M2].role = gao.OUTPUT
    loops = [] if host else [_loop(gao.INIT, [], [X])]
    loops += [_loop(gao.STENCIL3, [X], [B], flags=gao.STENCIL_BLUR),
              _loop(gao.STENCIL3, [B], [gx], flags=gao.STENCIL_SOBEL_X),
              _loop(gao.STENCIL3, [B], [gy], flags=gao.STENCIL_SOBEL_Y), _loop(gao.SQUARE, [gx], [sx]),
              _loop(gao.SQUARE, [gy], [sy]), _loop(gao.AXPY, [sx, sy], [M2], 1.0), _loop(gao.SUM, [M2], [e]),
              _loop(gao.COLMAX, [M2], [q])]
    outs = {"e": e, "q": q}
    if maps:
        outs["M2"] = M2
    return bufs, loops, outs


def _init_seed(seed):
    return (seed * 2654435761) % (1 << 24)


def _device_prog(spec, prec, seed, fuse):
    """The program on a device arena of the caller's, and its outputs as tensors over the arena."""
    bufs, loops, outs = spec
    nbytes = gao.prog_device_bytes(bufs, loops, gemm_prec=PREC[prec])
    raw = torch.empty(nbytes + 1024, dtype=torch.uint8, device=DEV)
    arena = raw[-raw.data_ptr() % 1024:][:nbytes]
    torch.cuda.synchronize()  # the library's stream is not torch's
    p = gao.prog_create(bufs, loops, seed=_init_seed(seed), gemm_prec=PREC[prec], fuse_chains=fuse, arena=arena)
    views = {}
    for name, b in outs.items():
        off = gao.prog_device_ptr(p, b) - arena.data_ptr()
        dt = torch.float64 if bufs[b].dtype == gao.F64 else torch.float32
        size = bufs[b].rows * bufs[b].cols * dt.itemsize
        views[name] = arena[off:off + size].view(dt).view(bufs[b].rows, bufs[b].cols)
    return p, views


def _prog_state(spec, prec, seed, fuse, read):
    gene = (1 << len(spec[1])) - 1
    if read == "host":
        bufs, loops, outs = spec
        p = gao.prog_create(bufs, loops, seed=_init_seed(seed), gemm_prec=PREC[prec], fuse_chains=fuse)
        return {"p": p, "gene": gene, "flags": 0, "host": outs, "views": None}
    p, views = _device_prog(spec, prec, seed, fuse)
    return {"p": p, "gene": gene, "flags": gao.RUN_KEEP_DEVICE | gao.RUN_NO_LOOP_TIMES, "host": None, "views": views}


def _batch_sizes(case):
    r = random.Random(case["sizes"])
    return [_log(r, case["lo"], case["hi"]) for _ in range(case["programs"])]


# ---- inputs --------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _normal(seed, *shape):
    return torch.randn(*shape, generator=_gen(seed), device=DEV, dtype=torch.float32)


def _frame(seed, h, w):
    """A camera-like frame in [0, 1]: smooth shading, a few edges and sensor noise."""
    r = random.Random(seed)
    y = torch.linspace(0, 1, h, device=DEV)[:, None]
    x = torch.linspace(0, 1, w, device=DEV)[None, :]
    X = 0.5 + 0.2 * torch.sin(6.0 * x + r.uniform(0, 6)) * torch.cos(5.0 * y + r.uniform(0, 6))
    for _ in range(6):
        a, c = r.uniform(-2, 2), r.uniform(-1, 2)
        X = X + r.uniform(-0.15, 0.15) * (y > a * x + c)
    X = X + 0.01 * _normal(seed, h, w)
    return X.clamp_(0, 1).float()


def _residual_inputs(case, seed):
    m, n, k = case["m"], case["n"], case["k"]
    A, B, C0 = _normal(seed, m, k), _normal(seed + 1, k, n), _normal(seed + 2, m, n)
    # the product being checked: bfloat16 operands, binary32 accumulation
    C = ALPHA * (A.bfloat16().float() @ B.bfloat16().float()) + BETA * C0
    g = _gen(seed + 3)
    x = torch.randint(0, 2, (n,), generator=g, device=DEV).double() * 2 - 1
    y = torch.randint(0, 2, (m,), generator=g, device=DEV).double() * 2 - 1
    return A, B, C0, C, x, y


def prepare(case, seed):
    kind = case["kind"]
    if kind == "six":
        return _prog_state(_six(case["n"]), case["prec"], seed, case["fuse"], case["read"])
    if kind == "gemm":
        return _prog_state(_gemm(case["m"], case["n"], case["k"], case["rowscale"]), case["prec"], seed, 0, "device")
    if kind == "twelve":
        return _prog_state(_twelve(case["m"], case["k"]), case["prec"], seed, case["fuse"], "device")
    if kind == "image":
        return _prog_state(_image(case["h"], case["w"], False, case["maps"]), "fp32", seed, case["fuse"], "device")
    if kind == "frame":
        st = _prog_state(_image(case["h"], case["w"], True, case["maps"]), "fp32", seed, case["fuse"], "host")
        frame = _frame(seed, case["h"], case["w"]).cpu().pin_memory()
        gao.prog_bind_host(st["p"], 0, frame)
        st["flags"] = gao.RUN_NO_LOOP_TIMES
        if case["maps"]:  # the edge map straight into the caller's own pinned frame
            M2 = torch.empty(case["h"], case["w"]).pin_memory()
            gao.prog_bind_host(st["p"], st["host"].pop("M2"), M2)
            st["views"] = {"M2": M2}
        return st
    if kind == "host_gemm":
        bufs, loops, outs = _host_gemm(case["m"], case["n"], case["k"])
        p = gao.prog_create(bufs, loops, gemm_prec=PREC[case["prec"]])
        for i in range(3):
            gao.prog_bind_host(p, i, _normal(seed * 3 + i, bufs[i].rows, bufs[i].cols).cpu().pin_memory())
        C = torch.empty(bufs[3].rows, bufs[3].cols).pin_memory()
        gao.prog_bind_host(p, 3, C)
        return {"p": p, "gene": 1, "flags": gao.RUN_NO_LOOP_TIMES, "host": None, "views": {"C": C}}
    if kind == "residual":
        A, B, C0, C, x, y = _residual_inputs(case, seed)
        nbytes = gao.gao_gemm_residual_scratch(case["m"], case["n"], case["k"])
        return {"in": (A, B, C0, C, x, y), "scratch": torch.empty(nbytes, dtype=torch.uint8, device=DEV),
                "r": torch.empty(case["m"], dtype=torch.float64, device=DEV),
                "s": torch.empty(case["n"], dtype=torch.float64, device=DEV), "shape": (case["m"], case["n"], case["k"])}
    if kind == "colmax":
        return {"X": _normal(seed, case["rows"], case["cols"]), "q": torch.empty(case["cols"], device=DEV)}
    progs, views = [], []
    for i, n in enumerate(_batch_sizes(case)):
        p, v = _device_prog(_six(n), case["prec"], seed + i, case["fuse"])
        progs.append(p)
        views.append(v)
    return {"batch": gao.batch_create(progs), "gene": 0b111111, "views": views}


def run(state):
    if "p" in state:
        p = state["p"]
        gao.prog_run(p, state["gene"], state["flags"])
        out = {} if state["views"] is None else dict(state["views"])
        if state["host"] is not None:
            out.update({name: gao.prog_output(p, b) for name, b in state["host"].items()})
        return out
    if "batch" in state:
        # changing the replica count forgets the measured times, so the gene is measured again
        gao.batch_set_replicas(state["batch"], 1)
        gao.batch_evaluate(state["batch"], [state["gene"]])
        return state["views"]
    if "q" in state:
        X = state["X"]
        st = gao.gao_colmax_noalloc(X.data_ptr(), X.shape[0], X.shape[1], state["q"].data_ptr(),
                                    torch.cuda.current_stream())
        if st != gao.GAO_OK:
            raise RuntimeError(gao.gao_last_error())
        return state["q"]
    A, B, C0, C, x, y = state["in"]
    m, n, k = state["shape"]
    norms = gao.gao_gemm_residual(A.data_ptr(), B.data_ptr(), C0.data_ptr(), C.data_ptr(), m, n, k, ALPHA, BETA,
                                  x.data_ptr(), y.data_ptr(), state["scratch"].data_ptr(), state["scratch"].numel(),
                                  state["r"].data_ptr(), state["s"].data_ptr(), torch.cuda.current_stream())
    return {"r": state["r"], "s": state["s"], "norms": norms}


# ---- what a pass cannot do without -----------------------------------------------------------


def work(case):
    kind = case["kind"]
    if kind == "six":
        n = case["n"]
        return {"bytes": 4 * n * n + 4 * n + 8, "flops": 2 * n ** 3}
    if kind in ("gemm", "host_gemm"):
        m, n, k = case["m"], case["n"], case["k"]
        read = 4 * (m * k + k * n + m * n) if kind == "host_gemm" else 0
        return {"bytes": read + 4 * m * n, "flops": 2 * m * n * k}
    if kind == "twelve":
        m, k = case["m"], case["k"]
        return {"bytes": 4 * m * m + 8 * m + 16, "flops": 2 * m * m * k}
    if kind in ("image", "frame"):
        h, w = case["h"], case["w"]
        return {"bytes": 4 * h * w * (1 + case["maps"]) + 4 * w + 8, "flops": 45 * h * w}
    if kind == "residual":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 4 * (m * k + k * n + 2 * m * n) + 16 * (m + n), "flops": 4 * (m * k + k * n + 2 * m * n)}
    if kind == "colmax":
        return {"bytes": 4 * (case["rows"] + 1) * case["cols"], "flops": case["rows"] * case["cols"]}
    sizes = _batch_sizes(case)
    return {"bytes": sum(4 * n * n + 4 * n + 8 for n in sizes), "flops": sum(2 * n ** 3 for n in sizes)}


# ---- the same results in 64 bits ---------------------------------------------------------------


def _shr(z, s):
    return (z >> s) & ((1 << (64 - s)) - 1)


def _i64(c):
    return c - (1 << 64) if c >= 1 << 63 else c


def _hash(state):
    """SplitMix64 (Steele, Lea & Flood 2014) of int64 states, wrapping."""
    z = state + _i64(0x9E3779B97F4A7C15)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _init(seed, buf, rows, cols):
    """Buffer `buf` of an INIT loop: two 24-bit values of U[-1, 1) per hash."""
    n = rows * cols
    key = _i64((seed << 40) & ((1 << 64) - 1)) ^ (buf << 36)
    h = _hash(torch.arange((n + 1) // 2, dtype=torch.int64, device=DEV) ^ key)
    u = torch.stack([_shr(h, 40), (h >> 16) & 0xFFFFFF], dim=1).reshape(-1)[:n]
    return ((u - (1 << 23)).double() / float(1 << 23)).view(rows, cols)


def _row_factors(seed, rows):
    """2^e per row, e in [-10, 10] from twelve 24-bit uniforms."""
    key = _i64((seed << 40) & ((1 << 64) - 1)) ^ (15 << 36)
    s = _shr(_hash(torch.arange(12 * rows, dtype=torch.int64, device=DEV) ^ key), 40).view(rows, 12).sum(1)
    num, den = (s - 6 * (1 << 24)) * 10, 3 * (1 << 24)
    e = torch.div(2 * num + den, 2 * den, rounding_mode="floor").clamp(-10, 10)
    return torch.pow(torch.full((rows, 1), 2.0, dtype=torch.float64, device=DEV), e.double()[:, None])


def _six_exact(n, seed):
    A, B, C = (_init(seed, b, n, n) for b in range(3))
    C = ALPHA * (A @ B) + BETA * C
    D = C + 2.0 * A
    return {"C": C, "r": D.sum(0)[:, None], "f": D.square().sum().sqrt().view(1, 1)}


def _stencil(X, w):
    """Zero-padded 3 x 3 correlation in binary64."""
    P = torch.nn.functional.pad(X[None, None], (1, 1, 1, 1))[0, 0]
    h, wd = X.shape
    out = torch.zeros_like(X)
    for a in range(3):
        for b in range(3):
            if w[a][b]:
                out += w[a][b] * P[a:a + h, b:b + wd]
    return out


def _image_exact(X, maps):
    B = _stencil(X, [[0.0625, 0.125, 0.0625], [0.125, 0.25, 0.125], [0.0625, 0.125, 0.0625]])
    gx = _stencil(B, [[-1, 0, 1], [-2, 0, 2], [-1, 0, 1]])
    gy = _stencil(B, [[-1, -2, -1], [0, 0, 0], [1, 2, 1]])
    M2 = gx.square_().add_(gy.square_())
    out = {"e": M2.sum().view(1, 1), "q": M2.amax(0, keepdim=True)}
    if maps:
        out["M2"] = M2
    return out


def exact(case, seed):
    kind, s = case["kind"], _init_seed(seed)
    if kind == "six":
        return _six_exact(case["n"], s)
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        A = _init(s, 0, m, k)
        if case["rowscale"]:
            A *= _row_factors(s, m)
        return {"C": ALPHA * (A @ _init(s, 1, k, n)) + BETA * _init(s, 2, m, n)}
    if kind == "twelve":
        m, k = case["m"], case["k"]
        C = ALPHA * (_init(s, 0, m, k) @ _init(s, 1, k, m)) + BETA * _init(s, 2, m, m)
        D = C + 2.0 * _init(s, 3, m, m)
        E = D.t()
        P = (E - 0.5 * E.clamp(min=0)).square() + 0.25 * D
        return {"C": C, "r": E.sum(1)[:, None], "f": E.square().sum().sqrt().view(1, 1),
                "q": P.amax(0, keepdim=True), "s": P.sum().view(1, 1)}
    if kind == "host_gemm":
        m, n, k = case["m"], case["n"], case["k"]
        A, B, C0 = (_normal(seed * 3 + i, *d).double() for i, d in enumerate([(m, k), (k, n), (m, n)]))
        return {"C": (ALPHA * (A @ B) + BETA * C0).cpu()}
    if kind == "image":
        return _image_exact(_init(s, 0, case["h"], case["w"]), case["maps"])
    if kind == "frame":
        return {name: v.cpu() for name, v in _image_exact(_frame(seed, case["h"], case["w"]).double(), case["maps"]).items()}
    if kind == "residual":
        A, B, C0, C, x, y = _residual_inputs(case, seed)
        A, B, C0, C = (t.double() for t in (A, B, C0, C))
        f, g = ALPHA * (A @ (B @ x)) + BETA * (C0 @ x), ALPHA * ((y @ A) @ B) + BETA * (y @ C0)
        r, t = C @ x - f, y @ C - g
        norms = {"right": (r.norm() / f.norm()).item(), "left": (t.norm() / g.norm()).item(),
                 "right_inf": (r.abs().max() / f.abs().max()).item(), "left_inf": (t.abs().max() / g.abs().max()).item(),
                 "right_argmax": None, "left_argmax": None}
        return {"r": r, "s": t, "norms": norms}
    if kind == "colmax":
        return _normal(seed, case["rows"], case["cols"]).double().amax(0)
    return [_six_exact(n, _init_seed(seed + i)) for i, n in enumerate(_batch_sizes(case))]
