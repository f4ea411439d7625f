"""The work that users of this library have it do, as measurable cases.

A case is one call sequence through the public binding
(paper_1901_06043_gb300.tucker): ST-HOSVD compressions in the precisions the
library offers (from device or host memory, one tensor or a batch, in the
natural or a given mode order), HOSVD, reconstructions, pre-/post-processing,
and the single steps a driver composes (Gram, truncated eigensolve, TTM).
Sizes come from the benchmark's and the tests' workloads (40x50x30,
200x200x200x50, 256x256x256x11xT, 500x500x500x11x8, batches of cubes and 4-way
tensors, mode sizes of 1500) and odd sizes between them; tensors are the
seeded Tucker tensors of synth.py (decaying core, orthonormal factors, noise).

Outputs.  Eigenvector signs are free, and vectors of neighbouring eigenvalues
near the cut are only determined up to the Gram's rounding, so a compression
returns its ranks, all eigenvalues, and a tensor rebuilt from core and
factors; single steps run with a given rank and return absolute values where
a vector's sign enters.
"""
import math

import numpy as np
import torch

from paper_1901_06043_gb300 import synth, tucker


def _ints(text):
    return tuple(int(v) for v in text.split("x"))


def _text(dims):
    return "x".join(str(int(v)) for v in dims)


def _prod(dims):
    return int(math.prod(int(d) for d in dims))


def listed():
    return [
        # a small double-precision compression with full reconstruction: launches and latency
        {"name": "compress small f64", "kind": "compress", "dims": "40x50x30", "core": "5x6x4",
         "decay": 0.0, "eta": 1e-4, "eps": 1e-3, "dtype": "f64", "prec": "fp64", "part": "40x50x30"},
        # a 3.2 GB double-precision run; one time step looked at afterwards
        {"name": "compress 4-way f64", "kind": "compress", "dims": "200x200x200x50",
         "core": "30x30x30x12", "decay": 0.15, "eta": 1e-6, "eps": 1e-4, "dtype": "f64",
         "prec": "fp64", "part": "200x200x200x1"},
        # a combustion-shaped run at low accuracy (space^3, 11 species, time)
        {"name": "compress 5-way mixed 1e-2", "kind": "compress", "dims": "256x256x256x11x8",
         "core": "40x40x40x11x8", "decay": 0.1, "eta": 1e-7, "eps": 1e-2, "dtype": "f32",
         "prec": "mixed", "part": "256x256x256x11x1"},
        # the benchmark's tensor, 44 GB
        {"name": "compress large mixed 1e-4", "kind": "compress", "dims": "500x500x500x11x8",
         "core": "60x60x60x11x6", "decay": 0.08, "eta": 1e-7, "eps": 1e-4, "dtype": "f32",
         "prec": "mixed", "part": "500x500x500x11x1"},
        # a snapshot that arrives in pinned host memory, odd sizes
        {"name": "compress host mixed", "kind": "host", "dims": "301x203x157x9",
         "core": "24x20x18x9", "decay": 0.12, "eta": 1e-6, "eps": 1e-4, "dtype": "f32",
         "prec": "mixed", "part": "301x203x157x1"},
        # given mode order (last mode first), plain single precision: strided views
        {"name": "compress order f32", "kind": "compress", "dims": "161x144x150x32",
         "core": "20x20x20x10", "decay": 0.12, "eta": 1e-5, "eps": 1e-3, "dtype": "f32",
         "prec": "fp32", "order": "3x2x1x0", "part": "161x144x150x1"},
        # many small tensors at once
        {"name": "batch mixed", "kind": "batch", "count": 64, "lo": 48, "hi": 256, "decay": 0.2,
         "eta": 1e-6, "eps": 1e-4, "dtype": "f32", "prec": "mixed"},
        # decompression of one time step of the benchmark's tensor
        {"name": "reconstruct mixed", "kind": "rebuild", "core": "54x54x54x11x6",
         "dims": "500x500x500x11x1", "decay": 0.08, "dtype": "f32", "prec": "mixed"},
        # full double-precision decompression
        {"name": "reconstruct f64", "kind": "rebuild", "core": "26x26x26x12",
         "dims": "200x200x200x50", "decay": 0.15, "dtype": "f64", "prec": "fp64"},
        # standardize every species, and back
        {"name": "standardize f32", "kind": "prepost", "dims": "250x250x250x11x4", "mode": 3,
         "method": "standardize", "dtype": "f32"},
        # the eigenvalue step at a large mode size
        {"name": "eigensolve 1500", "kind": "eig", "n": 1500, "rank": 401, "tail": 1e-10},
        # the steps of one middle mode, as a driver of its own calls them
        {"name": "mode step f64", "kind": "step", "dims": "151x149x163", "mode": 1,
         "core": "20x18x16", "decay": 0.15, "eta": 1e-6, "eps": 1e-4, "dtype": "f64",
         "prec": "fp64"},
    ]


# ---------------------------------------------------------------- drawn cases

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, most, first=512):
    """3 to 5 modes of sizes a run has: large ones first, then few species and time steps."""
    while True:
        n = rng.choice((3, 4, 4, 5))
        dims = [_log(rng, 24, first) for _ in range(3)]
        if n >= 4:
            dims.append(_log(rng, 5, 64))
        if n == 5:
            dims.append(_log(rng, 2, 16))
        if 2e4 <= _prod(dims) <= most:
            return dims


def draw(rng):
    kind = rng.choice(("compress", "compress", "compress", "compress", "host", "batch", "rebuild",
                       "rebuild", "prepost", "eig", "step", "step"))
    if kind == "eig":
        n = _log(rng, 16, 1500)
        return {"kind": "eig", "n": n, "rank": max(2, n // rng.randint(3, 8)),
                "tail": rng.choice((1e-6, 1e-8, 1e-10))}
    if kind == "batch":
        lo = rng.randint(24, 64)
        return {"kind": "batch", "count": rng.randint(8, 48), "lo": lo,
                "hi": lo + rng.randint(32, 128), "decay": 0.2, "eta": 1e-6,
                "eps": rng.choice((1e-2, 1e-3, 1e-4)), "dtype": "f32",
                "prec": rng.choice(("mixed", "mixed", "fp32"))}
    if kind == "prepost":
        dims = _shape(rng, 7e8)
        return {"kind": "prepost", "dims": _text(dims), "mode": rng.randrange(len(dims)),
                "method": rng.choice(("standardize", "standardize", "max")),
                "dtype": rng.choice(("f32", "f32", "f64"))}
    dtype, prec = rng.choice((("f64", "fp64"), ("f64", "fp64"), ("f32", "mixed"), ("f32", "mixed"),
                              ("f32", "fp64"), ("f32", "fp32")))
    dims = _shape(rng, {"fp64": 2e8, "fp32": 5e8, "mixed": 1.5e9}[prec],
                  320 if prec == "fp64" else 512)
    core = [max(2, min(d, 12 if k > 2 else d // rng.randint(4, 9))) for k, d in enumerate(dims)]
    case = {"kind": kind, "dims": _text(dims), "core": _text(core),
            "decay": rng.choice((0.1, 0.15, 0.2)), "dtype": dtype, "prec": prec}
    if kind == "rebuild":
        return case
    case.update(eta=1e-6, eps=rng.choice((1e-2, 1e-3, 1e-4)))
    if kind == "step":
        return dict(case, mode=rng.randrange(3))
    case["part"] = _text([d if k < 2 else rng.randint(1, d) for k, d in enumerate(dims)])
    if kind == "compress" and rng.random() < 0.3:
        order = list(range(len(dims)))
        rng.shuffle(order)
        case["order"] = _text(order)
    elif kind == "compress" and rng.random() < 0.2:
        case["kind"] = "hosvd"
    return case


# ------------------------------------------------------------------- inputs

def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _tensor(case, seed):
    return synth.tucker_torch(_ints(case["dims"]), _ints(case["core"]), case["decay"],
                              case["eta"], seed, _dtype(case))


def _batch(case, seed):
    """(dims, core) per tensor: cubes and 4-way tensors in turn.  The shapes
    belong to the case; the seed draws the values."""
    rng = np.random.default_rng(1000 + case["count"] + 7 * case["lo"] + 131 * case["hi"])
    out = []
    for k in range(case["count"]):
        if k % 2 == 0:
            dims = (int(rng.integers(case["lo"], case["hi"] + 1)),) * 3
        else:
            lo, hi = (case["lo"] * 2) // 3, (case["hi"] * 5) // 8
            dims = tuple(int(v) for v in rng.integers(lo, hi + 1, size=3)) + (
                int(rng.integers(4, 17)),)
        out.append((dims, tuple(min(d, int(rng.integers(8, 33))) for d in dims)))
    return out


def _spectrum(case, seed):
    """A Gram matrix with the spectrum of a Tucker mode: `rank` values falling
    geometrically to sqrt(tail) of the largest, then a noise floor."""
    n, r = case["n"], case["rank"]
    gen = torch.Generator("cuda").manual_seed(int(seed))
    k = 2 * n + 64
    s = torch.pow(10.0, torch.linspace(0.0, 0.5 * math.log10(case["tail"]), r, device="cuda",
                                       dtype=torch.float64))
    a = torch.randn(n, r, generator=gen, device="cuda", dtype=torch.float64) / math.sqrt(n)
    b = torch.randn(r, k, generator=gen, device="cuda", dtype=torch.float64) / math.sqrt(k)
    x = (a * s) @ b
    x += 1e-3 * math.sqrt(case["tail"] / (n * k)) * torch.randn(n, k, generator=gen, device="cuda",
                                                              dtype=torch.float64)
    S = x @ x.T
    return (S + S.T).mul_(0.5).contiguous()


def prepare(case, seed):
    st = {"case": case, "ctx": tucker.Context()}
    kind = case["kind"]
    if kind == "eig":
        st["S"] = _spectrum(case, seed)
    elif kind == "batch":
        shapes = _batch(case, seed)
        st["dims"] = [d for d, _ in shapes]
        st["xs"] = [synth.tucker_torch(d, c, case["decay"], case["eta"], 64 * seed + k,
                                       _dtype(case)) for k, (d, c) in enumerate(shapes)]
    elif kind == "prepost":
        dims = _ints(case["dims"])
        gen = torch.Generator("cuda").manual_seed(int(seed))
        N, m = len(dims), case["mode"]
        x = torch.randn(tuple(reversed(dims)), generator=gen, device="cuda", dtype=_dtype(case))
        # fields of their own offset and scale per slice
        sh = [1] * N
        sh[N - 1 - m] = dims[m]
        x.mul_(torch.exp(torch.randn(sh, generator=gen, device="cuda", dtype=x.dtype)))
        x.add_(3.0 * torch.randn(sh, generator=gen, device="cuda", dtype=x.dtype))
        st["x"] = x.reshape(-1)
    elif kind == "rebuild":
        core, dims = _ints(case["core"]), _ints(case["dims"])
        gen = torch.Generator("cuda").manual_seed(int(seed))
        idx = sum(torch.arange(c, device="cuda", dtype=torch.float64).reshape(
            [c if a == len(core) - 1 - n else 1 for a in range(len(core))])
            for n, c in enumerate(core))
        g = torch.randn(tuple(reversed(core)), generator=gen, device="cuda", dtype=torch.float64)
        st["core"] = (g * torch.pow(10.0, -case["decay"] * idx)).to(_dtype(case)).reshape(-1)
        # rows of orthonormal factors (random signs and sizes), stored column-major
        st["mats"] = [(torch.randn(c, d, generator=gen, device="cuda", dtype=torch.float64)
                       / math.sqrt(d)).t() for c, d in zip(core, dims)]
    else:
        st["x"] = _tensor(case, seed)
        if kind == "host":
            st["x"] = st["x"].cpu().pin_memory()
    torch.cuda.empty_cache()
    return st


# ------------------------------------------------------------------ one pass

def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "eig":
        w, U, R, disc = ctx.eig_trunc(st["S"], R=case["rank"])
        return {"eigvals": w, "vectors": U.abs()}
    if kind == "batch":
        res = ctx.sthosvd_batched(st["xs"], st["dims"], case["eps"], prec=case["prec"])
        out = {"ranks": np.array([r for q in res for r in q.ranks]),
               "eigvals": torch.cat([w for q in res for w in q.eigvals]),
               "slices": torch.cat([q.reconstruct([0] * len(d), d[:2] + (1,) * (len(d) - 2),
                                                  prec=case["prec"])
                                    for q, d in zip(res, st["dims"])])}
        for q in res:
            q.close()
        return out
    if kind == "prepost":
        y, shift, scale = ctx.preprocess(st["x"], _ints(case["dims"]), case["mode"],
                                         case["method"])
        back = ctx.slice_transform(y, _ints(case["dims"]), case["mode"], shift, scale,
                                   inverse=True)
        return {"y": y, "shift": shift, "scale": scale, "back": back}
    if kind == "rebuild":
        return ctx.multi_ttm(st["core"], _ints(case["core"]), st["mats"], _ints(case["dims"]),
                             prec=case["prec"])
    dims = _ints(case["dims"])
    if kind == "step":
        S = ctx.gram(st["x"], dims, case["mode"], prec=case["prec"])
        w, U, R, disc = ctx.eig_trunc(S, R=_ints(case["core"])[case["mode"]])
        z = ctx.ttm(st["x"], dims, case["mode"], U.t(), prec=case["prec"],
                    out_dtype=None if case["prec"] != "fp64" else tucker.F64)
        return {"gram": S, "eigvals": w, "z": z.abs()}
    if kind == "host":
        res = ctx.sthosvd_host(st["x"], dims, eps=case["eps"], prec=case["prec"])
    elif kind == "hosvd":
        res = ctx.hosvd(st["x"], dims, eps=case["eps"], prec=case["prec"])
    else:
        res = ctx.sthosvd(st["x"], dims, eps=case["eps"], prec=case["prec"],
                          mode_order=_ints(case["order"]) if "order" in case else None)
    out = {"ranks": list(res.ranks), "eigvals": res.eigvals,
           "part": res.reconstruct([0] * len(dims), _ints(case["part"]), prec=case["prec"])}
    res.close()
    return out


# ---------------------------------------------------------------------- work

def _chain(dims, core, order=None, gram=True):
    """Multiply-add flops of a compression: per mode the symmetric Gram and the TTM."""
    cur, f = list(dims), 0.0
    for n in (order or range(len(dims))):
        m = float(_prod(cur))
        f += (m * (cur[n] + 1) if gram else 0.0) + 2.0 * m * core[n]
        cur[n] = core[n]
    return f


def _expand(core, dims):
    cur, f = list(core), 0.0
    for n in sorted(range(len(core)), key=lambda k: dims[k] / core[k]):
        f += 2.0 * _prod(cur) * dims[n]
        cur[n] = dims[n]
    return f


def work(case):
    kind = case["kind"]
    if kind == "eig":
        n, r = case["n"], case["rank"]
        return {"bytes": 8.0 * (n * n + n * r + n), "flops": 4.0 / 3.0 * n ** 3 + 4.0 * n * n * r}
    es = 8 if case["dtype"] == "f64" else 4
    if kind == "batch":
        sh = _batch(case, 0)
        return {"bytes": float(es * sum(_prod(d) + _prod(c) for d, c in sh)),
                "flops": sum(_chain(d, c) for d, c in sh)}
    dims = _ints(case["dims"])
    if kind == "prepost":
        return {"bytes": 4.0 * es * _prod(dims), "flops": 12.0 * _prod(dims)}
    core = _ints(case["core"])
    if kind == "rebuild":
        return {"bytes": float(es * (_prod(core) + _prod(dims))), "flops": _expand(core, dims)}
    os_ = 8 if case["prec"] == "fp64" else es
    if kind == "step":
        m = case["mode"]
        n = _prod(dims)
        return {"bytes": float(es * n + os_ * (n // dims[m]) * core[m] + 8 * dims[m] ** 2),
                "flops": n * (dims[m] + 1.0) + 2.0 * n * core[m]}
    part = _ints(case["part"])
    order = _ints(case["order"]) if "order" in case else None
    flops = _chain(dims, core, order) + _expand(core, part)
    if kind == "hosvd":
        flops = sum(_prod(dims) * (d + 1.0) for d in dims) + _chain(dims, core, None, False) + \
            _expand(core, part)
    return {"bytes": float(es * _prod(dims) + os_ * (_prod(core) + _prod(part)) +
                           8 * sum(d * c for d, c in zip(dims, core))), "flops": flops}


def tolerance(case):
    kind, prec = case["kind"], case.get("prec")
    if kind == "prepost":
        # one rounding of the result in its own type; the way back adds another
        return {"rel": 2e-7 if case["dtype"] == "f32" else 1e-14}
    if kind == "eig":
        # vectors of the smallest kept values: rounding over their gaps
        # (7e-7 against numpy's at n = 1500)
        return {"rel": 4e-6, "max": 1e-3}
    if prec == "fp64":
        # 7e-11 against numpy's at 200x200x200x50: the last kept vectors turn
        # by rounding over their gap.  An FP32 output is rounded once.
        return {"rel": 2e-7 if kind == "rebuild" and case["dtype"] == "f32" else 1e-9}
    # single precision and its tensor-core splits: up to 2e-6 of a rebuilt tensor;
    # 3e-5 where an accuracy of 1e-2 lets the library take two digits
    return {"rel": 1.2e-4 if case.get("eps", 0.0) >= 1e-2 else 7e-6}


# --------------------------------------------------------------------- exact

def _axis(N, n):
    return N - 1 - n


def _unfold_gram(y, n):
    """Gram of the mode-n unfolding of y (reversed axes), FP64, in pieces."""
    a = _axis(y.dim(), n)
    L = _prod(y.shape[a + 1:])
    v = y.reshape(-1, y.shape[a], L)
    S = torch.zeros(v.shape[1], v.shape[1], dtype=torch.float64, device=y.device)
    if L == 1:
        u = v.reshape(-1, v.shape[1])
        for p in range(0, u.shape[0], 1 << 18):
            q = u[p:p + (1 << 18)].double()
            S += q.T @ q
        return S
    step = max(1, (1 << 27) // (v.shape[1] * L))
    for p in range(0, v.shape[0], step):
        q = v[p:p + step].double()
        S += torch.matmul(q, q.transpose(1, 2)).sum(0)
    return S


def _ttm(y, n, A):
    """y x_n A (A: K x I) in FP64."""
    a = _axis(y.dim(), n)
    sh = list(y.shape)
    v = y.reshape(-1, sh[a], _prod(sh[a + 1:])).double()
    sh[a] = A.shape[0]
    return torch.matmul(A, v).reshape(sh)


def _truncate(S, thr, rank=None):
    w, V = np.linalg.eigh(S.cpu().numpy())
    w, V = w[::-1].copy(), V[:, ::-1].copy()
    R, tail = len(w), 0.0
    while R > 1 and (tail + w[R - 1] <= thr if rank is None else R > rank):
        tail += w[R - 1]
        R -= 1
    return torch.from_numpy(w), torch.from_numpy(V[:, :R].copy()).cuda(), R


def _compress(x, dims, eps, order=None, hosvd=False):
    N = len(dims)
    y = x.reshape(tuple(reversed(dims)))
    flat = y.reshape(-1)
    norm = sum(float(torch.dot(p, p)) for p in (flat[k:k + (1 << 27)].double()
                                                for k in range(0, flat.numel(), 1 << 27)))
    thr = eps * eps * norm / N
    ws, Us, Rs = [None] * N, [None] * N, [None] * N
    src = y
    for n in (order or range(N)):
        ws[n], Us[n], Rs[n] = _truncate(_unfold_gram(src if hosvd else y, n), thr)
        y = _ttm(y, n, Us[n].T.contiguous())
    return ws, Us, Rs, y


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("eig", "batch") and _prod(_ints(case["dims"])) * 2.0 * max(
            _ints(case["dims"])) > 2e12:
        return None
    st = prepare(case, seed)
    if kind == "eig":
        w, U, R = _truncate(st["S"], 0.0, case["rank"])
        return {"eigvals": w, "vectors": U.abs()}
    if kind == "batch":
        ws, slices = [], []
        for x, d in zip(st["xs"], st["dims"]):
            w, Us, Rs, y = _compress(x, d, case["eps"])
            ws += w
            for n, U in enumerate(Us):
                y = _ttm(y, n, U[:1 if n >= 2 else d[n]].contiguous())
            slices.append(y.reshape(-1))
        return {"ranks": None, "eigvals": torch.cat(ws), "slices": torch.cat(slices)}
    dims = _ints(case["dims"])
    N = len(dims)
    if kind == "prepost":
        a = _axis(N, case["mode"])
        x = st["x"].reshape(tuple(reversed(dims))).double()
        rest = tuple(k for k in range(N) if k != a)
        if case["method"] == "standardize":
            shift = x.mean(rest, keepdim=True)
            scale = 1.0 / (x - shift).square().mean(rest, keepdim=True).sqrt()
        else:
            scale = 1.0 / x.abs().amax(rest, keepdim=True)
            shift = torch.zeros_like(scale)
        y = (x - shift) * scale
        return {"y": y.reshape(-1), "shift": shift.reshape(-1), "scale": scale.reshape(-1),
                "back": x.reshape(-1)}
    if kind == "rebuild":
        y = st["core"].double().reshape(tuple(reversed(_ints(case["core"]))))
        for n in range(N - 1, -1, -1):
            y = _ttm(y, n, st["mats"][n].contiguous())
        return y.reshape(-1)
    x = st["x"].cuda()
    if kind == "step":
        y = x.reshape(tuple(reversed(dims)))
        S = _unfold_gram(y, case["mode"])
        w, U, R = _truncate(S, 0.0, _ints(case["core"])[case["mode"]])
        return {"gram": S, "eigvals": w,
                "z": _ttm(y, case["mode"], U.T.contiguous()).abs().reshape(-1)}
    ws, Us, Rs, y = _compress(x, dims, case["eps"],
                              _ints(case["order"]) if "order" in case else None, kind == "hosvd")
    del x
    for n, p in enumerate(_ints(case["part"])):
        y = _ttm(y, n, Us[n][:p].contiguous())
    return {"ranks": Rs, "eigvals": ws, "part": y.reshape(-1)}
