"""Performance cases of the framework: what users of compressed hierarchical matrices have it do.

Every case goes through the public Python entry points (``hm.HMatrix``, ``hm.HLU``,
``hm.hm_codec_decode``) on data made from a seed: jittered Fibonacci points on the unit
sphere (the Laplace problem), uniform points in the unit cube (the Matern covariance),
right-hand sides x ~ U(-1, 1).  Three kinds of work:

* ``matvec``: y := alpha M x + beta y (or with M^H) for nrhs columns;
* ``lu``: x := U^-1 L^-1 b with compressed H-LU factors of the Matern matrix;
* ``decode``: a packed array back to FP64.
"""
import math

import numpy as np
import torch

from paper_2405_03456_gb300 import hm

MATVEC = {"kind": "matvec", "kernel": "laplace", "fmt": "h", "adm": "std", "codec": "aflp", "eps": 1e-6, "leaf": 64,
          "nrhs": 1, "adjoint": False, "beta": 0.0, "graph": False}
KEYS = {1e-4: 14, 1e-6: 20, 1e-8: 27}   # bits for an accuracy eps: ceil(-log2 eps)


def listed():
    return [
        # the smallest call: an iterative solver on a small matrix, the same vectors every step (graph replay)
        dict(MATVEC, name="sphere_small", n=2048, leaf=32, graph=True),
        # the benchmark's product: N = 131072, eps = 1e-6, one vector
        dict(MATVEC, name="sphere_product", n=131072),
        # a coarse preconditioner-like product that adds into y, FPX, a size that fills no tile
        dict(MATVEC, name="sphere_coarse", n=60001, codec="fpx", eps=1e-4, beta=1.0),
        # an accurate product (float-float arithmetic)
        dict(MATVEC, name="sphere_fine", n=32768, eps=1e-8),
        # the shared-basis formats, one vector
        dict(MATVEC, name="uniform_product", n=16384, fmt="uh"),
        dict(MATVEC, name="nested_product", n=32768, fmt="h2"),
        # the adjoint of a matrix that is not symmetric, separate couplings
        dict(MATVEC, name="adjoint_product", n=10007, kernel="laplace_w", fmt="uh_sep", codec="fpx", adjoint=True),
        # small batches of a serving loop: a few right-hand sides on one resident matrix
        dict(MATVEC, name="sphere_batch", n=32768, nrhs=5),
        # a full panel on a covariance matrix (sampling, block solvers)
        dict(MATVEC, name="cube_panel", n=16384, kernel="matern", nrhs=32),
        # an accurate covariance batch, as a serving loop packs requests
        dict(MATVEC, name="cube_fine_batch", n=8192, kernel="matern", eps=1e-8, nrhs=20),
        # triangular solves with a few right-hand sides (a preconditioner's application)
        {"name": "lu_solve", "kind": "lu", "n": 2048, "leaf": 32, "codec": "aflp", "eps": 1e-6, "nrhs": 3},
        # a packed array back to FP64
        {"name": "decode_array", "kind": "decode", "n": 1 << 24, "codec": "aflp", "eps": 1e-6},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["matvec"] * 8 + ["lu", "decode"])
    codec = rng.choice(["aflp", "aflp", "fpx"])
    eps = rng.choice([1e-4, 1e-6, 1e-6, 1e-8])
    if kind == "decode":
        return {"kind": kind, "n": _log_int(rng, 1 << 10, 1 << 24), "codec": codec, "eps": eps}
    if kind == "lu":
        return {"kind": kind, "n": _log_int(rng, 500, 2000), "leaf": rng.choice([32, 48, 64]), "codec": codec,
                "eps": eps, "nrhs": rng.randint(1, 3)}
    kernel = rng.choice(["laplace", "laplace", "laplace_w", "matern"])
    fmt = "h" if kernel == "matern" else rng.choice(["h", "h", "h", "uh", "h2", "uh_sep"])
    adm = rng.choice(["std", "std", "std", "hodlr", "blr"]) if fmt == "h" and kernel != "matern" else "std"
    if rng.random() < 0.1:
        codec = "none"
    nrhs = rng.choice([1, 1, 1, rng.randint(2, 8), rng.randint(9, 32), rng.randint(33, 64)])
    hi = 16384 if kernel == "matern" or fmt != "h" or adm != "std" else 65536
    if nrhs > 1:
        hi = min(hi, 32768 if eps > 1e-7 and codec != "none" else 8192)
    return dict(MATVEC, n=_log_int(rng, 1000, hi), kernel=kernel, fmt=fmt, adm=adm, codec=codec, eps=eps, nrhs=nrhs,
                leaf=rng.choice([32, 64, 64, 128]), adjoint=rng.random() < 0.2, beta=rng.choice([0.0, 0.0, 1.0]),
                graph=rng.random() < 0.3)


# ---------------------------------------------------------------- inputs
def _points(case, rng):
    n = case["n"]
    if case.get("kernel", "matern") == "matern":
        return rng.uniform(0.0, 1.0, (n, 3))
    i = np.arange(n)
    h = math.sqrt(4.0 * math.pi / n)
    z = np.clip(1.0 - (2.0 * i + 1.0) / n + rng.uniform(-0.5, 0.5, n) / n, -1.0, 1.0)
    phi = i * math.pi * (3.0 - math.sqrt(5.0)) + rng.uniform(-0.5, 0.5, n) * h
    r = np.sqrt(1.0 - z * z)
    return np.stack([r * np.cos(phi), r * np.sin(phi), z], axis=1)


def _columns(rng, n, nrhs):
    """(n,) or (n, nrhs) column-major FP64 on the GPU."""
    v = torch.from_numpy(rng.uniform(-1.0, 1.0, (nrhs, n))).to("cuda")
    return v[0] if nrhs == 1 else v.t()


def _vectors(case, rng):
    return (_columns(rng, case["n"], case["nrhs"]), _columns(rng, case["n"], case["nrhs"]))


def _packed(case, rng):
    """A packed array of n values and its header: normal values, as a dense block's entries spread."""
    part = min(case["n"], 1 << 20)
    v = rng.standard_normal(part)
    packed, hdr = hm.hm_codec_encode(v, case["codec"], KEYS[case["eps"]])
    times = -(-case["n"] // part)
    return np.tile(packed, times)[: case["n"] * hdr["B"]], hdr


def _matrix(case, pts):
    M = hm.HMatrix(pts, case["kernel"], case["leaf"], 2.0, case["fmt"], case["eps"], adm=case["adm"])
    M.compress(case["eps"], case["codec"], True)
    return M.graph(True) if case["graph"] else M


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "decode":
        packed, hdr = _packed(case, rng)
        return {"case": case, "packed": torch.from_numpy(packed).to("cuda"), "hdr": hdr,
                "out": torch.empty(case["n"], dtype=torch.float64, device="cuda")}
    pts = _points(case, rng)
    x, y0 = _vectors(case, rng)
    state = {"case": case, "x": x, "y0": y0, "y": torch.empty_like(y0)}
    if case["kind"] == "lu":
        state["F"] = hm.HLU(pts, "matern", case["leaf"], 2.0, case["eps"]).compress(case["eps"], case["codec"], True)
        return state
    state["M"] = _matrix(case, pts)
    if case["adjoint"]:   # the transposed matrix is laid out on first use, as a server does up front
        z = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
        state["M"].matvec(1.0, z, 0.0, torch.empty_like(z), adjoint=True)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "decode":
        hm.hm_codec_decode(state["packed"].data_ptr(), case["n"], state["hdr"], state["out"].data_ptr(),
                           torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if case["kind"] == "lu":
        return state["F"].solve(state["x"], state["y"])
    if case["beta"] != 0.0:
        state["y"].copy_(state["y0"])
    return state["M"].matvec(0.75, state["x"], case["beta"], state["y"], adjoint=case["adjoint"])


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    n, rng = case["n"], np.random.default_rng(0)
    if case["kind"] == "decode":
        hdr = _packed(dict(case, n=min(n, 1 << 12)), rng)[1]
        return {"bytes": (hdr["B"] + 8) * n, "flops": 2 * n}
    r = case["nrhs"]
    if case["kind"] == "lu":   # both factors' codes, b read and x written; a multiply-add per stored entry and column
        F = hm.HLU(_points(case, rng), "matern", case["leaf"], 2.0, case["eps"])
        i = F.compress(case["eps"], case["codec"], True).info()
        return {"bytes": i["bytes_values"] + 16 * n * r, "flops": 2 * r * (i["bytes_fp64"] // 8)}
    i = _matrix(case, _points(case, rng)).info()
    return {"bytes": i["bytes_values"] + (16 if case["beta"] == 0.0 else 24) * n * r,
            "flops": 2 * r * (i["bytes_fp64"] // 8)}


# ---------------------------------------------------------------- the same in 64 bits
def _rows(case, P, i0, i1):
    """Rows i0 .. i1 - 1 of the kernel matrix of the points P (FP64)."""
    d2 = torch.zeros(i1 - i0, P.shape[0], dtype=torch.float64, device=P.device)
    for c in range(3):
        d2 += (P[i0:i1, c, None] - P[None, :, c]) ** 2
    if case.get("kernel", "matern") == "matern":
        s = d2.sqrt_().mul_(math.sqrt(3.0) / 0.1)
        return (1.0 + s) * torch.exp(-s)
    d2[torch.arange(i1 - i0), torch.arange(i0, i1)] = 4.0 * math.pi / P.shape[0]   # h^2
    K = d2.rsqrt_().mul_(1.0 / (4.0 * math.pi))
    return K * (1.0 + 0.5 * P[i0:i1, :1]) if case["kernel"] == "laplace_w" else K


def exact(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "decode":
        return _exact_decode(case, rng)
    n = case["n"]
    P = torch.from_numpy(_points(case, rng)).to("cuda")
    x, y0 = _vectors(case, rng)
    if case["kind"] == "lu":
        return torch.linalg.solve(_rows(case, P, 0, n), x)
    y = case["beta"] * y0
    step = max(1, (1 << 27) // n)
    for i in range(0, n, step):
        K = _rows(case, P, i, min(n, i + step))
        if case["adjoint"]:
            y += 0.75 * (K.t() @ x[i:i + step])
        else:
            y[i:i + step] += 0.75 * (K @ x)
    return y


def _exact_decode(case, rng):
    packed, h = _packed(case, rng)
    B, code = h["B"], np.zeros(case["n"], dtype=np.uint64)
    for b in range(B):
        code |= packed[b::B].astype(np.uint64) << np.uint64(8 * b)
    if h["fmt"] == 0:      # FPX e8: the top of an FP32 pattern
        v = (code.astype(np.uint32) << np.uint32(32 - 8 * B)).view(np.float32).astype(np.float64)
    elif h["fmt"] != 2:    # FPX e11, raw: the top of an FP64 pattern
        v = (code << np.uint64(64 - 8 * B)).view(np.float64)
    else:                  # AFLP: sign | f (e bits) | mantissa (m bits), value +-(2^f (1 + mantissa) - 1) vmin
        f = ((code >> np.uint64(h["m"])) & np.uint64((1 << h["e"]) - 1)).astype(np.int64)
        mant = (code & np.uint64((1 << h["m"]) - 1)).astype(np.float64) * 2.0 ** -h["m"]
        v = np.where(f > 0, (np.ldexp(1.0 + mant, f) - 1.0) * h["vmin"], 0.0)
        v = np.where((code >> np.uint64(8 * B - 1)) & np.uint64(1), -v, v)
    return torch.from_numpy(v)
