"""Timed cases of the library: what its users have it do, through the ctypes binding.

The kinds of work, each over the sizes that the library's own configurations,
tests and benchmark name:

  jacobi   the Jacobi program, every nest on the GPU, transfers hoisted
           (oo_run_pattern_dev): a pattern measured by the search, or the
           solve that the search settled on; 33 x 33 x 65 x 50 is the small
           configuration, 257 x 257 x 513 x 200 the large one
  stencil  one sweep on the caller's own arrays (oo_stencil_dev)
  gemm     one matrix product on device buffers in a precision pattern
           (oo_gemm_f64_dev)
  fft      transforms of one length on device buffers (oo_fft_c128_dev)
  batch    uneven products and transforms as one captured graph (oo_batch_run)
  serve    mixed requests submitted to the serving loop and waited for
           (oo_submit / oo_wait, host buffers)

A context is made once and kept, as a program keeps it; inputs, plans and
output buffers are made by prepare().
"""
import math
import random

import numpy as np
import torch

from paper_2011_03602_gb300 import oo

PREC = {"fp64eq": oo.OO_PREC_FP64EQ, "split3_bf16": oo.OO_PREC_SPLIT3_BF16, "split3_tf32": oo.OO_PREC_SPLIT3_TF32}
COEFS = 12  # a0 a1 a2 a3 b0 b1 b2 c0 c1 c2 bnd wrk1


def listed():
    return [
        # the small configuration: a pattern the search measures, or one solve of a coarse grid
        {"name": "jacobi-33x33x65-50it", "kind": "jacobi", "I": 33, "J": 33, "K": 65, "iters": 50},
        # the large configuration: the solve the offload search is run for
        {"name": "jacobi-257x257x513-200it", "kind": "jacobi", "I": 257, "J": 257, "K": 513, "iters": 200},
        # the stencil nest alone on a caller's fields, a ragged grid between the two
        {"name": "stencil-150x131x270", "kind": "stencil", "I": 150, "J": 131, "K": 270},
        # a small product at FP64 accuracy, one call: latency counts
        {"name": "gemm-fp64eq-256", "kind": "gemm", "prec": "fp64eq", "m": 256, "n": 256, "k": 256},
        # an ordinary product with ragged sizes and an odd leading dimension
        {"name": "gemm-fp64eq-1000x777x1300", "kind": "gemm", "prec": "fp64eq", "m": 1000, "n": 777, "k": 1300},
        # the large product of the function-block configuration, at FP64 accuracy
        {"name": "gemm-fp64eq-4096", "kind": "gemm", "prec": "fp64eq", "m": 4096, "n": 4096, "k": 4096},
        # the same in the fast pattern
        {"name": "gemm-bf16-4096", "kind": "gemm", "prec": "split3_bf16", "m": 4096, "n": 4096, "k": 4096},
        # the smallest call: one short transform
        {"name": "fft-2e10", "kind": "fft", "log2n": 10, "batch": 1, "dir": -1},
        # many transforms of a middling length, backward
        {"name": "fft-2e14x64-inverse", "kind": "fft", "log2n": 14, "batch": 64, "dir": 1},
        # the longest transform of the function-block configuration
        {"name": "fft-2e22", "kind": "fft", "log2n": 22, "batch": 1, "dir": -1},
        # the batched configuration: uneven products and transforms, one graph
        {"name": "batch-4096gemm-2048fft", "kind": "batch", "gemms": 4096, "ffts": 2048},
        # the serving configuration's mix, a burst of requests that share the GPU
        {"name": "serve-32", "kind": "serve", "requests": 32},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(("jacobi", "jacobi", "stencil", "gemm", "gemm", "gemm", "fft", "fft", "batch", "serve"))
    if kind in ("jacobi", "stencil"):
        c = {"kind": kind, "I": _log_int(rng, 17, 257), "J": _log_int(rng, 17, 257), "K": _log_int(rng, 33, 513)}
        if kind == "jacobi":
            c["iters"] = _log_int(rng, 20, 200)
        return c
    if kind == "gemm":
        return {"kind": kind, "prec": rng.choice(("fp64eq", "fp64eq", "split3_bf16", "split3_tf32")),
                "m": _log_int(rng, 16, 4096), "n": _log_int(rng, 16, 4096), "k": _log_int(rng, 16, 4096)}
    if kind == "fft":
        log2n = rng.randint(8, 22)
        return {"kind": kind, "log2n": log2n, "batch": _log_int(rng, 1, 1 << (22 - log2n)), "dir": rng.choice((-1, 1))}
    if kind == "batch":
        gemms = _log_int(rng, 64, 4096)
        return {"kind": kind, "gemms": gemms, "ffts": gemms // 2}
    return {"kind": kind, "requests": _log_int(rng, 8, 32)}


# ------------------------------------------------------------------ contexts
_contexts = {}


def _context(what="calls"):
    """The program's context: one for direct calls, one that serves."""
    if what not in _contexts:
        stream = torch.cuda.Stream()
        ctx = oo.oo_create(0, stream)
        if what == "serve":
            oo.oo_serve_start(ctx, slots=8, hbm_budget_bytes=2 << 30, queue_cap=256)
        _contexts[what] = (ctx, stream)
    return _contexts[what][0]


# ----------------------------------------------------------- requests' sizes
def _batch_sizes(case):
    """Products with m, n, k log-uniform in [16, 512]; transforms of 2^8 .. 2^16.
    The sizes are the case's, the same for every seed."""
    rng = random.Random(1000 * case["gemms"] + case["ffts"])
    gemms = [tuple(_log_int(rng, 16, 512) for _ in range(3)) for _ in range(case["gemms"])]
    return gemms, [rng.randint(8, 16) for _ in range(case["ffts"])]


def _serve_sizes(case):
    """Half products (square, n log-uniform in [64, 2048]), three in ten transforms
    of 2^10 .. 2^20, one in five Jacobi solves of 100 iterations."""
    rng = random.Random(case["requests"])
    out = []
    for x in range(case["requests"]):
        r = x % 10
        if r in (0, 2, 4, 6, 8):
            out.append(("gemm", _log_int(rng, 64, 2048)))
        elif r in (1, 5, 7):
            out.append(("fft", rng.randint(10, 20)))
        else:
            out.append(("jacobi", rng.choice(((65, 65, 129), (129, 129, 257)))))
    return out


# -------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(gen, *shape):
    return torch.rand(*shape, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1


def _normal(gen, *shape):
    """Complex normal, E|z|^2 = 1."""
    return torch.view_as_complex(
        torch.randn(*shape, 2, generator=gen, device="cuda", dtype=torch.float64) * math.sqrt(0.5))


def _omega(seed, x=0):
    """The Jacobi program's own input: its relaxation factor (0.8 in its configurations)."""
    return float(np.float32(random.Random(int(seed) * 64 + x).uniform(0.7, 0.9)))


def _stencil_inputs(case, seed):
    """Twelve coefficient arrays near the program's values and a pressure field, in
    padded rows (the padding is not part of the grid)."""
    I, J, K = case["I"], case["J"], case["K"]
    pitch = oo.oo_jacobi_pitch(K)
    gen = _generator(seed)
    centre = (1, 1, 1, 1 / 6, 0, 0, 0, 1, 1, 1, 1, 0)
    coef = []
    for v in centre:
        noise = torch.rand(I, J, pitch, generator=gen, device="cuda", dtype=torch.float32)
        coef.append(v + 0.1 * (noise - 0.5))
    p = torch.rand(I, J, pitch, generator=gen, device="cuda", dtype=torch.float32)
    return pitch, coef, p


def _batch_inputs(case, seed):
    gemms, ffts = _batch_sizes(case)
    gen = _generator(seed)
    a = _uniform(gen, sum(m * k for m, _, k in gemms))
    b = _uniform(gen, sum(k * n for _, n, k in gemms))
    x = _normal(gen, sum(1 << e for e in ffts))
    return gemms, ffts, a, b, x


def _cut(gemms, ffts, a, b, c, x, y):
    """The requests' own pieces of the flat buffers."""
    ia = ib = ic = ix = 0
    for m, n, k in gemms:
        yield "gemm", (m, n, k), a[ia:ia + m * k], b[ib:ib + k * n], c[ic:ic + m * n]
        ia, ib, ic = ia + m * k, ib + k * n, ic + m * n
    for e in ffts:
        yield "fft", e, x[ix:ix + (1 << e)], None, y[ix:ix + (1 << e)]
        ix += 1 << e


def _serve_inputs(case, seed):
    gen = _generator(seed)
    for x, (kind, size) in enumerate(_serve_sizes(case)):
        if kind == "gemm":
            yield kind, size, _uniform(gen, size, size), _uniform(gen, size, size)
        elif kind == "fft":
            yield kind, size, _normal(gen, 1 << size), None
        else:
            yield kind, size, _omega(seed, x), None


# ------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "jacobi":
        I, J, K, iters = case["I"], case["J"], case["K"], case["iters"]
        s["prob"] = oo.jacobi(I, J, K, iters, omega=_omega(seed))
        s["p"] = torch.empty(I * J * K, dtype=torch.float32, device="cuda")
        s["res"] = torch.empty(iters, dtype=torch.float64, device="cuda")
    elif kind == "stencil":
        s["size"] = (case["I"], case["J"], case["K"])
        s["omega"] = _omega(seed)
        s["pitch"], s["coef"], s["p"] = _stencil_inputs(case, seed)
        s["wrk2"] = s["p"].clone()  # the sweep writes the interior only
        s["res"] = torch.empty(1, dtype=torch.float64, device="cuda")
    elif kind == "gemm":
        gen = _generator(seed)
        m, n, k = case["m"], case["n"], case["k"]
        s["size"], s["prec"] = (m, n, k), PREC[case["prec"]]
        s["A"], s["B"] = _uniform(gen, m, k), _uniform(gen, k, n)
        s["C"] = torch.empty(m, n, dtype=torch.float64, device="cuda")
    elif kind == "fft":
        n, batch = 1 << case["log2n"], case["batch"]
        s["size"], s["dir"] = (n, batch), case["dir"]
        s["x"] = _normal(_generator(seed), batch, n)
        s["X"] = torch.empty_like(s["x"])
    elif kind == "batch":
        gemms, ffts, a, b, x = _batch_inputs(case, seed)
        s["in"] = (a, b, x)
        s["C"] = torch.empty(sum(m * n for m, n, _ in gemms), dtype=torch.float64, device="cuda")
        s["X"] = torch.empty_like(x)
        reqs = []
        for what, size, u, v, w in _cut(gemms, ffts, a, b, s["C"], x, s["X"]):
            if what == "gemm":
                reqs.append({"kind": "gemm", "prec": oo.OO_PREC_FP64EQ, "m": size[0], "n": size[1], "k": size[2],
                             "A": u, "B": v, "C": w})
            else:
                reqs.append({"kind": "fft", "n": 1 << size, "x": u, "X": w, "dir": -1})
        s["batch"] = _Batch(_context(), reqs)
    else:
        s["reqs"], s["out"] = [], []
        for what, size, u, v in _serve_inputs(case, seed):
            if what == "gemm":
                c = np.empty((size, size))
                s["reqs"].append(oo.serve_request("gemm", A=u.cpu().numpy(), B=v.cpu().numpy(), C=c))
                s["out"].append(c)
            elif what == "fft":
                y = np.empty(1 << size, np.complex128)
                s["reqs"].append(oo.serve_request("fft", x=u.cpu().numpy(), X=y))
                s["out"].append(y)
            else:
                I, J, K = size
                p, res = np.empty(I * J * K, np.float32), np.empty(100)
                s["reqs"].append(oo.serve_request("jacobi", I=I, J=J, K=K, iters=100, omega=u, p=p, res=res))
                s["out"].append((p, res))
        _context("serve")
    s["ctx"] = _context("serve" if kind == "serve" else "calls")
    return s


class _Batch:
    """A batch plan, destroyed with the state that holds it."""

    def __init__(self, ctx, reqs):
        self.handle = oo.oo_batch_create(ctx, reqs)

    def __del__(self):
        torch.cuda.synchronize()
        oo.oo_batch_destroy(self.handle)


# ----------------------------------------------------------------------- run
def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "jacobi":
        oo.oo_run_pattern_dev(ctx, 0b111111, 1, s["prob"], s["p"], s["res"])
        return {"p": s["p"], "res": s["res"]}
    if kind == "stencil":
        I, J, K = s["size"]
        oo.oo_stencil_dev(ctx, I, J, K, s["pitch"], s["coef"], s["p"], s["omega"], s["wrk2"], s["res"])
        return {"wrk2": s["wrk2"], "res": s["res"]}
    if kind == "gemm":
        m, n, k = s["size"]
        oo.oo_gemm_f64_dev(ctx, m, n, k, s["A"], k, s["B"], n, s["C"], n, prec=s["prec"])
        return s["C"]
    if kind == "fft":
        n, batch = s["size"]
        oo.oo_fft_c128_dev(ctx, n, batch, s["dir"], s["x"], s["X"])
        return s["X"]
    if kind == "batch":
        oo.oo_batch_run(ctx, s["batch"].handle, 1)
        return {"C": s["C"], "X": s["X"]}
    tickets = [oo.oo_submit(ctx, r) for r in s["reqs"]]
    for t in tickets:
        oo.oo_wait(ctx, t)
    return s["out"]


# ---------------------------------------------------------------------- work
#: Operations of one grid point's update in plain arithmetic.
POINT_FLOPS = 44


def _jacobi_work(I, J, K, iters):
    """Per iteration each coefficient array and the field are read once and the new
    field is written once; the setup writes the fourteen arrays."""
    inner = (I - 2) * (J - 2) * (K - 2)
    return iters * inner * 4 * (COEFS + 2) + I * J * K * 4 * (COEFS + 2), iters * inner * POINT_FLOPS


def _gemm_work(m, n, k):
    return 8 * (m * k + k * n + m * n), 2 * m * n * k


def _fft_work(log2n, batch):
    return 32 * batch << log2n, 5 * log2n * batch << log2n


def work(case):
    kind = case["kind"]
    if kind == "jacobi":
        todo = [_jacobi_work(case["I"], case["J"], case["K"], case["iters"])]
    elif kind == "stencil":
        inner = (case["I"] - 2) * (case["J"] - 2) * (case["K"] - 2)
        todo = [(inner * 4 * (COEFS + 2), inner * POINT_FLOPS)]
    elif kind == "gemm":
        todo = [_gemm_work(case["m"], case["n"], case["k"])]
    elif kind == "fft":
        todo = [_fft_work(case["log2n"], case["batch"])]
    elif kind == "batch":
        gemms, ffts = _batch_sizes(case)
        todo = [_gemm_work(*g) for g in gemms] + [_fft_work(e, 1) for e in ffts]
    else:
        todo = []
        for what, size in _serve_sizes(case):
            todo.append(_gemm_work(size, size, size) if what == "gemm" else
                        _fft_work(size, 1) if what == "fft" else _jacobi_work(*size, 100))
    return {"bytes": sum(b for b, _ in todo), "flops": sum(f for _, f in todo)}


# --------------------------------------------------------------------- exact
def _sweep(c, p, omega):
    """The update of the interior in 64 bits: new values and the residual's terms."""
    def at(di, dj, dk):
        I, J, K = p.shape
        return p[1 + di:I - 1 + di, 1 + dj:J - 1 + dj, 1 + dk:K - 1 + dk]

    s0 = c[0] * at(1, 0, 0) + c[1] * at(0, 1, 0) + c[2] * at(0, 0, 1)
    s0 += c[4] * (at(1, 1, 0) - at(1, -1, 0) - at(-1, 1, 0) + at(-1, -1, 0))
    s0 += c[5] * (at(0, 1, 1) - at(0, 1, -1) - at(0, -1, 1) + at(0, -1, -1))
    s0 += c[6] * (at(1, 0, 1) - at(1, 0, -1) - at(-1, 0, 1) + at(-1, 0, -1))
    s0 += c[7] * at(-1, 0, 0) + c[8] * at(0, -1, 0) + c[9] * at(0, 0, -1) + c[11]
    ss = (s0 * c[3] - at(0, 0, 0)) * c[10]
    return at(0, 0, 0) + omega * ss, ss


def _exact_jacobi(I, J, K, iters, omega):
    # the program's coefficients: b0..b2 and wrk1 are zero, the others one but a3
    sixth = float(np.float32(1 / 6))
    k = torch.arange(K, device="cuda", dtype=torch.float64)
    p = (k * k / (K - 1) ** 2).float().double().expand(I, J, K).contiguous()
    q = p.clone()
    res = []
    for _ in range(iters):
        mid = p[1:-1, 1:-1, 1:-1]
        ss = (p[2:, 1:-1, 1:-1] + p[:-2, 1:-1, 1:-1] + p[1:-1, 2:, 1:-1] + p[1:-1, :-2, 1:-1] +
              p[1:-1, 1:-1, 2:] + p[1:-1, 1:-1, :-2]) * sixth - mid
        res.append(ss.square().sum())
        q[1:-1, 1:-1, 1:-1] = mid + omega * ss
        p, q = q, p
    return p.reshape(-1), torch.stack(res) if res else torch.empty(0, device="cuda", dtype=torch.float64)


def exact(case, seed):
    kind = case["kind"]
    if kind == "jacobi":
        p, res = _exact_jacobi(case["I"], case["J"], case["K"], case["iters"], _omega(seed))
        return {"p": p, "res": res}
    if kind == "stencil":
        K = case["K"]
        _, coef, p = _stencil_inputs(case, seed)
        new, ss = _sweep([c[1:-1, 1:-1, 1:K - 1].double() for c in coef], p[:, :, :K].double(), _omega(seed))
        out = p.double()
        out[1:-1, 1:-1, 1:K - 1] = new
        return {"wrk2": out, "res": ss.square().sum().reshape(1)}
    if kind == "gemm":
        gen = _generator(seed)
        A, B = _uniform(gen, case["m"], case["k"]), _uniform(gen, case["k"], case["n"])
        return A @ B
    if kind == "fft":
        x = _normal(_generator(seed), case["batch"], 1 << case["log2n"])
        return torch.fft.fft(x) if case["dir"] < 0 else torch.fft.ifft(x)
    if kind == "batch":
        gemms, ffts, a, b, x = _batch_inputs(case, seed)
        C = torch.empty(sum(m * n for m, n, _ in gemms), dtype=torch.float64, device="cuda")
        X = torch.empty_like(x)
        for what, size, u, v, w in _cut(gemms, ffts, a, b, C, x, X):
            if what == "gemm":
                m, n, k = size
                w.copy_((u.view(m, k) @ v.view(k, n)).reshape(-1))
            else:
                w.copy_(torch.fft.fft(u))
        return {"C": C, "X": X}
    out = []
    for what, size, u, v in _serve_inputs(case, seed):
        if what == "gemm":
            out.append((u @ v).cpu().numpy())
        elif what == "fft":
            out.append(torch.fft.fft(u).cpu().numpy())
        else:
            p, res = _exact_jacobi(*size, 100, u)
            out.append((p.cpu().numpy(), res.cpu().numpy()))
    return out
