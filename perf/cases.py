"""Performance cases: the work that programs give this library, through its public entry points.

A case is one call (or one short sequence of calls) with its sizes.  The kinds:
  solve      one problem through the host-pointer call: samples in a numpy array, (t, c) back
  batch      many problems of one size, samples resident on the GPU
  uneven     many problems of uneven n and m in one call, samples resident on the GPU
  product    the Toeplitz block product T X or T^* X alone, in each of the product arithmetics
  refine     Levenberg-Marquardt refinement of (t, c) on noisy samples
  gradient   loss and gradients of the exponential sum through autograd, for a torch optimiser
  eval       the fitted sum at arbitrary integer points, host arrays in and out
Solves and refinements carry the FP32 arithmetic of their products and sums, so the programs here keep
their estimates in single precision.  Node separations, noise levels and sizes are those of the
repository's workloads: nodes at least 2/n apart on the torus, |c| in [0.5, 1.5], additive circular noise.
"""
import math
import random

import numpy as np
import torch

from paper_2012_11430_gb300 import binding
from paper_2012_11430_gb300.refine import expsum, refine_lm

SEED = 2012114300                      # the library's default seed (of mu and V_0)
MU_STREAM = 0x4D55
_context = []


def _ctx():
    """One library context for the whole program, as its users keep it."""
    if not _context:
        _context.append(binding.Context(0))
    return _context[0]


# ----------------------------------------------------------------------------- cases
def listed():
    return [
        # a direction-finding or spectroscopy loop: one small clean problem at a time, latency only
        {"name": "solve-d2-n15-m5", "kind": "solve", "d": 2, "n": 15, "m": 5, "snr": 0.0, "precision": "bf16x3"},
        # one ordinary noisy problem, still a single call from host memory
        {"name": "solve-d2-n63-m20", "kind": "solve", "d": 2, "n": 63, "m": 20, "snr": 40.0, "precision": "bf16x3"},
        # throughput on the largest configuration: three dimensions, a batch resident on the GPU
        {"name": "batch64-d3-n19-m40", "kind": "batch", "count": 64, "d": 3, "n": 19, "m": 40, "snr": 50.0,
         "precision": "bf16x3"},
        # throughput on thousands of small problems of uneven size
        {"name": "uneven4096-d2", "kind": "uneven", "count": 4096, "d": 2, "n_lo": 7, "n_hi": 31, "m_hi": 12,
         "snr": 30.0, "precision": "bf16x3"},
        # the block product of one power iteration, with the rows of every shifted matrix (box of n + 2)
        {"name": "product-bf16x3-d3-n19-r40", "kind": "product", "d": 3, "n": 19, "r": 40, "ext": True,
         "adjoint": False, "precision": "bf16x3"},
        # the adjoint product at odd sizes in the TF32 split
        {"name": "product-tf32x3-d2-n50-r37", "kind": "product", "d": 2, "n": 50, "r": 37, "ext": False,
         "adjoint": True, "precision": "tf32x3"},
        # the FP32 product that the others are held against
        {"name": "product-fp32-d2-n63-r40", "kind": "product", "d": 2, "n": 63, "r": 40, "ext": False,
         "adjoint": False, "precision": "fp32"},
        # the FFT product
        {"name": "product-fft32-d2-n63-r40", "kind": "product", "d": 2, "n": 63, "r": 40, "ext": True,
         "adjoint": False, "precision": "fft32"},
        # estimate polished on strongly noisy samples
        {"name": "refine-d2-n63-m20", "kind": "refine", "d": 2, "n": 63, "m": 20, "snr": 20.0, "steps": 50},
        # one step of a gradient optimiser on the same problem
        {"name": "gradient-d2-n63-m20", "kind": "gradient", "d": 2, "n": 63, "m": 20, "snr": 20.0},
        # ... and on a three-dimensional sample box
        {"name": "gradient-d3-n19-m40", "kind": "gradient", "d": 3, "n": 19, "m": 40, "snr": 50.0},
        # the fitted model resampled at scattered points
        {"name": "eval-d3-m40-K65536", "kind": "eval", "d": 3, "m": 40, "K": 65536, "reach": 64},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _terms(rng, d, n, m_hi):
    """A number of terms that fits n: half of the cells of width 2/n at most, and the library's limits."""
    most = min(m_hi, max(1, (n // 2) ** d // 2), 6144 // (d * (n + 1)))
    return rng.randint(min(2, most), most)


def draw(rng):
    kind = rng.choice(["solve", "solve", "batch", "batch", "uneven", "product", "product", "product", "refine",
                       "gradient", "eval"])
    d = rng.choice([1, 2, 2, 2, 3, 3])
    n = _log_int(rng, {1: 16, 2: 7, 3: 5}[d], {1: 250, 2: 63, 3: 19}[d])
    if kind in ("solve", "batch"):
        m = _terms(rng, d, n, 40)
        fits = d == 1 or (d == 2 and n <= 63) or (d == 3 and n <= 7)
        case = {"kind": kind, "d": d, "n": n, "m": m, "snr": rng.choice([0.0, 30.0, 40.0, 50.0]),
                "precision": rng.choice(["bf16x3", "bf16x3", "bf16x3", "fp32"] + ["fft32"] * fits)}
        if kind == "batch":
            # products of a solve in 1e12 flops: at most a few hundred problems, below the largest listed case
            one = 5 * 8.0 * ((n + 1) ** d) ** 2 * 1.5 * m / 1e12 * (8 if case["precision"] == "fp32" else 1)
            case["count"] = _log_int(rng, 2, max(2, min(304, int(4.0 / (one + 0.004)))))
        return case
    if kind == "uneven":
        n_lo = rng.randint(7, 15)
        return {"kind": "uneven", "count": _log_int(rng, 16, 3000), "d": 2, "n_lo": n_lo, "n_hi": rng.randint(n_lo + 4, 31),
                "m_hi": rng.randint(4, 12), "snr": rng.choice([0.0, 30.0]), "precision": "bf16x3"}
    if kind == "product":
        precision = rng.choice(["bf16x3", "bf16x3", "bf16x2", "tf32x3", "fp32", "fft32"])
        if precision == "fft32" and d == 3:
            n = rng.randint(4, 7)
        ext = rng.random() < 0.5
        return {"kind": "product", "d": d, "n": n, "r": _log_int(rng, 1, min(40, (n + 1) ** d)), "ext": ext,
                "adjoint": not ext and rng.random() < 0.7, "precision": precision}
    if kind == "refine":
        d = rng.choice([1, 2, 2, 3])
        n = _log_int(rng, {1: 31, 2: 15, 3: 7}[d], {1: 250, 2: 63, 3: 15}[d])
        return {"kind": "refine", "d": d, "n": n, "m": _terms(rng, d, n, 20), "snr": rng.choice([20.0, 30.0]),
                "steps": rng.randint(10, 50)}
    if kind == "gradient":
        return {"kind": "gradient", "d": d, "n": n, "m": _terms(rng, d, n, 40), "snr": rng.choice([20.0, 50.0])}
    return {"kind": "eval", "d": d, "m": rng.randint(1, 40), "K": _log_int(rng, 1, 100000), "reach": _log_int(rng, 8, 512)}


# ----------------------------------------------------------------------------- synthetic problems
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed) * 7919 + 17)


def _nodes(gen, count, m, d, sep):
    """count x m nodes, every two of a problem at least `sep` apart (infinity norm on the torus): darts thrown
    until they fit; a problem that gets stuck takes cells of a jittered lattice."""
    dev = _device()
    t = torch.zeros(count, m, d, dtype=torch.float64, device=dev)
    stuck = torch.zeros(count, dtype=torch.bool, device=dev)
    for j in range(m):
        cand = torch.rand(count, 256, d, dtype=torch.float64, device=dev, generator=gen)
        if j:
            gap = (cand[:, :, None, :] - t[:, None, :j, :] + 0.5).remainder(1.0).sub_(0.5).abs_().amax(-1)
            fits = gap.amin(-1) >= sep
            stuck |= ~fits.any(1)
            cand = cand.gather(1, fits.int().argmax(1)[:, None, None].expand(-1, 1, d))
        t[:, j] = cand[:, 0]
    g = max(1, int(1.0 / sep + 1e-12))
    while g ** d < m:
        g += 1
    cell = torch.rand(count, g ** d, dtype=torch.float64, device=dev, generator=gen).argsort(1)[:, :m]
    place = torch.stack([cell // g ** l % g for l in range(d)], -1).double()
    half = max(0.0, (1.0 / g - sep) / 2)
    lattice = (place + 0.5) / g + half * (2 * torch.rand(count, m, d, dtype=torch.float64, device=dev, generator=gen) - 1)
    return torch.where(stuck[:, None, None], lattice.remainder(1.0), t)


def _coefficients(gen, *shape):
    u = torch.rand(*shape, 2, dtype=torch.float64, device=_device(), generator=gen)
    return torch.polar(0.5 + u[..., 0], 2 * math.pi * u[..., 1])


def _waves(t, x):
    """exp(-2 pi i t x): (..., len(x))"""
    ph = (t[..., None] * x).remainder(1.0)
    return torch.polar(torch.ones_like(ph), -2 * math.pi * ph)


def _samples(t, c, n):
    """(count, G, .., G) samples of the sums on {-n..n+1}^d."""
    count, m, d = t.shape
    x = torch.arange(-n, n + 2, dtype=torch.float64, device=t.device)
    left = c[:, :, None]
    for l in range(d - 1):
        left = (left[:, :, :, None] * _waves(t[:, :, l], x)[:, :, None, :]).flatten(2)
    return torch.matmul(left.transpose(1, 2), _waves(t[:, :, d - 1], x)).reshape((count,) + (2 * n + 2,) * d)


def _noise(gen, f, snr):
    if snr <= 0:
        return f
    power = f.abs().square().flatten(1).mean(1) / 10 ** (snr / 10)
    z = torch.randn(f.shape, dtype=torch.complex128, device=f.device, generator=gen)
    return f + power.sqrt().reshape((-1,) + (1,) * (f.dim() - 1)) * z


def _sizes(case):
    """n and m of every problem of a call: the layout of a case, the same for each seed."""
    if case["kind"] != "uneven":
        k = case.get("count", 1)
        return [case["n"]] * k, [case["m"]] * k
    r = random.Random(case["count"])
    ns = [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case["count"])]
    return ns, [r.randint(2, min(case["m_hi"], (n // 2) ** case["d"])) for n in ns]


def _problems(case, seed):
    """[(indexes, n, samples)]: the problems of a call, those of one n together."""
    gen = _generator(seed)
    ns, ms = _sizes(case)
    for n in sorted(set(ns)):
        at = [i for i, k in enumerate(ns) if k == n]
        m = torch.tensor([ms[i] for i in at], device=_device())
        most = int(m.max())
        t = _nodes(gen, len(at), most, case["d"], 2.0 / n)
        c = _coefficients(gen, len(at), most)
        c = torch.where(torch.arange(most, device=c.device)[None, :] < m[:, None], c, torch.zeros_like(c))
        yield at, n, _noise(gen, _samples(t, c, n), case["snr"])


def _fit_problem(case, seed):
    """Nodes and coefficients near the truth, and noisy complex64 samples on {-n..n+1}^d."""
    gen = _generator(seed)
    d, n, m = case["d"], case["n"], case["m"]
    t, c = _nodes(gen, 1, m, d, 2.0 / n), _coefficients(gen, 1, m)
    y = _noise(gen, _samples(t, c, n), case["snr"])[0].to(torch.complex64).reshape(-1)
    off = torch.randn(m, d, dtype=torch.float64, device=t.device, generator=gen)
    t0 = (t[0] + off * (0.01 / n)).remainder(1.0)
    c0 = c[0] * (1 + 0.02 * torch.randn(m, dtype=torch.complex128, device=t.device, generator=gen))
    return t0, c0, y


def _product_inputs(case, seed):
    """Samples of a sum with noise (so that T is not of low rank), and a block of Gaussian columns."""
    gen = _generator(seed)
    d, n, r = case["d"], case["n"], case["r"]
    m = max(1, min(20, (n // 2) ** d // 2))
    grid = _noise(gen, _samples(_nodes(gen, 1, m, d, 2.0 / n), _coefficients(gen, 1, m), n), 30.0)[0]
    X = torch.randn(r, (n + 1) ** d, dtype=torch.complex64, device=grid.device, generator=gen)
    return grid.contiguous(), X


def _eval_inputs(case, seed):
    r = np.random.default_rng(seed)
    t = r.random((case["m"], case["d"]))
    c = (0.5 + r.random(case["m"])) * np.exp(2j * np.pi * r.random(case["m"]))
    return t, c, r.integers(-case["reach"], case["reach"] + 1, (case["K"], case["d"])).astype(np.int32)


# ----------------------------------------------------------------------------- prepare and run
def _opts(case):
    o = binding.PronyOpts()
    binding.load().prony_default_opts(o)
    o.precision = binding.PRECISIONS[case["precision"]]
    return o


def prepare(case, seed):
    s = {"case": case, "ctx": _ctx()}
    kind, d = case["kind"], case["d"]
    if torch.cuda.is_available() and kind not in ("solve", "eval"):
        s["stream"] = torch.cuda.Stream()
    if kind == "solve":
        s["opts"] = _opts(case)
        s["grid"] = next(_problems(case, seed))[2][0].cpu().numpy()
    elif kind in ("batch", "uneven"):
        ns, ms = _sizes(case)
        sizes = [(2 * n + 2) ** d for n in ns]
        soff = np.concatenate([[0], np.cumsum(sizes)])
        ooff = np.concatenate([[0], np.cumsum(ms)])
        samples = torch.empty(int(soff[-1]), dtype=torch.complex128, device=_device())
        for at, n, f in _problems(case, seed):
            where = torch.as_tensor(soff[at], device=_device())[:, None] + torch.arange((2 * n + 2) ** d, device=_device())
            samples[where.flatten()] = f.flatten()
        s |= {"opts": _opts(case), "samples": samples, "ds": np.full(len(ns), d, np.int32), "ns": np.array(ns, np.int32),
              "ms": np.array(ms, np.int32), "soff": soff[:-1].astype(np.int64), "ooff": ooff[:-1].astype(np.int64),
              "t": torch.zeros(int(ooff[-1]) * d, dtype=torch.float64, device=_device()),
              "c": torch.zeros(int(ooff[-1]), dtype=torch.complex128, device=_device())}
    elif kind == "product":
        s["grid"], s["X"] = _product_inputs(case, seed)
        s["L"] = case["n"] + (2 if case["ext"] else 1)
        s["Y"] = torch.empty(case["r"], s["L"] ** d, dtype=torch.complex64, device=_device())
    elif kind in ("refine", "gradient"):
        t0, c0, y = _fit_problem(case, seed)
        s |= {"y": y, "lo": [-case["n"]] * d, "len": [2 * case["n"] + 2] * d}
        if kind == "refine":
            s |= {"t0": t0, "c0": c0}
        else:
            s |= {"t": t0.float().requires_grad_(True), "c": c0.to(torch.complex64).requires_grad_(True)}
    else:
        s["t"], s["c"], s["k"] = _eval_inputs(case, seed)
    return s


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "solve":
        r = ctx.solve(s["grid"], case["d"], case["n"], case["m"], s["opts"])
        return {"t": r.t.astype(np.float32), "c": r.c.astype(np.complex64)}
    if kind == "eval":
        return ctx.eval(s["t"], s["c"], s["k"])
    with torch.cuda.stream(s["stream"]):
        if kind in ("batch", "uneven"):
            ctx.solve_batched_dev(s["samples"], s["ds"], s["ns"], s["ms"], s["soff"], s["ooff"], s["t"], s["c"],
                                  s["opts"], s["stream"].cuda_stream)
            return {"t": s["t"].float(), "c": s["c"].to(torch.complex64)}
        if kind == "product":
            ctx.toeplitz_mm_dev(s["grid"], case["d"], case["n"], s["X"], s["L"], int(case["adjoint"]), case["precision"],
                                s["Y"], s["stream"].cuda_stream)
            return s["Y"]
        if kind == "refine":
            t, c, losses = refine_lm(s["t0"], s["c0"], s["y"], ctx, s["lo"], s["len"], steps=case["steps"])
            return {"t": t.float(), "c": c.to(torch.complex64), "losses": losses.float()}
        s["t"].grad = s["c"].grad = None
        e = expsum(s["t"].double(), s["c"], ctx, s["lo"], s["len"]) - s["y"]
        loss = (e.real.square() + e.imag.square()).sum()
        loss.backward()
        return {"loss": loss.detach(), "t": s["t"].grad, "c": s["c"].grad}


# ----------------------------------------------------------------------------- work
def work(case):
    """Bytes in and out, and the floating-point operations of the method as the library's documentation counts
    them: dense complex block products (8 per entry and column; five products of a solve) or FFT products, the
    Gram matrices of the fit, or one complex exponential and its uses per point and term."""
    kind, d = case["kind"], case["d"]
    if kind in ("solve", "batch", "uneven"):
        b = f = 0.0
        for n, m in zip(*_sizes(case)):
            N, Nx = (n + 1) ** d, (n + 2) ** d
            b += 16 * (2 * n + 2) ** d + m * (8 * d + 16)
            r0 = min(2 * m, N)
            f += 8.0 * N * (Nx * (r0 + 2 * m) + N * (r0 + m)) if case["precision"] != "fft32" else 0
            f += 8.0 * N * 6 * r0 * r0
        return {"bytes": b, "flops": f}
    if kind == "product":
        n, r = case["n"], case["r"]
        N, rows, grid = (n + 1) ** d, (n + (2 if case["ext"] else 1)) ** d, (2 * n + 2) ** d
        if case["precision"] == "fft32":
            flops = (2 * r + 1) * 5.0 * grid * math.log2(grid) + 6.0 * grid * r
        else:
            flops = 8.0 * N * rows * r
        return {"bytes": 16 * grid + 8 * r * (N + rows), "flops": flops}
    if kind == "eval":
        return {"bytes": case["K"] * (4 * d + 16) + case["m"] * (8 * d + 16), "flops": case["K"] * case["m"] * (8.0 + 2 * d)}
    K, m = (2 * case["n"] + 2) ** d, case["m"]
    if kind == "refine":
        step = K * m * (8.0 + 2 * d) * 2 + K * m * m * 2.0 * (d + 1) * (d + 2) + (m * (d + 2)) ** 3 / 3
        return {"bytes": 8 * K + m * (8 * d + 16) * 2, "flops": step * case["steps"]}
    return {"bytes": 8 * K + m * (8 * d + 16) * 2, "flops": K * m * (2 * (8.0 + 2 * d) + 8 + 4 * d)}


# ----------------------------------------------------------------------------- 64-bit values
def _mu(d):
    """The unit vector of the random combination C_mu = sum_l mu_l S_l: Philox4x64-10 draws of the default seed."""
    v = []
    for l in range(d):
        bits = np.random.Philox(key=[SEED, MU_STREAM], counter=(l - 1) % (1 << 256)).random_raw(2)
        u = [((int(b) >> 11) + 0.5) * 2.0 ** -53 for b in bits]
        v.append(math.sqrt(-math.log(u[0])) * complex(math.cos(2 * math.pi * u[1]), math.sin(2 * math.pi * u[1])))
    v = np.array(v)
    return v / np.linalg.norm(v)


class _Toeplitz:
    """T = [f(k - h)] of several problems of one n, by circulant embedding in 64 bits."""

    def __init__(self, f, n):
        self.n, self.d = n, f.dim() - 1
        self.axes = tuple(range(-self.d, 0))
        self.G = (2 * n + 2,) * self.d
        # point x of {-n..n+1}^d at index x mod G
        self.F = torch.fft.fftn(torch.roll(f, (-n,) * self.d, self.axes), dim=self.axes)[:, None]

    def times(self, X, adjoint=False, rows=None):
        """(count, r, N) -> (count, r, rows^d)"""
        rows = rows or self.n + 1
        X = X.reshape(X.shape[:2] + (self.n + 1,) * self.d)
        Z = torch.fft.fftn(X, s=self.G, dim=self.axes)
        Z = torch.fft.ifftn(Z * (self.F.conj() if adjoint else self.F), dim=self.axes)
        return Z[(slice(None), slice(None)) + (slice(rows),) * self.d]


def _orthonormal(X):
    """Rows of X (count, r, N) as an orthonormal basis of their span; null directions stay null."""
    for _ in range(2):
        w, Q = torch.linalg.eigh(torch.matmul(X.conj(), X.transpose(1, 2)))
        scale = torch.where(w > 1e-22 * w[:, -1:], w.clamp_min(1e-300).rsqrt(), torch.zeros_like(w))
        X = torch.matmul((Q * scale[:, None, :]).transpose(1, 2), X)
    return X


def _prony64(f, n, ms):
    """The multivariate matrix-pencil estimate in 64 bits for problems of one n: leading singular subspace by
    subspace iteration, S_l, the eigenbasis of C_mu, nodes, least-squares coefficients; sorted by node."""
    count, d, dev = f.shape[0], f.dim() - 1, f.device
    N, top = (n + 1) ** d, max(ms)
    r = min(N, 2 * top + 4)
    T = _Toeplitz(f, n)
    gen = torch.Generator(device=dev).manual_seed(1)
    V = _orthonormal(torch.randn(count, r, N, dtype=torch.complex128, device=dev, generator=gen))
    for _ in range(14):
        U = _orthonormal(T.times(V).flatten(2))
        V = _orthonormal(T.times(U, adjoint=True).flatten(2))
    Y = T.times(V, rows=n + 2)
    inner = (slice(None), slice(None)) + (slice(n + 1),) * d
    shifted = [Y[inner[:2] + tuple(slice(1, n + 2) if k == l else slice(n + 1) for k in range(d))].flatten(2) for l in range(d)]
    U = _orthonormal(Y[inner].flatten(2))
    A = torch.matmul(U.conj(), Y[inner].flatten(2).transpose(1, 2)).cpu().numpy()
    B = [torch.matmul(U.conj(), s.transpose(1, 2)).cpu().numpy() for s in shifted]
    mu = _mu(d)
    nodes = []
    for i, m in enumerate(ms):
        u, sg, vh = np.linalg.svd(A[i])
        S = [u[:, :m].conj().T @ B[l][i] @ vh[:m].conj().T / sg[:m] for l in range(d)]
        W = np.linalg.eig(sum(a * s for a, s in zip(mu, S)))[1]
        z = np.stack([np.diag(np.linalg.solve(W, s @ W)) for s in S], 1)
        nodes.append(np.mod(-np.angle(z) / (2 * np.pi), 1.0))
    t = torch.zeros(count, top, d, dtype=torch.float64, device=dev)
    keep = torch.zeros(count, top, dtype=torch.bool, device=dev)
    for i, v in enumerate(nodes):
        t[i, : ms[i]] = torch.as_tensor(v, device=dev)
        keep[i, : ms[i]] = True
    x = torch.arange(n + 1, dtype=torch.float64, device=dev)
    E = keep.to(torch.complex128)[:, :, None]
    gram = torch.ones(count, top, top, dtype=torch.complex128, device=dev)
    for l in range(d):
        w = _waves(t[:, :, l], x)
        E = (E[:, :, :, None] * w[:, :, None, :]).flatten(2)
        gram = gram * torch.matmul(w.conj(), w.transpose(1, 2))
    both = keep[:, :, None] & keep[:, None, :]
    gram = torch.where(both, gram, torch.eye(top, dtype=torch.complex128, device=dev))
    box = f[(slice(None),) + (slice(n, 2 * n + 1),) * d].flatten(1)
    c = torch.linalg.solve(gram, torch.matmul(E.conj(), box[:, :, None]))[:, :, 0].cpu().numpy()
    out = []
    for i, v in enumerate(nodes):
        order = np.lexsort(v.T[::-1])
        out.append((v[order], c[i, : ms[i]][order]))
    return out


def _exact_solve(case, seed):
    ns, ms = _sizes(case)
    found = [None] * len(ns)
    for at, n, f in _problems(case, seed):
        step = max(1, int(2e8 / ((2 * n + 2) ** case["d"] * (2 * max(ms) + 4) * 16)))
        for b in range(0, len(at), step):
            part = at[b: b + step]
            for i, r in zip(part, _prony64(f[b: b + step], n, [ms[i] for i in part])):
                found[i] = r
    t, c = np.concatenate([r[0] for r in found]), np.concatenate([r[1] for r in found])
    return {"t": t if case["kind"] == "solve" else t.reshape(-1), "c": c}


def _model64(t, c, case):
    """The points, weights and exponentials of a sample box, in 64 bits: e (m, K), k (K, d)."""
    x = torch.arange(-case["n"], case["n"] + 2, dtype=torch.float64, device=t.device)
    e = torch.ones(t.shape[0], 1, dtype=torch.complex128, device=t.device)
    for l in range(case["d"]):
        e = (e[:, :, None] * _waves(t[:, l], x)[:, None, :]).flatten(1)
    k = torch.cartesian_prod(*[x] * case["d"]).reshape(-1, case["d"])
    return e, k


def _exact_refine(case, seed):
    """The same damped Gauss-Newton iteration in 64 bits."""
    t, c, y = _fit_problem(case, seed)
    y, m, d, lam = y.to(torch.complex128), case["m"], case["d"], 1e-3

    def loss_of(t, c):
        e, k = _model64(t, c, case)
        r = c @ e - y
        return e, k, r, r.abs().square().sum()

    e, k, r, loss = loss_of(t, c)
    losses = [loss]
    for _ in range(case["steps"]):
        J = torch.cat([(-2j * math.pi) * c[:, None] * e * k[:, l] for l in range(d)] + [e, 1j * e])
        J = torch.cat([J.real, J.imag], 1)
        H, g = J @ J.T, J @ torch.cat([r.real, r.imag])
        step = torch.linalg.solve(H + lam * torch.diag(torch.diag(H)), -g).reshape(d + 2, m)
        t1, c1 = (t + step[:d].T).remainder(1.0), c + torch.complex(step[d], step[d + 1])
        trial = loss_of(t1, c1)
        if bool(trial[3] < loss):
            t, c, (e, k, r, loss), lam = t1, c1, trial, max(lam / 3, 1e-12)
        else:
            lam = min(lam * 4, 1e12)
        losses.append(loss)
    return {"t": t, "c": c, "losses": torch.stack(losses)}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch", "uneven"):
        return _exact_solve(case, seed)
    if kind == "product":
        grid, X = _product_inputs(case, seed)
        Y = _Toeplitz(grid[None], case["n"]).times(X[None].to(torch.complex128), case["adjoint"], case["n"] + (2 if case["ext"] else 1))
        return Y[0].flatten(1)
    if kind == "refine":
        return _exact_refine(case, seed)
    if kind == "gradient":
        t0, c0, y = _fit_problem(case, seed)
        t, c = t0.float().double(), c0.to(torch.complex64).to(torch.complex128)
        e, k = _model64(t, c, case)
        r = c @ e - y.to(torch.complex128)
        gc = 2 * (e.conj() @ r)
        gt = torch.stack([2 * (r.conj() * (-2j * math.pi) * c[:, None] * e * k[:, l]).sum(1).real for l in range(case["d"])], 1)
        return {"loss": r.abs().square().sum(), "t": gt, "c": gc}
    t, c, k = _eval_inputs(case, seed)
    out = np.zeros(case["K"], np.complex128)
    for j in range(case["m"]):
        ph = np.zeros(case["K"])
        for l in range(case["d"]):
            ph += np.mod(t[j, l] * k[:, l], 1.0)
        out += c[j] * np.exp(-2j * np.pi * ph)
    return out
