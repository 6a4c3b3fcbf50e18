"""Tensor-core products at the edges of their table formats and launch shapes: windows that fit as pairs and
ones that do not, two CTAs per SM for narrow blocks, and the short row passes of the Gram sums."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24
REL = {"bf16x3": lambda N: (2 * N + 32) * U32, "bf16x2": lambda N: (2 * N + 16) * U32 + 3 * 2.0 ** -16,
       "tf32x3": lambda N: (2 * N + 16) * U32 + 4 * 2.0 ** -22}


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_11430_gb300 import Context
    with Context(0) as c:
        yield c


@pytest.mark.parametrize("prec", ["bf16x3", "bf16x2", "tf32x3"])
@pytest.mark.parametrize("d,n,r,ext,adjoint", [
    (1, 16383, 7, 1, 0), (1, 20001, 24, 0, 1),         # one line, many row tiles
    (2, 126, 8, 1, 0), (2, 127, 24, 0, 1), (2, 127, 25, 1, 0), (2, 13, 3, 1, 0), (2, 14, 9, 0, 1),
    (3, 23, 16, 1, 0), (3, 24, 17, 0, 1), (3, 25, 1, 0, 0), (4, 10, 5, 1, 0), (4, 11, 24, 0, 1),
])
def test_products_by_format(ctx, monkeypatch, prec, d, n, r, ext, adjoint):
    """Direct products (no axis transform) against FP64 sums for the first rows, the last ones and some between."""
    import torch
    monkeypatch.setenv("PRONY_AXIS", "0")
    rng = np.random.Generator(np.random.PCG64(300 * d + n))
    L, N = n + (2 if ext else 1), (n + 1) ** d
    grid = rng.standard_normal((2 * n + 2,) * d) + 1j * rng.standard_normal((2 * n + 2,) * d)
    X = (rng.standard_normal((r, N)) + 1j * rng.standard_normal((r, N))).astype(np.complex64)
    Y = torch.full((r, L ** d), float("nan"), dtype=torch.complex64, device="cuda")
    ctx.toeplitz_mm_dev(torch.from_numpy(grid.reshape(-1)).cuda(), d, n, torch.from_numpy(X).cuda(), L, adjoint, prec, Y)
    Y = Y.cpu().numpy()
    assert np.all(np.isfinite(Y))
    Xd, M = X.astype(np.complex128), L ** d
    H = np.stack(np.unravel_index(np.arange(N), (n + 1,) * d), -1)
    for row in np.unique(np.r_[0:min(M, 3), rng.integers(0, M, 20), max(0, M - 3):M]):
        k = np.array(np.unravel_index(row, (L,) * d))
        x = (H - k if adjoint else k - H) + n
        a = grid[tuple(x.T)]
        a = np.conj(a) if adjoint else a
        ref, scale = Xd @ a, np.abs(Xd) @ np.abs(a)
        assert np.all(np.abs(Y[:, row] - ref) <= REL[prec](N) * scale), (row, float(np.max(np.abs(Y[:, row] - ref) / scale)))


@pytest.mark.parametrize("prec", ["bf16x3", "bf16x2", "tf32x3"])
@pytest.mark.parametrize("shapes", [
    [(1, 3, 1), (1, 15, 3), (1, 40, 6), (1, 127, 9)],
    [(2, 3, 1), (2, 6, 2), (2, 7, 3), (2, 10, 4), (2, 11, 5), (2, 22, 5), (2, 31, 8)],
    [(3, 3, 1), (3, 4, 1), (3, 6, 4), (1, 127, 4), (2, 32, 6), (4, 3, 1)],
])
def test_narrow_batches(ctx, prec, shapes):
    """Many narrow noise-free problems in one call: every copy of a problem gives the same bits, and its parameters."""
    from paper_2012_11430_gb300 import default_opts
    probs = [W.make_problem(f"nb{i}", d, n, m, 8100 + i) for i, (d, n, m) in enumerate(shapes)]
    count = 700
    idx = [i % len(probs) for i in range(count)]
    outs, rc = ctx.solve_batched([probs[i].grid for i in idx], [probs[i].d for i in idx], [probs[i].n for i in idx],
                                 [probs[i].m for i in idx], default_opts(precision=prec))
    assert rc == 0
    tol = 2e-4 if prec == "bf16x2" else 2e-6           # 3 * 2^-16 and FP32 rounding, times the conditioning
    for k, i in enumerate(idx):
        te, ce = W.match_to_truth(outs[k].t, outs[k].c, probs[i].t, probs[i].c)
        assert te <= tol and ce <= 20 * tol, (k, te, ce)
        assert np.array_equal(outs[k].t, outs[i].t) and np.array_equal(outs[k].c, outs[i].c)


@pytest.mark.parametrize("prec", ["bf16x3", "fp32"])
@pytest.mark.parametrize("d,n,r,ext", [(2, 47, 1, 1), (2, 63, 40, 0), (3, 15, 64, 1), (3, 19, 40, 0), (3, 15, 128, 1)])
def test_transformed_products(ctx, monkeypatch, prec, d, n, r, ext):
    """Products through the transform of the leading axis with few and with many lines, against FP64 FFTs: FP32 sums of
    N terms, statistically well below N u of the result's norm."""
    import torch
    monkeypatch.setenv("PRONY_AXIS", "1")
    rng = np.random.Generator(np.random.PCG64(600 + 10 * d + n))
    L, N = n + (2 if ext else 1), (n + 1) ** d
    grid = rng.standard_normal((2 * n + 2,) * d) + 1j * rng.standard_normal((2 * n + 2,) * d)
    X = (rng.standard_normal((r, N)) + 1j * rng.standard_normal((r, N))).astype(np.complex64)
    Y = torch.full((r, L ** d), float("nan"), dtype=torch.complex64, device="cuda")
    ctx.toeplitz_mm_dev(torch.from_numpy(grid.reshape(-1)).cuda(), d, n, torch.from_numpy(X).cuda(), L, 0, prec, Y)
    ax = tuple(range(1, d + 1))
    G = np.fft.fftn(np.roll(grid, (-n,) * d, axis=tuple(range(d))))
    ref = np.fft.ifftn(G * np.fft.fftn(X.reshape((r,) + (n + 1,) * d), s=G.shape, axes=ax), axes=ax)
    ref = ref[(slice(None),) + (slice(0, L),) * d].reshape(r, -1)
    assert np.linalg.norm(Y.cpu().numpy() - ref) <= 64 * U32 * np.sqrt(N) * np.linalg.norm(ref)
