"""Toeplitz products with the leading axis diagonalised by a DFT (kernels_axis.cu), forced on at sizes
where the library would not choose them: even and odd n + 1, the smallest n, partial chunks and tiles,
every dimension and arithmetic, and the samples that a product does not read."""
import numpy as np
import pytest

import workloads as W
from oracle import prony_oracle as O

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24
# relative error per term of a dot product of `N` complex terms in each arithmetic (FP32 sums)
REL = {"fp32": lambda N: (2 * N + 16) * U32, "bf16x3": lambda N: (2 * N + 32) * U32,
       "bf16x2": lambda N: (2 * N + 16) * U32 + 3 * 2.0 ** -16, "tf32x3": lambda N: (2 * N + 16) * U32 + 4 * 2.0 ** -22}


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2012_11430_gb300 import Context
    with Context(0) as c:
        yield c


def _reference(grid, d, n, L, adjoint, X):
    """The product in FP64, and the sum that bounds its error: with F^ = DFT of f over the leading axis,
    |F^(w; x')| <= A(x') = sum_x0 |f(x_0, x')| and |X^(w; h')| <= B(h') = sum_h0 |X|, so an arithmetic of relative
    error rel per sub-product and transform is within rel * sum_h' A(k' - h') B(h') of the exact value."""
    g = grid
    if adjoint:                                        # T^* = [conj f(h - k)]: mirror, zero outside the grid
        g = np.zeros_like(grid)
        g[(slice(0, 2 * n + 1),) * d] = np.conj(grid[(slice(0, 2 * n + 1),) * d][(slice(None, None, -1),) * d])
    if L == n + 1:                                     # differences of I_n only
        g = g.copy()
        g[2 * n + 1] = 0
    K, H = O.box_set([L] * d, d), O.index_set(n, d)
    ref = O.sample(g, n, K[:, None, :] - H[None, :, :]) @ X.T
    A = np.abs(g).sum(axis=0)
    B = np.abs(X).reshape(X.shape[0], n + 1, -1).sum(axis=1)
    Ks, Hs = O.box_set([L] * (d - 1), d - 1), O.index_set(n, d - 1)
    bound = A[tuple(np.moveaxis(Ks[:, None, :] - Hs[None, :, :] + n, -1, 0))] @ B.T
    return ref, np.tile(bound, (L, 1))


@pytest.mark.parametrize("prec", ["bf16x3", "bf16x2", "tf32x3", "fp32"])
@pytest.mark.parametrize("d,n,r,ext,adjoint", [
    (2, 1, 1, 1, 0), (2, 2, 3, 0, 1), (2, 3, 4, 1, 0), (2, 30, 17, 1, 0), (2, 31, 24, 0, 1), (2, 32, 33, 0, 0),
    (2, 62, 40, 1, 0), (2, 63, 9, 0, 1), (3, 1, 5, 1, 0), (3, 4, 7, 0, 1), (3, 9, 40, 1, 0), (3, 12, 64, 0, 1),
    (4, 2, 6, 1, 0), (4, 3, 11, 0, 1),
])
def test_axis_product(ctx, monkeypatch, prec, d, n, r, ext, adjoint):
    import torch
    monkeypatch.setenv("PRONY_AXIS", "1")
    rng = np.random.Generator(np.random.PCG64(9000 + 100 * d + n))
    L, N = n + (2 if ext else 1), (n + 1) ** d
    grid = rng.standard_normal((2 * n + 2,) * d) + 1j * rng.standard_normal((2 * n + 2,) * d)
    if not ext and not adjoint:
        grid[2 * n + 1] = np.nan                       # x_0 = n + 1: not read by a product over I_n
    X = (rng.standard_normal((r, N)) + 1j * rng.standard_normal((r, N))).astype(np.complex64)
    Y = torch.full((r, L ** d), float("nan"), dtype=torch.complex64, device="cuda")
    ctx.toeplitz_mm_dev(torch.from_numpy(grid.reshape(-1)).cuda(), d, n, torch.from_numpy(X).cuda(), L, adjoint, prec, Y)
    ref, scale = _reference(grid, d, n, L, adjoint, X.astype(np.complex128))
    rel = REL[prec]((n + 1) ** (d - 1)) + (4 * (n + 1) + 32) * U32
    err = np.abs(Y.cpu().numpy().T - ref)
    assert np.all(err <= rel * scale), float(np.max(err / (rel * scale)))


@pytest.mark.parametrize("prec", ["bf16x3", "fp32"])
@pytest.mark.parametrize("d,n", [(2, 95), (2, 96)])
def test_axis_largest_n(ctx, prec, d, n):
    """The largest n of the transformed products and the first beyond it, chosen by the library."""
    import torch
    rng = np.random.Generator(np.random.PCG64(77 + n))
    r, N, L = 3, (n + 1) ** d, n + 2
    grid = rng.standard_normal((2 * n + 2,) * d) + 1j * rng.standard_normal((2 * n + 2,) * d)
    X = (rng.standard_normal((r, N)) + 1j * rng.standard_normal((r, N))).astype(np.complex64)
    Y = torch.full((r, L ** d), float("nan"), dtype=torch.complex64, device="cuda")
    ctx.toeplitz_mm_dev(torch.from_numpy(grid.reshape(-1)).cuda(), d, n, torch.from_numpy(X).cuda(), L, 0, prec, Y)
    G = np.fft.fftn(np.roll(grid, (-n,) * d, axis=(0, 1)))
    ref = np.fft.ifftn(G * np.fft.fftn(X.reshape(r, n + 1, n + 1), s=G.shape, axes=(1, 2)), axes=(1, 2))[:, :L, :L].reshape(r, -1)
    # direct FP32 sums of N terms, statistically: well below N u32 of the result's norm
    assert np.linalg.norm(Y.cpu().numpy() - ref) <= 64 * U32 * np.sqrt(N) * np.linalg.norm(ref)


@pytest.mark.parametrize("prec", ["bf16x3", "fp32"])
def test_axis_solves_mixed_batch(ctx, monkeypatch, prec):
    """Problems of uneven d, n and m in one batch, with the transformed products and without: the same
    nodes and coefficients to the tolerances of noise-free solves, repeated solves bit-identical."""
    from paper_2012_11430_gb300 import default_opts
    probs = [W.make_problem(f"ax{i}", d, n, m, 900 + i) for i, (d, n, m) in
             enumerate([(2, 11, 5), (3, 5, 3), (2, 30, 9), (4, 3, 2), (2, 8, 4)])]
    args = ([p.grid for p in probs], [p.d for p in probs], [p.n for p in probs], [p.m for p in probs], default_opts(precision=prec))
    outs = {}
    for axis in ("0", "1", "1"):
        monkeypatch.setenv("PRONY_AXIS", axis)
        got, rc = ctx.solve_batched(*args)
        assert rc == 0
        if axis in outs and axis == "1":
            again, rc = ctx.solve_batched(*args)
            assert rc == 0 and all(np.array_equal(a.t, b.t) and np.array_equal(a.c, b.c) for a, b in zip(got, again))
        outs[axis] = got
    for p, a, b in zip(probs, outs["0"], outs["1"]):
        for r in (a, b):
            te, ce = W.match_to_truth(r.t, r.c, p.t, p.c)
            assert te <= 1e-6 and ce <= 1e-5, (p.name, te, ce)


@pytest.mark.parametrize("prec", ["bf16x3", "bf16x2", "tf32x3"])
@pytest.mark.parametrize("d,n,direct", [(3, 12, True), (4, 6, True), (3, 13, False), (4, 7, False), (2, 45, False)])
def test_small_products_of_three_dimensions_stay_direct(ctx, monkeypatch, prec, d, n, direct):
    """Below 2500 points with d > 2 the transforms round more than the direct sums: the default is the direct product
    there; where it is not, its error against FP64 is no larger (by more than the tenth two runs of one size differ)."""
    import torch
    rng = np.random.Generator(np.random.PCG64(300 + 10 * d + n))
    r, N, L = 12, (n + 1) ** d, n + 2
    grid = rng.standard_normal((2 * n + 2,) * d) + 1j * rng.standard_normal((2 * n + 2,) * d)
    X = (rng.standard_normal((r, N)) + 1j * rng.standard_normal((r, N))).astype(np.complex64)
    out = {}
    for axis in ("", "0"):
        if axis:
            monkeypatch.setenv("PRONY_AXIS", axis)
        Y = torch.full((r, L ** d), float("nan"), dtype=torch.complex64, device="cuda")
        ctx.toeplitz_mm_dev(torch.from_numpy(grid.reshape(-1)).cuda(), d, n, torch.from_numpy(X).cuda(), L, 0, prec, Y)
        out[axis] = Y.cpu().numpy()
    ax = tuple(range(-d, 0))
    G = np.fft.fftn(np.roll(grid, (-n,) * d, axis=ax), axes=ax)
    ref = np.fft.ifftn(G * np.fft.fftn(X.reshape((r,) + (n + 1,) * d), s=G.shape, axes=ax), axes=ax)
    ref = ref[(slice(None),) + (slice(L),) * d].reshape(r, -1)
    assert np.array_equal(out[""], out["0"]) == direct
    err = {k: np.linalg.norm(v - ref) for k, v in out.items()}
    assert err[""] <= 1.1 * err["0"]
