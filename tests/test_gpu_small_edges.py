"""The clustered small steps at the edges of their sizes: block widths at which the number of CTAs, threads
and column groups change, U wider than V, and batches large enough for the narrower clusters."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_11430_gb300 import Context
    with Context(0) as c:
        yield c


@pytest.mark.parametrize("d,m,a", [(1, 1, 1), (2, 2, 5), (1, 8, 8), (3, 9, 16), (2, 16, 128), (2, 17, 17), (4, 32, 33),
                                   (2, 33, 64), (3, 63, 65), (4, 64, 128)])
def test_small_steps_sizes(ctx, d, m, a):
    """Q = U_0 diag(sigma) V_0^* and M_l = Q V_0 S_l V_0^* with S_l = W diag(z(l)) W^{-1}: sigma to FP64 rounding,
    z and t to the second order of the FP32 eigenvectors (1e-11; kappa(W) is below 20 here)."""
    rng = np.random.Generator(np.random.PCG64(500 + 10 * m + d))
    gauss = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    U0 = np.linalg.qr(gauss(a, m))[0]
    V0 = np.linalg.qr(gauss(m, m))[0]
    sigma = np.sort(1.0 + 4.0 * rng.random(m))[::-1]
    Wm = np.linalg.qr(gauss(m, m))[0] + 0.3 * gauss(m, m) / np.sqrt(m)
    t = np.stack([(rng.permutation(m) + 0.5 + 0.2 * rng.uniform(-1, 1, m)) / m for _ in range(d)], 1)
    S = [Wm @ np.diag(np.exp(-2j * np.pi * t[:, l])) @ np.linalg.inv(Wm) for l in range(d)]
    Q = U0 @ np.diag(sigma) @ V0.conj().T
    # U^* T_l V = U_0 (S_l Sigma) V_0^* for the singular pairs (U_0, V_0)
    M = np.array([U0 @ S[l] @ np.diag(sigma) @ V0.conj().T for l in range(d)])
    sig, Sg, z, tg, status = ctx.small_steps(Q, M)
    assert status == 0
    assert np.max(np.abs(sig - sigma) / sigma) <= 64 * 2.0 ** -53 * m
    o, og = np.lexsort(t.T[::-1]), np.lexsort(tg.T[::-1])
    assert np.max(np.abs(z[og] - np.exp(-2j * np.pi * t[o]))) <= 1e-11
    assert np.max(W.torus_dist(tg[og], t[o])) <= 2e-12
    for l in range(d):                                 # S_l up to the phases of the singular vectors
        assert np.max(np.abs(np.abs(Sg[l]) - np.abs(S[l]))) <= 1e-9


@pytest.mark.parametrize("count,n,m", [(60, 15, 36), (100, 15, 36), (310, 13, 34), (100, 11, 18), (310, 11, 18), (100, 9, 12)])
def test_batches_of_every_cluster_width(ctx, count, n, m):
    """Noise-free problems in batches for which a problem gets four, two or one CTAs."""
    probs = [W.make_problem(f"cw{i}", 2, n, m, 7000 + i) for i in range(5)]
    idx = [i % 5 for i in range(count)]
    outs, rc = ctx.solve_batched([probs[i].grid for i in idx], [2] * count, [n] * count, [m] * count)
    assert rc == 0
    for k, i in enumerate(idx):
        te, ce = W.match_to_truth(outs[k].t, outs[k].c, probs[i].t, probs[i].c)
        assert te <= 1e-6 and ce <= 1e-5, (k, te, ce)
        assert np.array_equal(outs[k].t, outs[i].t) and np.array_equal(outs[k].c, outs[i].c)


def _close_pairs(m, a, gap):
    """Q with pairs of singular values a relative `gap` apart, and M_l of known eigenvalues exp(-2 pi i t)."""
    rng = np.random.Generator(np.random.PCG64(900 + m))
    gauss = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    U0 = np.linalg.qr(gauss(a, m))[0]
    V0 = np.linalg.qr(gauss(m, m))[0]
    sigma = np.linspace(2.0, 1.0, m // 2).repeat(2)
    sigma[1::2] *= 1 - gap
    Wm = np.linalg.qr(gauss(m, m))[0] + 0.3 * gauss(m, m) / np.sqrt(m)
    t = np.stack([(rng.permutation(m) + 0.5 + 0.2 * rng.uniform(-1, 1, m)) / m for _ in range(2)], 1)
    S = [Wm @ np.diag(np.exp(-2j * np.pi * t[:, l])) @ np.linalg.inv(Wm) for l in range(2)]
    Q = U0 @ np.diag(sigma) @ V0.conj().T
    return Q, np.array([U0 @ S[l] @ np.diag(sigma) @ V0.conj().T for l in range(2)]), sigma, t


CLOSE = [(m, a, gap) for m, a in ((12, 24), (32, 64), (40, 80), (64, 128)) for gap in (1e-3, 1e-4)]


@pytest.mark.parametrize("m,a,gap", CLOSE)
def test_close_singular_values_repeat(ctx, m, a, gap):
    """Close singular values take three or more refinement steps, after an odd number of which V lies where
    S_1 is written: every run gives the same bits."""
    Q, M, _, _ = _close_pairs(m, a, gap)
    first = ctx.small_steps(Q, M)
    assert first[-1] == 0
    for _ in range(30):
        assert all(np.array_equal(x, y) for x, y in zip(first, ctx.small_steps(Q, M)))


@pytest.mark.parametrize("m,a,gap", CLOSE)
def test_close_singular_values_converge(ctx, m, a, gap):
    """... and are refined until they converge: sigma to FP64 rounding, z (which no basis of a pair changes) as in
    test_small_steps_sizes."""
    Q, M, sigma, t = _close_pairs(m, a, gap)
    sig, _, z, tg, status = ctx.small_steps(Q, M)
    assert status == 0
    sigma = np.sort(sigma)[::-1]
    assert np.max(np.abs(sig - sigma) / sigma) <= 64 * 2.0 ** -53 * m
    o, og = np.lexsort(t.T[::-1]), np.lexsort(tg.T[::-1])
    assert np.max(np.abs(z[og] - np.exp(-2j * np.pi * t[o]))) <= 1e-11


@pytest.mark.parametrize("n,m", [(15, 10), (23, 30), (31, 45), (31, 64)])
def test_pivoted_blocks_repeat(ctx, n, m):
    """The pivoted elimination of blocks of 1 to 4 column groups (r0 = 2 m): equal problems of a call and of
    repeated calls give the same bits."""
    p = W.make_problem(f"pv{m}", 2, n, m, 7100 + m, snr_db=40.0)
    runs = [ctx.solve_batched([p.grid] * 24, [2] * 24, [n] * 24, [m] * 24) for _ in range(3)]
    first = runs[0][0][0]
    te, ce = W.match_to_truth(first.t, first.c, p.t, p.c)
    assert te <= 1e-2 / n and ce <= 0.1              # (noise of 40 dB)
    for outs, rc in runs:
        assert rc == 0
        assert all(np.array_equal(o.t, first.t) and np.array_equal(o.c, first.c) for o in outs)


@pytest.mark.parametrize("count", [40, 80, 160])
@pytest.mark.parametrize("n,m", [(23, 50), (27, 58), (31, 64)])
def test_wide_problems_in_batches(ctx, count, n, m):
    """The widest blocks (r0 = 2 m up to 128) in batches for which a problem gets four, two or one CTAs: its columns of
    U_Q are then taken a few at a time."""
    probs = [W.make_problem(f"wd{i}", 2, n, m, 7300 + m + i) for i in range(3)]
    outs, rc = ctx.solve_batched([probs[i % 3].grid for i in range(count)], [2] * count, [n] * count, [m] * count)
    assert rc == 0
    for k in range(count):
        p = probs[k % 3]
        te, ce = W.match_to_truth(outs[k].t, outs[k].c, p.t, p.c)
        assert te <= 1e-6 and ce <= 1e-5, (k, te, ce)
        assert np.array_equal(outs[k].t, outs[k % 3].t) and np.array_equal(outs[k].c, outs[k % 3].c)


def test_one_wide_problem_among_many(ctx):
    """The block sizes of a call are those of its widest problem."""
    wide, narrow = W.make_problem("wm", 2, 31, 64, 7400), W.make_problem("wn", 2, 9, 3, 7401)
    ps = [narrow] * 199 + [wide]
    outs, rc = ctx.solve_batched([p.grid for p in ps], [p.d for p in ps], [p.n for p in ps], [p.m for p in ps])
    assert rc == 0
    for o, p in zip(outs, ps):
        te, ce = W.match_to_truth(o.t, o.c, p.t, p.c)
        assert te <= 1e-6 and ce <= 1e-5


@pytest.mark.parametrize("unit", [1e-30, 1e-12, 1e-11, 1e8, 1e30])
@pytest.mark.parametrize("m,a", [(5, 10), (20, 40), (40, 80)])
def test_small_steps_in_any_unit(ctx, m, a, unit):
    """Q and M_l in another unit: sigma in that unit, S_l and z unchanged, as accurate as in test_small_steps_sizes."""
    Q, M, sigma, t = _close_pairs(m + m % 2, a, 1e-2)
    sig, S, z, tg, status = ctx.small_steps(unit * Q, unit * M)
    assert status == 0
    sigma = np.sort(sigma)[::-1] * unit
    assert np.max(np.abs(sig - sigma) / sigma) <= 64 * 2.0 ** -53 * len(sigma)
    o, og = np.lexsort(t.T[::-1]), np.lexsort(tg.T[::-1])
    assert np.max(np.abs(z[og] - np.exp(-2j * np.pi * t[o]))) <= 1e-11


@pytest.mark.parametrize("prec", ["bf16x3", "fp32", "fft32"])
@pytest.mark.parametrize("n,m", [(15, 5), (31, 20)])
def test_solve_in_any_unit(ctx, prec, n, m):
    """A noise-free solve with samples of any size: the same nodes, coefficients in the samples' unit."""
    from paper_2012_11430_gb300 import default_opts
    p = W.make_problem(f"un{m}", 2, n, m, 7500 + m)
    for unit in (1e-12, 1e-11, 1.0, 1e8):
        r = ctx.solve(unit * p.grid, 2, n, m, default_opts(precision=prec))
        te, ce = W.match_to_truth(r.t, r.c / unit, p.t, p.c)
        assert r.info["status"] == 0 and te <= 1e-6 and ce <= 1e-5, (unit, te, ce)


@pytest.mark.parametrize("unit", [1e-20, 1e-12, 1e-8, 1e6, 1e12, 1e20])
@pytest.mark.parametrize("m,a", [(5, 10), (20, 40), (40, 80)])
def test_small_steps_eigenvalues_of_any_size(ctx, m, a, unit):
    """M_l in another unit than Q: z in the unit of M_l, t unchanged, as accurate as in test_small_steps_sizes."""
    Q, M, sigma, t = _close_pairs(m + m % 2, a, 1e-2)
    _, _, z, tg, status = ctx.small_steps(Q, unit * M)
    assert status == 0
    o, og = np.lexsort(t.T[::-1]), np.lexsort(tg.T[::-1])
    assert np.max(np.abs(z[og] / unit - np.exp(-2j * np.pi * t[o]))) <= 1e-11
    assert np.max(W.torus_dist(tg[og], t[o])) <= 2e-12


@pytest.mark.parametrize("m", [16, 40])
def test_defective_matrix_reports_enoconv(ctx, m):
    """C_mu a single Jordan block: no eigenvector basis, W singular to FP32, its inverse does not converge."""
    from paper_2012_11430_gb300 import PRONY_ENOCONV
    J = np.exp(-0.7j) * np.eye(m) + np.eye(m, k=1)
    sig, S, z, t, status = ctx.small_steps(np.eye(m), J[None])
    assert status == PRONY_ENOCONV
    assert np.all(np.isfinite(sig)) and np.all(np.isfinite(S))
