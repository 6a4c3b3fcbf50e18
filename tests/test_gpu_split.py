"""The K split of the tensor-core products: batches whose smallest problem has fewer K chunks than the largest
needs ranges, and sizes no split of which fits shared memory."""
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


@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("sizes", [
    [(1, 14, 2), (2, 95, 5)],                          # one K chunk beside windows that need a split of two
    [(1, 53, 4), (4, 6, 8), (2, 19, 6)],               # two chunks, and the largest sorted before the smallest
    [(2, 72, 5), (4, 1, 1), (1, 355, 5), (2, 11, 5)],  # more than 128 (64) chunks in one range
])
def test_mixed_chunk_counts(ctx, prec, sizes):
    from paper_2012_11430_gb300 import default_opts
    ps = [W.make_problem(f"mc{i}", d, n, m, 7700 + i) for i, (d, n, m) in enumerate(sizes)]
    outs, rc = ctx.solve_batched([p.grid for p in ps], [p.d for p in ps], [p.n for p in ps], [p.m for p in ps],
                                 default_opts(precision=prec))
    assert rc == 0
    for o, p in zip(outs, ps):
        te, ce = W.match_to_truth(o.t, o.c, p.t, p.c)
        assert te <= 1e-6 and ce <= 1e-5, (p.d, p.n, te, ce)


@pytest.mark.parametrize("d,n,r,prec,fits", [(4, 7, 128, "tf32x3", True), (4, 8, 80, "tf32x3", True),
                                             (4, 8, 128, "tf32x3", False), (3, 96, 1, "bf16x3", False)])
def test_windows_that_do_not_fit_are_refused(ctx, monkeypatch, d, n, r, prec, fits):
    """Direct products: the largest sizes whose sample windows fit, and larger ones, which return PRONY_EINVAL."""
    import torch
    from paper_2012_11430_gb300 import PronyError
    from paper_2012_11430_gb300.binding import PRONY_EINVAL
    monkeypatch.setenv("PRONY_AXIS", "0")
    gen = torch.Generator(device="cuda").manual_seed(n)
    grid = torch.randn((2 * n + 2,) * d, dtype=torch.complex128, device="cuda", generator=gen)
    X = torch.randn(r, (n + 1) ** d, dtype=torch.complex64, device="cuda", generator=gen)
    L = n + 2
    Y = torch.empty(r, L ** d, dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    if not fits:
        with pytest.raises(PronyError) as e:
            ctx.toeplitz_mm_dev(grid.reshape(-1), d, n, X, L, 0, prec, Y)
        assert e.value.code == PRONY_EINVAL
        return
    ctx.toeplitz_mm_dev(grid.reshape(-1), d, n, X, L, 0, prec, Y)
    ax = tuple(range(-d, 0))
    F = torch.fft.fftn(torch.roll(grid, (-n,) * d, ax), dim=ax)
    Z = torch.fft.ifftn(F * torch.fft.fftn(X.to(torch.complex128).reshape((r,) + (n + 1,) * d), s=F.shape, dim=ax), dim=ax)
    Z = Z[(slice(None),) + (slice(L),) * d].reshape(r, -1)
    # the accumulator truncates once per MMA: 64 chunks of 24 MMAs at most, 2^-23 each of a partial sum
    assert (Y - Z).abs().square().sum().sqrt() <= 64 * 24 * 2.0 ** -23 * Z.abs().square().sum().sqrt()


def test_sample_counts_beyond_32_bits_are_refused(ctx):
    """d = 4, n = 107: (n + 1)^4 is within the limit on points, (2n + 2)^4 is not below 2^31.  Refused before anything is
    read or allocated."""
    import ctypes

    import torch
    from paper_2012_11430_gb300 import PronyError
    from paper_2012_11430_gb300.binding import PRONY_EINVAL
    x = torch.zeros((1, 8), dtype=torch.complex64, device="cuda")
    g = torch.zeros(8, dtype=torch.complex128, device="cuda")
    for prec in ("fp32", "bf16x3"):
        with pytest.raises(PronyError) as e:
            ctx.toeplitz_mm_dev(g, 4, 107, x, 108, 0, prec, x)
        assert e.value.code == PRONY_EINVAL
    z = np.zeros(16)
    ptr = z.ctypes.data_as(ctypes.c_void_p)
    assert ctx._lib.prony_solve(ctx._h, ptr, 4, 107, 1, None, ptr, ptr, None) == PRONY_EINVAL
