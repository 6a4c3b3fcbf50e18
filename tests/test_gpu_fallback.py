"""Products through the transform of the leading axis give way to the direct ones when their buffers cannot be
allocated (PRONY_ALLOC_MAX refuses the larger of the two)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_11430_gb300 import Context
    with Context(0) as c:
        yield c


def _solve(ctx, p, count, precision):
    from paper_2012_11430_gb300 import default_opts
    outs, rc = ctx.solve_batched([p.grid] * count, [p.d] * count, [p.n] * count, [p.m] * count, default_opts(precision=precision))
    assert rc == 0
    te, ce = W.match_to_truth(outs[0].t, outs[0].c, p.t, p.c)
    assert te <= 1e-6 and ce <= 1e-5
    return outs


def _same(a, b):
    return all(np.array_equal(x.t, y.t) and np.array_equal(x.c, y.c) for x, y in zip(a, b))


def test_direct_products_after_a_refused_transform(ctx, monkeypatch):
    """64 problems of n = 63, m = 5 take two CTAs per SM for the 8192 sub-products (a B' buffer of 252 MB) and one
    for the direct ones (126 MB): between the two the call gives what the direct products give."""
    monkeypatch.setenv("PRONY_TC_TUNE", "0")
    p = W.make_problem("fb", 2, 63, 5, 7200)
    monkeypatch.setenv("PRONY_ALLOC_MAX", str(160 << 20))
    got = _solve(ctx, p, 64, "bf16x3")
    monkeypatch.delenv("PRONY_ALLOC_MAX")
    monkeypatch.setenv("PRONY_AXIS", "0")
    assert _same(got, _solve(ctx, p, 64, "bf16x3"))
    monkeypatch.delenv("PRONY_AXIS")
    _solve(ctx, p, 64, "bf16x3")


def test_layout_known_before_a_refused_one(ctx, monkeypatch):
    """A layout whose sub-problem descriptors are on the device, a larger one whose descriptors replace them but whose
    blocks are refused (170 of 128 MB, the direct products' largest 87), then the first again."""
    small, large = W.make_problem("kl", 2, 63, 5, 7201), W.make_problem("kl", 2, 63, 20, 7202)
    first = _solve(ctx, small, 2, "fp32")
    monkeypatch.setenv("PRONY_ALLOC_MAX", str(128 << 20))
    got = _solve(ctx, large, 64, "fp32")
    assert _same(_solve(ctx, small, 2, "fp32"), first)
    monkeypatch.delenv("PRONY_ALLOC_MAX")
    assert _same(_solve(ctx, small, 2, "fp32"), first)
    monkeypatch.setenv("PRONY_AXIS", "0")
    assert _same(got, _solve(ctx, large, 64, "fp32"))


def test_refused_transform_keeps_no_memory(ctx, monkeypatch):
    """After a refused attempt a context holds what the direct products hold (PRONY_AXIS=0 from the start), and further
    calls of the layout change nothing."""
    import torch
    from paper_2012_11430_gb300 import Context
    monkeypatch.setenv("PRONY_TC_TUNE", "0")
    p = W.make_problem("km", 2, 63, 20, 7203)

    def held(context, **env):
        free = torch.cuda.mem_get_info()[0]
        for k, v in env.items():
            monkeypatch.setenv(k, v)
        used = []
        for _ in range(3):
            _solve(context, p, 64, "bf16x3")
            used.append(free - torch.cuda.mem_get_info()[0])
        for k in env:
            monkeypatch.delenv(k)
        return used

    _solve(ctx, p, 2, "bf16x3")                        # kernels and graph memory of the process
    with Context(0) as direct:
        a = held(direct, PRONY_AXIS="0")
    with Context(0) as refused:                        # B' tiles: 629 MB transformed, 315 MB direct
        b = held(refused, PRONY_ALLOC_MAX=str(512 << 20))
    assert b[0] == b[1] == b[2]
    assert abs(a[0] - b[0]) <= 32 << 20


def test_mixed_batch_memory(ctx, monkeypatch):
    """200 problems of d = 2 beside one of d = 3, whose sub-products have 13 K chunks instead of 2: the transformed
    products hold about twice the blocks of the direct ones (2 (n + 1) (n + 2)^(d - 1) rows for (n + 2)^d), whatever
    the widest sub-product of the batch."""
    import torch
    from paper_2012_11430_gb300 import Context, default_opts
    monkeypatch.setenv("PRONY_TC_TUNE", "0")
    p2, p3 = W.make_problem("mb2", 2, 63, 6, 7204), W.make_problem("mb3", 3, 19, 6, 7205)
    ps = [p2] * 200 + [p3]
    used = {}
    for axis in ("0", "1"):
        monkeypatch.setenv("PRONY_AXIS", axis)
        with Context(0) as c:
            free = torch.cuda.mem_get_info()[0]
            outs, rc = c.solve_batched([p.grid for p in ps], [p.d for p in ps], [p.n for p in ps], [p.m for p in ps],
                                       default_opts(precision="bf16x3"))
            used[axis] = free - torch.cuda.mem_get_info()[0]
        assert rc == 0
        for o, p in ((outs[0], p2), (outs[199], p2), (outs[200], p3)):
            te, ce = W.match_to_truth(o.t, o.c, p.t, p.c)
            assert te <= 1e-6 and ce <= 1e-5
    assert used["1"] <= 3 * used["0"]


def test_failed_launch_is_reported_every_time(ctx):
    """65536 problems are one more than a grid's second dimension holds: the call that captures the solve reports the
    failed launch, and so does a repeated one (no graph without those kernels is kept); other calls go on."""
    from paper_2012_11430_gb300 import PronyError, default_opts
    from paper_2012_11430_gb300.binding import PRONY_ECUDA
    P = 65536
    grid = np.ones(4, dtype=np.complex128)
    o = default_opts(precision="fp32")
    for _ in range(2):
        with pytest.raises(PronyError) as e:
            ctx.solve_batched([grid] * P, [1] * P, [1] * P, [1] * P, o)
        assert e.value.code == PRONY_ECUDA
    _solve(ctx, W.make_problem("fl", 2, 15, 5, 7206), 3, "fp32")


def test_failed_launch_before_the_autotuner(ctx):
    """... and where the first call of a batch shape runs step by step from the host (tensor-core products not tuned yet)."""
    from paper_2012_11430_gb300 import PronyError, default_opts
    from paper_2012_11430_gb300.binding import PRONY_ECUDA
    P = 65536
    grid = np.ones(4, dtype=np.complex128)
    for _ in range(2):
        with pytest.raises(PronyError) as e:
            ctx.solve_batched([grid] * P, [1] * P, [1] * P, [1] * P, default_opts(precision="bf16x3"))
        assert e.value.code == PRONY_ECUDA
    _solve(ctx, W.make_problem("fl", 2, 15, 5, 7207), 3, "bf16x3")
