"""prony_eval for few and many points (the direct kernel and the one with tables) against exact phases."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_11430_gb300 import Context
    with Context(0) as c:
        yield c


@pytest.mark.parametrize("d,m,K,reach", [(1, 1, 8191, 5), (1, 1, 8192, 5), (2, 64, 128, 1000000), (3, 40, 1001, 300),
                                         (4, 7, 20000, 64)])
def test_eval_many_points(ctx, d, m, K, reach):
    """Both sides of the size rule of prony_eval, phases on both sides of every table boundary: FP64
    sums of m terms, each within a few units in the last place of |c|."""
    rng = np.random.default_rng(m)
    t, c = rng.random((m, d)), (0.5 + rng.random(m)) * np.exp(2j * np.pi * rng.random(m))
    t[0] = 2.0 ** -15                                  # phases k / 2^15: exactly between two table points
    k = rng.integers(-reach, reach + 1, (K, d)).astype(np.int32)
    T = (np.floor(t * 2.0 ** 53).astype(np.uint64) << np.uint64(11))
    ph = (T[None] * k.astype(np.int64).astype(np.uint64)[:, None, :]).sum(-1, dtype=np.uint64)   # exact mod 2^64
    e = np.exp(-2j * np.pi * (ph.astype(np.int64).astype(np.float64) * 2.0 ** -64))
    assert np.max(np.abs(ctx.eval(t, c, k) - e @ c)) <= 8 * 2.0 ** -53 * (m + 8) * np.sum(np.abs(c)) / m ** 0.5


@pytest.mark.parametrize("d,m,K,reach", [(1, 1, 65535, 300), (1, 1, 65536, 300), (2, 11, 5957, 64), (2, 11, 5958, 64),
                                         (3, 12, 682, 64), (3, 12, 683, 64)])
def test_eval_sides_of_the_size_rule(ctx, d, m, K, reach):
    """Few terms take the tables from 65536 exponentials on, twelve from 8192: the bound of test_eval_many_points on
    both sides."""
    test_eval_many_points(ctx, d, m, K, reach)
