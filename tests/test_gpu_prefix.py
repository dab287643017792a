"""The parallel product over time against float64 matrix products: sizes round
the edges of its tiles, odd numbers of matrices, repeated pairs, and weights so far apart that
the scaled sums underflow and are taken again."""
import numpy as np
import pytest

from paper_1701_03038_gb300 import synth

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _lse(x, axis):
    m = x.max(axis=axis, keepdims=True)
    m = np.where(np.isneginf(m), 0.0, m)
    with np.errstate(divide="ignore"):
        return np.squeeze(m, axis) + np.log(np.exp(x - m).sum(axis=axis))


@pytest.mark.parametrize("spread", [1.0, 150.0])
@pytest.mark.parametrize("Q,n", [(1, 3), (3, 1), (31, 2), (32, 5), (33, 6), (63, 9), (64, 17), (65, 13), (97, 7), (130, 33),
                                 (5, 37), (9, 40), (33, 75), (64, 41)])  # (repeated pairs of symbols, even and odd)
def test_product_over_time(Q, n, spread):
    from paper_1701_03038_gb300.fst import Fst
    rng = np.random.default_rng(1000 * Q + n)
    V = 3
    # theta = -cost; a third of the arcs are missing, some states neither
    # start nor final, one state is reached by nothing
    M = -(rng.random((V, Q, Q)) * spread).astype(np.float32)
    M[rng.random((V, Q, Q)) < 1 / 3] = -np.inf
    M[:, np.arange(Q), (np.arange(Q) + 1) % Q] = -spread
    if Q > 2:
        M[:, :, 2] = -np.inf
        M[:, 1, 3 % Q] = 0.0
    start, final = np.zeros(Q, np.float32), (-rng.random(Q)).astype(np.float32)
    if Q > 2:
        start[1::2] = -np.inf
        final[2::3] = -np.inf
    s, i, j = np.nonzero(np.isfinite(M))
    perm = rng.permutation(len(s))
    s, i, j = (x[perm].astype(np.int32) for x in (s, i, j))
    fa = synth.FstArrays(Q, V, V, i, j, s, s, -M[s, i, j], -start, -final)
    f = Fst.from_arrays(fa)
    ids = rng.integers(0, V, n).astype(np.int32)
    lz, best, st = f.prefix_log_z(ids)
    a, v = start.astype(np.float64), start.astype(np.float64)
    for x in ids:
        m = M[x].astype(np.float64)
        a, v = _lse(a[:, None] + m, 0), (v[:, None] + m).max(axis=0)
    want, vbest = _lse(a + final, 0), (v + final).max()
    if np.isneginf(want):
        assert st != 0 and np.isneginf(lz) and np.isneginf(best)
        return
    # a level adds an error of four float32 roundings to values of the size of
    # the sum of its largest entries; each row's and column's scale cancels
    # only down to that size
    levels = int(np.ceil(np.log2(max(n, 2)))) + 1
    tol = 4 * levels * 2.0**-24 * (spread * n + 8.0)
    assert st == 0 and abs(lz - want) <= tol, (lz, want, tol)
    assert abs(best - vbest) <= tol, (best, vbest, tol)


@pytest.mark.parametrize("Q", [4, 16, 33, 70])
def test_scales_that_cancel(Q):
    # rows and columns whose largest entries do not meet: the scales add up to
    # 58, the entries of the product stay near 0 and are as accurate as there
    from paper_1701_03038_gb300.fst import Fst
    rng = np.random.default_rng(Q)
    i, j = (x.ravel().astype(np.int32) for x in np.meshgrid(np.arange(Q), np.arange(Q), indexing="ij"))
    start, final = np.full(Q, np.inf, np.float32), np.full(Q, np.inf, np.float32)
    start[0] = final[Q - 1] = 0.0
    for _ in range(12):
        M = rng.uniform(-1.0, 1.0, (2, Q, Q)).astype(np.float32)
        M[0, :, 0] += 29.0
        M[1, 0] = -200.0
        M[1, 1] += 29.0
        M[0, :, 1] = -200.0
        lab = np.repeat(np.arange(2), Q * Q).astype(np.int32)
        fa = synth.FstArrays(Q, 2, 2, np.tile(i, 2), np.tile(j, 2), lab, lab, -M.ravel(), start, final)
        lz, _, st = Fst.from_arrays(fa).prefix_log_z(np.array([0, 1], np.int32))
        x = M[0, 0].astype(np.float64) + M[1, :, Q - 1].astype(np.float64)
        want = np.log(np.exp(x - x.max()).sum()) + x.max()
        # roundings, of 2^-24: two exponentials (within 2 ulp), Q additions, a
        # logarithm and the sums of its parts, the result
        tol = 2.0**-24 * (8 + Q + 4 + 2 * abs(want))
        assert st == 0 and abs(lz - want) <= tol, (lz, want, lz - want, tol)
