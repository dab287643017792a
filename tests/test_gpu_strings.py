"""The kernels that run a string per warp or block, against the per-position
kernels (the persistent driver) and the oracle, over frontiers whose widths
cross every line between their parts: one arc, a warp, a warp's table, a
block's, shared dense positions, and back."""
import numpy as np
import pytest

import oracle
from paper_1701_03038_gb300 import synth

from gpu_util import assert_counts_close, assert_logz_close, assert_viterbi_equal, ensure_built

pytestmark = pytest.mark.gpu

Q = 6000
STEP, GATHER, SCATTER, DEAD, FAN = 0, 1, 2, 3, 4  # FAN + i: WIDTHS[i] arcs out of states 0..3
WIDTHS = [2, 31, 32, 33, 64, 65, 96, 97, 128, 129, 512, 1024, 1025, 2049, 4096, 5999]
RUNS = [1, 2, 3, 31, 32, 33, 34, 64, 65]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.fixture(scope="module")
def fans():
    rng = np.random.default_rng(5)
    q = np.arange(Q)
    parts = [(q, (q + 1) % Q, STEP), (q, q % 3, GATHER),
             (np.repeat(q, 3), rng.integers(0, Q, 3 * Q), SCATTER)]  # (several arcs into one state)
    for i, w in enumerate(WIDTHS):
        for s in range(4):
            # one arc a destination, and every fourth one a second arc from the same source
            d = rng.choice(Q, w, replace=False)
            d[3::4] = d[2:-1:4] if w > 3 else d[3::4]
            parts.append((np.full(w, s), d, FAN + i))
    src = np.concatenate([p[0] for p in parts]).astype(np.int32)
    dst = np.concatenate([p[1] for p in parts]).astype(np.int32)
    lab = np.concatenate([np.full(len(p[0]), p[2]) for p in parts]).astype(np.int32)
    perm = rng.permutation(len(src))
    w = rng.uniform(0.1, 4.0, len(src)).astype(np.float32)
    w[rng.random(len(src)) < 0.25] = 1.0  # equal values
    start = np.full(Q, np.inf, np.float32)
    start[:2] = [0.5, 0.25]
    final = rng.uniform(0.0, 2.0, Q).astype(np.float32)
    final[5::7] = np.inf
    fa = synth.FstArrays(Q, FAN + len(WIDTHS), Q, src[perm], dst[perm], lab[perm], dst[perm], w, start, final)
    from paper_1701_03038_gb300.fst import Fst
    return Fst.from_arrays(fa), oracle.Fst(fa)


def _strings(widths, count):
    """`count` strings: a fan, a run of one-arc steps, and so on."""
    rng = np.random.default_rng(widths)
    out = [[], [STEP], [DEAD], [STEP] * 40 + [DEAD], [STEP] * 33 + [DEAD] + [STEP] * 5]
    while len(out) < count:
        s = [STEP] * int(rng.choice(RUNS)) + [GATHER]
        for _ in range(int(rng.integers(1, 4))):
            s.append(FAN + int(rng.choice(widths)))
            if rng.random() < 0.3:
                s.append(SCATTER)
            s += [STEP] * int(rng.choice([0] + RUNS))
            if rng.random() < 0.8:
                s.append(GATHER)
                s += [STEP] * int(rng.choice([0] + RUNS))
                s.append(GATHER)
        out.append(s)
    off = np.concatenate([[0], np.cumsum([len(s) for s in out])]).astype(np.int64)
    return synth.Strings(np.concatenate([np.asarray(s, np.int32) for s in out]).astype(np.int32), off)


@pytest.mark.parametrize("count", [7, 60, 900])
@pytest.mark.parametrize("widths", [[0, 1, 2, 3], [4, 5, 6, 7, 8, 9], [10, 11, 12, 13], [14, 15], list(range(16))],
                         ids=["warp", "table", "block", "dense", "all"])
def test_string_kernels_match_per_position_kernels(fans, widths, count):
    import torch
    from paper_1701_03038_gb300 import _lib
    f, o = fans
    strs = _strings(widths, count)
    ids, off = torch.from_numpy(strs.ids).cuda(), torch.from_numpy(strs.offsets).cuda()
    w = torch.rand(strs.count, device="cuda")
    res = []
    for driver in (_lib.DRIVER_LAUNCH, _lib.DRIVER_PERSISTENT):
        # (compact accumulators could run full)
        p = f.plan(ids, off, flags=_lib.PLAN_DENSE_ACC if driver == _lib.DRIVER_PERSISTENT else 0)
        if driver == _lib.DRIVER_PERSISTENT:
            p.set_driver(driver)
        for _ in range(2):  # (the second run meets the first one's storage)
            p.viterbi()
            p.forward_backward(weights=w)
        torch.cuda.synchronize()
        res.append(p)
    a, b = res
    B, N = strs.count, len(strs.ids)
    for k, n in (("status", B), ("scores", B), ("paths", N), ("olabels", N), ("logz", B)):
        assert torch.equal(getattr(a, k)[:n], getattr(b, k)[:n]), k
    # sums of the same float32 posteriors in float64, in another order, then
    # rounded to float32: at most one rounding apart
    np.testing.assert_allclose(a.counts.cpu().numpy(), b.counts.cpu().numpy(), rtol=2.0**-23, atol=1e-12)
    sc, pa, st = a.scores.cpu().numpy(), a.paths.cpu().numpy(), a.status.cpu().numpy()
    for i in list(range(5)) + [strs.count - 1]:
        lo, hi = strs.offsets[i], strs.offsets[i + 1]
        assert_viterbi_equal(sc[i], pa[lo:hi], None, st[i], o.viterbi(strs.get(i)))


def _same_as_per_position(f, strs, runs):
    """The string kernels' outputs, run after run, against the persistent driver's."""
    import torch
    from paper_1701_03038_gb300 import _lib
    ids, off = torch.from_numpy(strs.ids).cuda(), torch.from_numpy(strs.offsets).cuda()
    B, N = strs.count, len(strs.ids)
    p = f.plan(ids, off, flags=_lib.PLAN_DENSE_ACC)
    p.set_driver(_lib.DRIVER_PERSISTENT)
    p.viterbi()
    p.forward_backward()
    torch.cuda.synchronize()
    q = f.plan(ids, off)
    for _ in range(runs):
        q.viterbi()
        q.forward_backward()
        torch.cuda.synchronize()
        for k, n in (("status", B), ("scores", B), ("paths", N), ("olabels", N), ("logz", B)):
            assert torch.equal(getattr(q, k)[:n], getattr(p, k)[:n]), k
        # the same float32 posteriors added up in float64 in another order: at
        # most one float32 rounding apart
        np.testing.assert_allclose(q.counts.cpu().numpy(), p.counts.cpu().numpy(), rtol=2.0**-23, atol=1e-12)


@pytest.mark.parametrize("count", [1, 40])
def test_table_and_dense_positions_in_turn(fans, count):
    # a heavy block's every change between its table and dense positions that
    # it works through alone, with no other barrier between them
    f, _ = fans
    turn = [FAN + 9, STEP, GATHER, FAN + 13, GATHER, FAN + 12, STEP, STEP, GATHER]
    out = [turn * (60 + b % 3) for b in range(count)]
    off = np.concatenate([[0], np.cumsum([len(s) for s in out])]).astype(np.int64)
    _same_as_per_position(f, synth.Strings(np.concatenate(out).astype(np.int32), off), 6)


@pytest.mark.parametrize("count", [1, 3])
def test_idle_blocks_look_for_jobs(fans, count):
    # few strings of many shared positions: hundreds of blocks without a
    # string find a job, or look for one that others have taken, at each
    f, _ = fans
    turn = [FAN + 15, SCATTER, STEP, GATHER, STEP, STEP]
    out = [turn * (50 + b) for b in range(count)]
    off = np.concatenate([[0], np.cumsum([len(s) for s in out])]).astype(np.int64)
    _same_as_per_position(f, synth.Strings(np.concatenate(out).astype(np.int32), off), 6)


@pytest.mark.parametrize("starts", [96, 97, 128, 129, 1000, 4095, 4096, 4097, 6000])
def test_many_start_states(starts):
    # the first position (and the last of the backward pass) over start states
    # on both sides of every line: a table's entries, a light warp's, a block's
    # by itself, shared out; few arcs, many, and none out of them
    from paper_1701_03038_gb300.fst import Fst
    rng = np.random.default_rng(starts)
    q = np.arange(Q)
    parts = [(q, (q + 1) % Q, 0), (q[::40], (q[::40] * 7) % Q, 1), (np.repeat(q, 3), rng.integers(0, Q, 3 * Q), 2),
             (q[::40], q[::40] % 3, 3)]
    src, dst = (np.concatenate([p[k] for p in parts]).astype(np.int32) for k in (0, 1))
    lab = np.concatenate([np.full(len(p[0]), p[2]) for p in parts]).astype(np.int32)
    w = rng.uniform(0.1, 4.0, len(src)).astype(np.float32)
    start = np.full(Q, np.inf, np.float32)
    start[rng.choice(Q, starts, replace=False)] = rng.uniform(0.0, 2.0, starts)
    fa = synth.FstArrays(Q, 5, 5, src, dst, lab, lab, w, start, rng.uniform(0.0, 2.0, Q).astype(np.float32))
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    out = [[], [0], [1], [2], [3], [4], [1, 0, 0], [2, 1, 0], [3, 0, 2, 2], [0, 2, 1], [4, 0], [2, 4, 1]]
    out += [list(rng.integers(0, 4, int(rng.integers(1, 9)))) for _ in range(40)]
    # (narrow positions after the wide ones: the string kernels take the batch)
    out = [s + [3] + [0] * (4 * len(s)) if s else s for s in out]
    off = np.concatenate([[0], np.cumsum([len(s) for s in out])]).astype(np.int64)
    strs = synth.Strings(np.concatenate([np.asarray(s, np.int32) for s in out]).astype(np.int32), off)
    _same_as_per_position(f, strs, 2)
    from paper_1701_03038_gb300 import _lib
    f.set_plain_method(_lib.PLAIN_FRONTIER)
    for s in out[:8]:
        x = np.asarray(s, np.int32)
        score, path, olab, st = f.viterbi(x)
        assert_viterbi_equal(score, path, olab, st, o.viterbi(x))
        ofb = o.forward_backward(x)
        lz, cnt, _ = f.forward_backward(x)
        assert_logz_close(lz, ofb["logz"])
        assert_counts_close(cnt, ofb["counts"])


def test_counts_of_one_string_are_repeatable(fans):
    # a string by itself adds its float64 counts in the order of its positions,
    # also where a run of one-arc positions uses an arc again and again
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300.fst import Fst
    rng = np.random.default_rng(6)
    q = np.arange(8)
    fan = rng.integers(0, 8, 64)
    src = np.concatenate([q, np.repeat(q, 8), q]).astype(np.int32)
    dst = np.concatenate([(q + 1) % 8, fan, np.zeros(8, int)]).astype(np.int32)
    lab = np.concatenate([np.zeros(8), np.ones(64), np.full(8, 2)]).astype(np.int32)
    start = np.full(8, np.inf, np.float32)
    start[0] = 0.0
    small = Fst.from_arrays(synth.FstArrays(8, 3, 3, src, dst, lab, lab, rng.uniform(0.1, 2.0, 80).astype(np.float32), start,
                                            np.zeros(8, np.float32)))
    runs = np.concatenate([[1] * 5 + [2] + [0] * int(rng.integers(40, 90)) for _ in range(12)]).astype(np.int32)
    f, _ = fans
    wide = _strings(list(range(16)), 12)
    for h, x in [(small, runs)] + [(f, wide.get(b)) for b in (8, 11)]:
        h.set_plain_method(_lib.PLAIN_FRONTIER)
        want = h.forward_backward(x)[1].view(np.uint32)
        for _ in range(8):
            assert np.array_equal(h.forward_backward(x)[1].view(np.uint32), want)
