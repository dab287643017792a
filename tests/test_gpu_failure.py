"""Failure paths of the batched method, made on the host (no GPU fault).

A run whose live pool overflows must report FST_ERR_OOM for every string of
its wave, write the no-result markers, and leave the plan usable: the next
run on the same plan clears what the overflowing one left behind and is
exact again.  The overflow is forced by capping the pool
(fst_plan_limit_pool), which allocates nothing and touches no memory out of
bounds.
"""
import math
import time

import numpy as np
import pytest

import oracle
from paper_1701_03038_gb300 import synth

from gpu_util import assert_counts_close, assert_logz_close, assert_viterbi_equal, ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def test_pool_overflow_reports_oom_then_recovers():
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300._lib import PLAN_NO_FB, PLAN_NO_VITERBI
    from paper_1701_03038_gb300.fst import Fst
    fa, strs = synth.make_config("c2", scale=0.02, strings=24)
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    ids = torch.from_numpy(strs.ids).cuda()
    off = torch.from_numpy(strs.offsets).cuda()
    pv = f.plan(ids, off, flags=PLAN_NO_FB)
    pf = f.plan(ids, off, flags=PLAN_NO_VITERBI | _lib.PLAN_DENSE_ACC)
    pf.set_pull(1)  # the forward pass's dense vectors must survive an overflowed run
    B, N = strs.count, len(strs.ids)
    ov = [o.viterbi(strs.get(b)) for b in range(B)]
    ofb = o.fb_batch(strs.ids, strs.offsets, nthreads=8)

    def check_exact():
        pv.viterbi()
        pf.forward_backward()
        torch.cuda.synchronize()
        sc, pa, ol, st = (pv.scores.cpu().numpy(), pv.paths.cpu().numpy(), pv.olabels.cpu().numpy(),
                          pv.status.cpu().numpy())
        for b in range(B):
            lo, hi = strs.offsets[b], strs.offsets[b + 1]
            assert_viterbi_equal(sc[b], pa[lo:hi], ol[lo:hi], st[b], ov[b])
            assert_logz_close(pf.logz[b].item(), ofb["logz"][b])
        assert (pf.status[:B].cpu().numpy() == 0).all()
        assert_counts_close(pf.counts.cpu().numpy(), ofb["counts"], batch=True)

    check_exact()
    # every string has at least one live state per position, so 8 entries
    # cannot hold the run's live states
    for limit in (8, 1):
        pv.limit_pool(limit)
        pf.limit_pool(limit)
        pv.viterbi()
        pf.forward_backward()
        torch.cuda.synchronize()
        assert (pv.status[:B].cpu().numpy() == _lib.OOM).all()
        assert (pf.status[:B].cpu().numpy() == _lib.OOM).all()
        assert np.isneginf(pv.scores[:B].cpu().numpy()).all()
        assert (pv.paths[:N].cpu().numpy() == -1).all()
        assert np.isneginf(pf.logz[:B].cpu().numpy()).all()
        assert (pf.counts.cpu().numpy() == 0).all()
        # the cap lifted, the same plans are exact again
        pv.limit_pool(0)
        pf.limit_pool(0)
        check_exact()


def test_table_overflow_reports_oom_then_recovers():
    # the compact accumulator tables capped at 8 slots cannot hold one
    # position's live states (24 strings, each with at least one): the run
    # reports FST_ERR_OOM everywhere, and with the cap lifted the same plans
    # are exact again (the overflowing run's leftovers are cleared)
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300._lib import PLAN_NO_FB, PLAN_NO_VITERBI
    from paper_1701_03038_gb300.fst import Fst
    fa, strs = synth.make_config("c2", scale=0.02, strings=24)
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    ids = torch.from_numpy(strs.ids).cuda()
    off = torch.from_numpy(strs.offsets).cuda()
    pv = f.plan(ids, off, flags=PLAN_NO_FB)
    pf = f.plan(ids, off, flags=PLAN_NO_VITERBI)
    B, N = strs.count, len(strs.ids)
    ofb = o.fb_batch(strs.ids, strs.offsets, nthreads=8)
    for rnd in range(2):
        pv.limit_table(8)
        pf.limit_table(8)
        pv.viterbi()
        pf.forward_backward()
        torch.cuda.synchronize()
        assert (pv.status[:B].cpu().numpy() == _lib.OOM).all()
        assert (pf.status[:B].cpu().numpy() == _lib.OOM).all()
        assert (pv.paths[:N].cpu().numpy() == -1).all()
        assert (pf.counts.cpu().numpy() == 0).all()
        pv.limit_table(0)
        pf.limit_table(0)
        pv.viterbi()
        pf.forward_backward()
        torch.cuda.synchronize()
        sc, pa, ol, st = (pv.scores.cpu().numpy(), pv.paths.cpu().numpy(), pv.olabels.cpu().numpy(),
                          pv.status.cpu().numpy())
        for b in range(B):
            lo, hi = strs.offsets[b], strs.offsets[b + 1]
            assert_viterbi_equal(sc[b], pa[lo:hi], ol[lo:hi], st[b], o.viterbi(strs.get(b)))
            assert_logz_close(pf.logz[b].item(), ofb["logz"][b])
        assert_counts_close(pf.counts.cpu().numpy(), ofb["counts"], batch=True)
    with pytest.raises(_lib.FstError):
        pv.limit_table(-1)


def test_pool_limit_rejects_negative():
    import torch
    from paper_1701_03038_gb300._lib import FstError
    from paper_1701_03038_gb300.fst import Fst
    fa, strs = synth.make_config("c1", scale=0.2, strings=2)
    f = Fst.from_arrays(fa)
    p = f.plan(torch.from_numpy(strs.ids).cuda(), torch.from_numpy(strs.offsets).cuda())
    with pytest.raises(FstError):
        p.limit_pool(-1)


def test_persistent_barrier_timeout_reports_and_recovers():
    # the persistent passes' grid barriers are told to wait for one block
    # that does not exist: every wait runs out after its limit (0.2 s here),
    # the run ends early with FST_ERR_TIMEOUT for every string, the GPU keeps
    # answering, and the next run on the same plans is exact
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300._lib import PLAN_NO_FB, PLAN_NO_VITERBI
    from paper_1701_03038_gb300.fst import Fst
    fa, strs = synth.make_config("c2", scale=0.02, strings=16)
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    ids = torch.from_numpy(strs.ids).cuda()
    off = torch.from_numpy(strs.offsets).cuda()
    pv = f.plan(ids, off, flags=PLAN_NO_FB)
    pf = f.plan(ids, off, flags=PLAN_NO_VITERBI)
    for p in (pv, pf):
        p.set_driver(_lib.DRIVER_PERSISTENT, 0, 200_000)
    B = strs.count
    ov = [o.viterbi(strs.get(b)) for b in range(B)]
    ofb = o.fb_batch(strs.ids, strs.offsets, nthreads=8)
    for p in (pv, pf):
        p.fault_inject(_lib.FAULT_BARRIER_STALL, 1)
    t0 = time.perf_counter()
    pv.viterbi()
    torch.cuda.synchronize()
    pf.forward_backward()
    torch.cuda.synchronize()
    waited = time.perf_counter() - t0
    assert waited < 30.0
    assert (pv.status[:B].cpu().numpy() == _lib.TIMEOUT).all()
    assert (pf.status[:B].cpu().numpy() == _lib.TIMEOUT).all()
    assert np.isneginf(pv.scores[:B].cpu().numpy()).all()
    assert np.isneginf(pf.logz[:B].cpu().numpy()).all()
    assert (pf.counts.cpu().numpy() == 0).all()
    # the context is still usable: the same plans, injection off, are exact
    for p in (pv, pf):
        p.fault_inject(_lib.FAULT_NONE)
    pv.viterbi()
    pf.forward_backward()
    torch.cuda.synchronize()
    sc, pa, ol, st = pv.scores.cpu().numpy(), pv.paths.cpu().numpy(), pv.olabels.cpu().numpy(), pv.status.cpu().numpy()
    for b in range(B):
        lo, hi = strs.offsets[b], strs.offsets[b + 1]
        assert_viterbi_equal(sc[b], pa[lo:hi], ol[lo:hi], st[b], ov[b])
        assert_logz_close(pf.logz[b].item(), ofb["logz"][b])
    assert_counts_close(pf.counts.cpu().numpy(), ofb["counts"], batch=True)


def _chain_fst(states=64, symbols=3, wide=0):
    """A ring whose symbols 0 .. symbols-1 each lead every state on by 1 + the
    symbol, and (wide) one more symbol of `wide` arcs out of every state."""
    q = np.arange(states)
    parts = [(q, (q + 1 + a) % states, a) for a in range(symbols)]
    if wide:
        rng = np.random.default_rng(wide)
        parts.append((np.repeat(q[:8], wide), rng.integers(0, states, 8 * wide), symbols))
    src, dst = (np.concatenate([p[k] for p in parts]).astype(np.int32) for k in (0, 1))
    lab = np.concatenate([np.full(len(p[0]), p[2]) for p in parts]).astype(np.int32)
    w = np.random.default_rng(1).uniform(0.1, 2.0, len(src)).astype(np.float32)
    start = np.full(states, np.inf, np.float32)
    start[0] = 0.0
    m = symbols + (1 if wide else 0)
    return synth.FstArrays(states, m, m, src, dst, lab, lab, w, start, np.zeros(states, np.float32))


def _plans(f, strs, **kw):
    import torch
    from paper_1701_03038_gb300._lib import PLAN_NO_FB, PLAN_NO_VITERBI
    ids, off = torch.from_numpy(strs.ids).cuda(), torch.from_numpy(strs.offsets).cuda()
    return f.plan(ids, off, flags=PLAN_NO_FB, **kw), f.plan(ids, off, flags=PLAN_NO_VITERBI, **kw)


@pytest.mark.parametrize("parts", [1, 2])
def test_string_waits_run_out_and_recover(parts):
    # two strings of 20,000 one-arc positions (some 10 ms) under a limit of a
    # microsecond: the workers without a string give up, the run reports
    # FST_ERR_TIMEOUT everywhere, and with the limit back the same plans are
    # exact
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300.fst import Fst
    fa = _chain_fst()
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    rng = np.random.default_rng(2)
    n = 20_000
    strs = synth.Strings(rng.integers(0, 3, 2 * n).astype(np.int32), np.array([0, n, 2 * n], np.int64))
    pv, pf = _plans(f, strs, parts=parts)
    for limit_us in (1, 2_000_000):
        for p in (pv, pf):
            p.set_driver(_lib.DRIVER_LAUNCH, 0, limit_us)
        pv.viterbi()
        pf.forward_backward()
        torch.cuda.synchronize()
        if limit_us == 1:
            assert (pv.status[:2].cpu().numpy() == _lib.TIMEOUT).all()
            assert (pf.status[:2].cpu().numpy() == _lib.TIMEOUT).all()
            assert np.isneginf(pv.scores[:2].cpu().numpy()).all()
            assert (pv.paths[:2 * n].cpu().numpy() == -1).all()
            assert np.isneginf(pf.logz[:2].cpu().numpy()).all()
    ofb = o.fb_batch(strs.ids, strs.offsets, nthreads=2)
    for b in range(2):
        lo, hi = strs.offsets[b], strs.offsets[b + 1]
        assert_viterbi_equal(pv.scores[b].item(), pv.paths[lo:hi].cpu().numpy(), pv.olabels[lo:hi].cpu().numpy(),
                             pv.status[b].item(), o.viterbi(strs.get(b)))
        assert_logz_close(pf.logz[b].item(), ofb["logz"][b])
    assert_counts_close(pf.counts.cpu().numpy(), ofb["counts"], batch=True)


def test_shared_position_waits_run_out_and_recover():
    # strings whose every position is shared out among the blocks, under a
    # limit of a microsecond: owners stop waiting for chunks that others hold
    # and leave their accumulators unclean; the runs after that are exact
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300.fst import Fst
    fa = _chain_fst(states=20_000, wide=6_000)
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    rng = np.random.default_rng(3)
    B, n = 12, 120
    x = rng.integers(0, 3, (B, n)).astype(np.int32)
    x[:, 0] = 3
    strs = synth.Strings(x.reshape(-1), np.arange(B + 1, dtype=np.int64) * n)
    pv, pf = _plans(f, strs)
    ov = [o.viterbi(strs.get(b)) for b in range(B)]
    ofb = o.fb_batch(strs.ids, strs.offsets, nthreads=8)
    for _ in range(3):
        for p in (pv, pf):
            p.set_driver(_lib.DRIVER_LAUNCH, 0, 1)
        pv.viterbi()
        pf.forward_backward()
        torch.cuda.synchronize()
        assert (pv.status[:B].cpu().numpy() == _lib.TIMEOUT).all()
        assert (pf.status[:B].cpu().numpy() == _lib.TIMEOUT).all()
        assert (pv.paths[:B * n].cpu().numpy() == -1).all()
        for p in (pv, pf):
            p.set_driver(_lib.DRIVER_LAUNCH, 0, 2_000_000)
        pv.viterbi()
        pf.forward_backward()
        torch.cuda.synchronize()
        for b in range(B):
            lo, hi = strs.offsets[b], strs.offsets[b + 1]
            assert_viterbi_equal(pv.scores[b].item(), pv.paths[lo:hi].cpu().numpy(), pv.olabels[lo:hi].cpu().numpy(),
                                 pv.status[b].item(), ov[b])
            assert_logz_close(pf.logz[b].item(), ofb["logz"][b])
        assert_counts_close(pf.counts.cpu().numpy(), ofb["counts"], batch=True)


@pytest.mark.parametrize("wide", [0, 6_000])
def test_backward_pass_that_gives_up_spoils_the_counts(wide):
    # a forward pass that ends, then a backward pass under a limit of a
    # microsecond: its counts would be partial, and are NaN; the next pair of
    # passes is exact
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300.fst import Fst
    fa = _chain_fst(states=20_000 if wide else 64, wide=wide)
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    rng = np.random.default_rng(4)
    B, n = (6, 100) if wide else (2, 20_000)
    x = rng.integers(0, 3, (B, n)).astype(np.int32)
    if wide:
        x[:, 0] = 3
    strs = synth.Strings(x.reshape(-1), np.arange(B + 1, dtype=np.int64) * n)
    _, pf = _plans(f, strs)
    ofb = o.fb_batch(strs.ids, strs.offsets, nthreads=8)
    for limit_us in (1, 2_000_000):
        pf.set_driver(_lib.DRIVER_LAUNCH, 0, 2_000_000)
        pf.forward()
        pf.set_driver(_lib.DRIVER_LAUNCH, 0, limit_us)
        pf.backward(torch.ones(B, device="cuda"), states=True)
        torch.cuda.synchronize()
        assert (pf.status[:B].cpu().numpy() == 0).all()
        if limit_us == 1:
            for c in (pf.counts, pf.start_counts, pf.final_counts):
                assert np.isnan(c.cpu().numpy()).all()
    for b in range(B):
        assert_logz_close(pf.logz[b].item(), ofb["logz"][b])
    assert_counts_close(pf.counts.cpu().numpy(), ofb["counts"], batch=True)
    assert abs(pf.start_counts.sum().item() - B) < 1e-4 and abs(pf.final_counts.sum().item() - B) < 1e-4


def test_long_runs_of_one_arc_positions_count_as_progress():
    # a string whose passes take several times the limit: its positions are
    # progress to the workers that wait, in both passes
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300.fst import Fst
    fa = _chain_fst()
    f, o = Fst.from_arrays(fa), oracle.Fst(fa)
    n = 600_000  # (at least 0.2 us a position: 120 ms)
    ids = np.random.default_rng(5).integers(0, 3, n + 5).astype(np.int32)
    strs = synth.Strings(ids, np.array([0, n, n + 5], np.int64))
    pv, pf = _plans(f, strs)
    for p in (pv, pf):
        p.set_driver(_lib.DRIVER_LAUNCH, 0, 25_000)
    pv.viterbi()
    pf.forward_backward()
    torch.cuda.synchronize()
    assert (pv.status[:2].cpu().numpy() == 0).all() and (pf.status[:2].cpu().numpy() == 0).all()
    for b in range(2):
        lo, hi = strs.offsets[b], strs.offsets[b + 1]
        assert_viterbi_equal(pv.scores[b].item(), pv.paths[lo:hi].cpu().numpy(), pv.olabels[lo:hi].cpu().numpy(),
                             pv.status[b].item(), o.viterbi(strs.get(b)))
        # one path: its weight, and a posterior of 1 at every position
        assert_logz_close(pf.logz[b].item(), -fa.weight[pv.paths[lo:hi].cpu().numpy()].astype(np.float64).sum())
    used = np.bincount(pv.paths[:n + 5].cpu().numpy(), minlength=fa.num_arcs)
    assert_counts_close(pf.counts.cpu().numpy(), used, batch=True)


def test_fault_inject_rejects_bad_arguments():
    import torch
    from paper_1701_03038_gb300 import _lib
    from paper_1701_03038_gb300._lib import FstError
    from paper_1701_03038_gb300.fst import Fst
    fa, strs = synth.make_config("c1", scale=0.2, strings=2)
    f = Fst.from_arrays(fa)
    p = f.plan(torch.from_numpy(strs.ids).cuda(), torch.from_numpy(strs.offsets).cuda())
    for kind, value in ((7, 0), (_lib.FAULT_BARRIER_STALL, -1), (_lib.FAULT_BARRIER_STALL, 5000)):
        with pytest.raises(FstError):
            p.fault_inject(kind, value)
    with pytest.raises(FstError):
        p.set_driver(5)
    with pytest.raises(FstError):
        p.set_driver(_lib.DRIVER_PERSISTENT, 10 ** 7)  # far more blocks than can be co-resident
