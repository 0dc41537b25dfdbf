"""The folded full-grid likelihood (mixed precision) on the GPU against the
FP64 oracle, where it can go wrong: one to four detectors, grids of one chunk, a
ragged last chunk, more chunks than are anchored at once, batches around the
grid size of the launch, and parameter vectors outside the prior box the folded
weights serve (summed bin by bin).

Bound: the repository's parity bound |dlogL| <= 1e-6 |logL| + 1e-6; on the grids
below its absolute part never exceeds 0.1.
"""
import dataclasses
import math

import numpy as np
import pytest

import swig_inputs as si
from oracle import events, physics
from oracle import likelihood as L

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")


def _draws(params, n, seed):
    rng = np.random.default_rng(seed)
    ns = sum(1 for p in params if p.mode == si.MODE_SAMPLE)
    return np.array([physics.prior_transform(rng.random(ns), params)[0] for _ in range(n)])


def _event(dets, f_min, f_max, df, seed=3):
    wl = dataclasses.replace(si.config2(seed_index=seed), detectors=dets, f_min=f_min, f_max=f_max, df=df)
    ev, th = events.build_event(wl)
    return wl, ev, th


def _context(wl, ev):
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ctx.set_sampler(nlive=100, nrep=10, precision=swig.PREC_MIXED)
    return ctx


def _check(got, want):
    assert np.all(np.abs(got - want) <= 1e-6 * np.abs(want) + 1e-6), np.max(np.abs(got - want))


@pytest.mark.parametrize("dets,f_min,f_max,df", [
    (("H1",), 20.0, 512.0, 1 / 16),                # one detector
    (("H1", "L1", "V1", "H1"), 20.0, 300.0, 1 / 8),  # four
    (("H1", "V1"), 40.0, 43.7, 1 / 16),            # a single ragged chunk (60 bins)
    (("H1", "L1"), 19.0, 1990.0, 1 / 11),          # odd spacing, ragged end
])
def test_grids_against_the_oracle(dets, f_min, f_max, df):
    wl, ev, th = _event(dets, f_min, f_max, df)
    ctx = _context(wl, ev)
    thetas = np.concatenate([_draws(wl.params, 8, 1), np.tile(th, (4, 1))])
    thetas[8:, 0] *= 1.0 + 1e-4 * np.arange(4)
    _check(ctx.loglike_batch(thetas), np.array([L.loglike(ev, t) for t in thetas]))
    ctx.close()


def test_more_chunks_than_a_panel_of_anchors():
    """A wide t_c range and mass box: more chunks than are anchored at once."""
    wl, ev, th = _event(("H1",), 20.0, 1024.0, 1 / 32)
    params = list(wl.params)
    params[0] = si.Param(si.PRIOR_UNIFORM, 0.9, 3.0)
    params[11] = si.Param(si.PRIOR_UNIFORM, -3.0, 3.0, block=6)
    wl = dataclasses.replace(wl, params=params)
    ev = L.Event(ev.freqs, ev.df, ev.data, ev.psds, ev.detectors, ev.gmst, params)
    ctx = _context(wl, ev)
    thetas = _draws(params, 10, 5)
    _check(ctx.loglike_batch(thetas), np.array([L.loglike(ev, t) for t in thetas]))
    ctx.close()


def test_batch_sizes_around_the_launch_and_invalid_vectors():
    wl, ev, th = _event(("H1", "L1", "V1"), 20.0, 400.0, 1 / 4)
    ctx = _context(wl, ev)
    thetas = _draws(wl.params, 700, 2)
    thetas[5, 1] = 1.5
    thetas[303, 6] = -1.0
    thetas[304, 0] = np.nan
    full = ctx.loglike_batch(thetas)
    bad = np.isneginf(full)
    assert sorted(np.flatnonzero(bad)) == [5, 303, 304]
    idx = [0, 6, 150, 302, 305, 699]
    want = np.array([L.loglike(ev, thetas[i]) for i in idx])
    _check(full[idx], want)
    for n in (1, 2, 31, 33, 151, 152, 153, 303, 304, 305, 609):  # the work split depends on the batch
        got = ctx.loglike_batch(thetas[:n])
        assert np.array_equal(np.isneginf(got), bad[:n])
        m = sum(i < n for i in idx)
        _check(got[idx[:m]], want[:m])
    ctx.close()


def test_vectors_outside_the_prior_box():
    """Far from the box the folded weights do not serve the template: these
    vectors are summed bin by bin; a context whose box holds them folds."""
    wl, ev, th = _event(("H1", "V1"), 20.0, 900.0, 1 / 16)
    ctx = _context(wl, ev)
    rng = np.random.default_rng(8)
    thetas = _draws(wl.params, 12, 3)
    thetas[:, 0] = rng.uniform(0.9, 1.2, 12)      # box: 1.5 .. 2.5
    thetas[::2, 11] = rng.uniform(0.5, 2.0, 6)    # box: -0.1 .. 0.1
    thetas[3, 4:6] = 3e4                          # box: 0 .. 5000
    want = np.array([L.loglike(ev, t) for t in thetas])
    _check(ctx.loglike_batch(thetas), want)
    mixed = np.concatenate([thetas, _draws(wl.params, 5, 4)])
    got = ctx.loglike_batch(mixed)
    assert np.array_equal(got[:12], ctx.loglike_batch(thetas))
    _check(got, np.array([L.loglike(ev, t) for t in mixed]))
    params = list(wl.params)
    params[0] = si.Param(si.PRIOR_UNIFORM, 0.85, 2.5)
    params[11] = si.Param(si.PRIOR_UNIFORM, -2.1, 2.1, block=6)
    params[4] = si.Param(si.PRIOR_UNIFORM, 0.0, 3.1e4)
    params[5] = si.Param(si.PRIOR_UNIFORM, 0.0, 3.1e4)
    ctx.set_prior(params)
    _check(ctx.loglike_batch(thetas), want)
    assert math.isfinite(want.sum())
    ctx.close()


def test_without_a_prior():
    wl, ev, th = _event(("H1",), 20.0, 512.0, 1 / 8)
    ctx = swig.Context(0)
    ctx.set_grid(wl.f_min, wl.f_max, wl.df)
    ctx.set_detector(0, *si.site_vectors("H1"))
    ctx.set_data(0, ev.data[0])
    ctx.set_psd(0, ev.psds[0])
    ctx.set_time_ref(ev.gmst)
    thetas = _draws(wl.params, 6, 9)
    thetas[:, 12] = np.linspace(0.0, 6.0, 6)
    plain = list(wl.params)
    plain[12] = si.Param(si.PRIOR_UNIFORM, 0.0, 2 * math.pi)
    ev2 = L.Event(ev.freqs, ev.df, ev.data, ev.psds, ev.detectors, ev.gmst, plain)
    _check(ctx.loglike_batch(thetas), np.array([L.loglike(ev2, t) for t in thetas]))
    ctx.close()
