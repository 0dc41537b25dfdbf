"""The batched heterodyned likelihood on the GPU against the FP64 oracle where
its work split can go wrong: batches of one, odd and even numbers of vectors per
block, vectors that take chunks edge by edge next to vectors that do not, one to
four detectors, more chunks than are anchored at once, a ragged last chunk.

Bound: the repository's parity bound |dlogL| <= 1e-6 |logL| + 1e-6."""
import dataclasses

import numpy as np
import pytest

import swig_inputs as si
from oracle import events, physics
from oracle import likelihood as L

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")


def _check(got, want):
    assert np.all(np.abs(got - want) <= 1e-6 * np.abs(want) + 1e-6), np.max(np.abs(got - want))


def _draws(wl, n, seed):
    rng = np.random.default_rng(seed)
    return np.array([physics.prior_transform(rng.random(len(wl.sampled())), wl.params)[0] for _ in range(n)])


@pytest.mark.parametrize("spacing", [0, 1])
def test_batch_sizes_with_edge_by_edge_chunks(spacing):
    wl = si.config1()
    ev, th = events.build_event(wl)
    het = L.het_setup(ev, th, 450, spacing="phase" if spacing == 0 else "geometric")
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ctx.set_sampler(nlive=100, nrep=10, likelihood=swig.LIKE_HET, het_bins=450, het_spacing=spacing, het_fiducial=th)
    thetas = _draws(wl, 1300, 1)
    thetas[::2] = th
    thetas[::2, 0] *= 1.0 + 1e-5 * np.arange(650)  # near the fiducial beside prior draws
    thetas[7, 1] = 2.0
    idx = np.r_[0:12, 300:312, 1290:1300]
    want = np.array([L.het_loglike(ev, het, thetas[i]) if i != 7 else -np.inf for i in idx])
    for n in (1, 2, 152, 153, 307, 611, 1300):
        got = ctx.loglike_batch(thetas[:n])
        use = idx < n
        ok = use & np.isfinite(want)
        assert np.array_equal(np.flatnonzero(np.isneginf(got)), [7] if n > 7 else [])
        _check(got[idx[ok]], want[ok])
    ctx.close()


@pytest.mark.parametrize("dets,bins", [(("H1",), 33), (("H1", "V1"), 9000), (("H1", "L1", "V1"), 1000),
                                       (("H1", "L1", "V1", "H1"), 700)])
def test_detectors_and_chunk_counts(dets, bins):
    wl = dataclasses.replace(si.config2(seed_index=4), detectors=dets, f_max=1024.0, df=1 / 16)
    ev, th = events.build_event(wl)
    het = L.het_setup(ev, th, bins)
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ctx.set_sampler(nlive=100, nrep=10, likelihood=swig.LIKE_HET, het_bins=bins, het_fiducial=th)
    thetas = np.concatenate([_draws(wl, 320, 2), np.tile(th, (5, 1))])
    thetas[320:, 0] *= 1.0 + 5e-5 * np.arange(5)
    got = ctx.loglike_batch(thetas)
    idx = [0, 1, 2, 3, 160, 319, 320, 321, 324]
    _check(got[idx], np.array([L.het_loglike(ev, het, thetas[i]) for i in idx]))
    ctx.close()
