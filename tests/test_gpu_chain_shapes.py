"""How many points of a slice step are evaluated at a time changes neither the
draws nor the decisions: every launch shape gives the same points and counts.

The shapes differ in the rungs and draws of a round, in whether draws are taken
ahead of the bracket and in how candidates are paired, so the sums' grouping
differs: logL within the parity bound 1e-6 |logL| + 1e-6 of the shape compared
with.  Chains: fewer than SMs, and more (a CTA takes several)."""
import numpy as np
import pytest

import swig_inputs as si
from oracle import events

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")


def _run(wl, ev, th, nrep, het, **shape):
    extra = dict(likelihood=swig.LIKE_HET, het_bins=300, het_fiducial=th) if het else {}
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ctx.set_sampler(nlive=wl.nlive, nrep=nrep, steps_per_dim=2, seed=7, precision=swig.PREC_MIXED, max_iter=4, **shape,
                    **extra)
    r = ctx.run()
    out = ctx.get_samples()
    ctx.close()
    return r, out


@pytest.mark.parametrize("nrep", [40, 200])
@pytest.mark.parametrize("het", [False, True])
def test_shapes_give_the_same_points(nrep, het):
    wl = si.config1(nlive=600)
    ev, th = events.build_event(wl)
    want, (t0, l0, w0) = _run(wl, ev, th, nrep, het)
    for shape in (dict(flow_parts=2), dict(flow_parts=3), dict(flow_parts=4), dict(stepout_one_end=1),
                  dict(flow_parts=4, stepout_one_end=1)):
        got, (t, l, w) = _run(wl, ev, th, nrep, het, **shape)
        assert (got.n_evals, got.n_sweep_evals, got.n_dead) == (want.n_evals, want.n_sweep_evals, want.n_dead), shape
        assert np.array_equal(t, t0), shape
        assert np.all(np.abs(l - l0) <= 1e-6 * np.abs(l0) + 1e-6), shape
