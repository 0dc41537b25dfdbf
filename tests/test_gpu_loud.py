"""A loud signal: Z and <h|h> / 2 are tens of thousands and cancel in logL, so that
their roundings, and not |logL|, set the error of the sampled points.  Every dead
point's logL against the FP64 likelihood of the reported parameters (itself held to
the oracle elsewhere), within the parity bound 1e-6 |logL| + 1e-6."""
import numpy as np
import pytest

import swig_inputs as si
from oracle import events

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")


@pytest.mark.parametrize("marg", [False, True])
def test_every_dead_point_of_a_loud_signal(marg):
    wl = si.config1()
    th = wl.injection.copy()
    th[0], th[1], th[6] = 1.2933, 0.9724, 21.36
    wl.injection, wl.target_snr = th, 0.0
    if marg:
        params = list(wl.params)
        params[12] = si.Param(si.PRIOR_UNIFORM, 0.0, 2 * np.pi, si.MODE_MARG)
        wl.params = params
    ev, _ = events.build_event(wl)
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ref = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ref.set_sampler(nlive=200, nrep=20, precision=swig.PREC_FP64)
    for seed in (1, 2):
        ctx.set_sampler(nlive=200, nrep=20, steps_per_dim=5, seed=seed, precision=swig.PREC_MIXED)
        assert ctx.run().status == 0
        thd, ll, _ = ctx.get_samples()
        want = ref.loglike_batch(thd)
        err = np.abs(ll - want) / (1e-6 * np.abs(want) + 1e-6)
        assert err.max() <= 1.0, err.max()
    ctx.close()
    ref.close()
