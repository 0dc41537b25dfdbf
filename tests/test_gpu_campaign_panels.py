"""Events that share a launch get the results of separate runs also where their
chunks do not fit in shared memory at once and another event's live set makes
the launch's scratch, and with it the panels of chunks, longer."""
import dataclasses

import numpy as np
import pytest

import swig_inputs as si
from oracle import events

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")


def _contexts():
    out = []
    for i, nlive in enumerate((300, 6000)):
        wl = dataclasses.replace(si.config2(nlive=nlive, seed_index=5 + i), f_max=1024.0, df=1 / 16, detectors=("H1",))
        ev, th = events.build_event(wl)
        params = list(wl.params)  # a wide box: several hundred chunks
        params[0] = si.Param(si.PRIOR_UNIFORM, 0.9, 3.0, block=params[0].block)
        params[11] = si.Param(si.PRIOR_UNIFORM, -3.0, 3.0, block=params[11].block)
        ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
        ctx.set_prior(params)
        ctx.set_sampler(nlive=nlive, nrep=30, steps_per_dim=5, seed=11 + i, precision=swig.PREC_MIXED, max_iter=3)
        out.append(ctx)
    return out


def test_shared_launch_equals_separate_runs():
    single = []
    for ctx in _contexts():
        r = ctx.run()
        single.append((r, ctx.get_samples()))
        ctx.close()
    ctxs = _contexts()
    res = swig.run_batch(ctxs)
    for (r1, (t1, l1, w1)), r2, ctx in zip(single, res, ctxs):
        t2, l2, w2 = ctx.get_samples()
        assert (r1.logz, r1.n_evals, r1.n_dead) == (r2.logz, r2.n_evals, r2.n_dead)
        assert np.array_equal(t1, t2) and np.array_equal(l1, l2) and np.array_equal(w1, w2)
        ctx.close()
