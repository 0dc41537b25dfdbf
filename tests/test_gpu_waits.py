"""The bounded waits of the persistent sampler cap the time without progress: a
CTA whose chains are done waits for the longest chain of the iteration as long
as any chain advances, and gives up where none does."""
import pytest

import swig_inputs as si
from oracle import events

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")

# A poll takes about a microsecond: far longer than a round (tens of
# microseconds) or a boundary, far shorter than the chains' differences below.
LIMIT = 3000


def _context(het=False, free=False, **extra):
    wl = si.config1(nlive=200)
    ev, th = events.build_event(wl)
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    if free:  # projection-only blocks alone: no round needs the CTA
        params = list(wl.params)
        for i, p in enumerate(params):
            if p.mode == si.MODE_SAMPLE and i not in (6, 7, 8, 12):
                params[i] = si.Param(p.kind, p.lo, p.hi, si.MODE_FIXED, th[i])
        ctx.set_prior(params)
    if het:
        extra.update(likelihood=swig.LIKE_HET, het_bins=300, het_fiducial=th)
    ctx.set_sampler(nlive=200, nrep=40, seed=3, precision=swig.PREC_MIXED, max_iter=2, **extra)
    return ctx


@pytest.mark.parametrize("kind", ["full", "het", "free"])
def test_long_chains_are_waited_for(kind):
    """Chains of thousands of steps end tens of milliseconds apart."""
    ctx = _context(het=kind == "het", free=kind == "free", sweeps=4, steps_per_dim=400 if kind == "free" else 150)
    ctx.set_wait_limit(LIMIT)
    r = ctx.run()
    assert r.n_iter == 2
    ctx.close()


def test_no_progress_is_a_timeout():
    ctx = _context()
    ctx.set_wait_limit(0)
    with pytest.raises(swig.SwigError) as e:
        ctx.run()
    assert e.value.code == swig.SWIG_E_TIMEOUT
    ctx.set_wait_limit(10_000_000)
    assert ctx.run().n_iter == 2
    ctx.close()
