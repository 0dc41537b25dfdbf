"""The folded sums' rounding does not depend on how few warps share a vector.

A lane adds its nodes in FP32 over 32 chunks at most and in double-float beyond
that (blocks, lanes, warps).  With N chunks on one warp a block of 32 is 1 / N of |Z|
for a lane and each of its 64 additions errs by 2^-24 of it at most, of random sign:
over the N blocks of all lanes sqrt(64 N) / N x 2^-24 |Z| = 8 / sqrt(N) x 2^-24 |Z|,
0.9 x 2^-24 |Z| for N = 78, and a third of that as a root mean square (roundings are
uniform, partials grow from zero): 0.3 x 2^-24 |Z|.  Smaller blocks and sixteen warps
a vector err by less.  One FP32 sum over all chunks, lanes added in FP32 and kappa
rounded to FP32 come to half of 2^-24 |Z|."""
import numpy as np
import pytest

import swig_inputs as si
from oracle import events

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")


def test_large_and_small_batches_round_alike():
    wl = si.config2()
    ev, th = events.build_event(wl)
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ctx.set_sampler(nlive=100, nrep=10, precision=swig.PREC_MIXED)
    rng = np.random.default_rng(5)
    n = 3000  # beyond eight vectors per SM: a warp each
    thetas = np.tile(th, (n, 1))
    thetas[:, 0] *= 1.0 + 2e-6 * rng.standard_normal(n)  # near the peak: |Z| about SNR^2 = 625
    thetas[:, 11] += 2e-5 * rng.standard_normal(n)
    thetas[:, 12] = rng.uniform(0.0, 2.0 * np.pi, n)
    large = ctx.loglike_batch(thetas)
    small = np.concatenate([ctx.loglike_batch(thetas[i:i + 100]) for i in range(0, n, 100)])
    rms = np.sqrt(np.mean((large - small) ** 2))
    assert rms <= 0.3 * 2.0**-24 * 625.0, rms
    ctx.close()
