"""Batches beyond what one launch takes (16,384 vectors; 4,096 in FP64), on host
arrays, on device pointers and in a captured graph: the vectors on both sides of a
boundary against the FP64 oracle.

Bound: the repository's parity bound |dlogL| <= 1e-6 |logL| + 1e-6."""
import numpy as np
import pytest

import swig_inputs as si
from oracle import events
from oracle import likelihood as L

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")
torch = pytest.importorskip("torch")


def _case(kind, n):
    wl = si.config1()
    ev, th = events.build_event(wl)
    rng = np.random.default_rng(6)
    thetas = np.tile(th, (n, 1))
    thetas[:, 0] *= 1.0 + 1e-4 * rng.standard_normal(n)
    thetas[:, 11] += 1e-3 * rng.standard_normal(n)
    extra, value = {}, lambda t: L.loglike(ev, t)
    if kind == "het":
        het = L.het_setup(ev, th, 300)
        extra, value = dict(likelihood=swig.LIKE_HET, het_bins=300, het_fiducial=th), lambda t: L.het_loglike(ev, het, t)
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    ctx.set_sampler(nlive=100, nrep=10, precision=swig.PREC_FP64 if kind == "fp64" else swig.PREC_MIXED, **extra)
    return ctx, thetas, value


def _check(got, thetas, value, idx):
    want = np.array([value(thetas[i]) for i in idx])
    assert np.all(np.abs(got[idx] - want) <= 1e-6 * np.abs(want) + 1e-6)


def _device(ctx, thetas):
    t = torch.from_numpy(thetas).cuda()
    out = torch.full((len(thetas),), np.nan, dtype=torch.float64, device="cuda")
    return t, out, lambda: ctx.loglike_batch_dev(t.data_ptr(), len(thetas), out.data_ptr(),
                                                 torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("kind,piece", [("mixed", 16384), ("het", 16384), ("fp64", 4096)])
def test_both_sides_of_a_piece(kind, piece):
    ctx, thetas, value = _case(kind, 2 * piece + 37)
    idx = [0, piece - 1, piece, 2 * piece - 1, 2 * piece, 2 * piece + 36]
    host = ctx.loglike_batch(thetas)
    assert np.all(np.isfinite(host))
    _check(host, thetas, value, idx)
    _, out, call = _device(ctx, thetas)
    call()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), host)
    ctx.close()


@pytest.mark.parametrize("kind", ["mixed", "het", "fp64"])
def test_captured_in_pieces_of_the_scratch(kind):
    ctx, thetas, value = _case(kind, 10000)
    ctx.loglike_batch(thetas[:4500])  # the scratch
    t, out, call = _device(ctx, thetas)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    graph.replay()
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.all(np.isfinite(got))
    _check(got, thetas, value, [0, 4095, 4096, 4499, 4500, 8999, 9000, 9999])
    ctx.close()
