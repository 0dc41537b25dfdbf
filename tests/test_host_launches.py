"""What the host code asks of the device and in which order, on the CPU: the
library's own objects linked with a runtime that has no device
(fake_runtime.cu) and driven through the Python binding."""
import ctypes
import dataclasses
import os
import shutil
import subprocess

import numpy as np
import pytest

import swig_inputs as si
from oracle import events
from paper_2607_28265_gb300 import build, swig

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    objs = [os.path.join(build.LIBDIR, "obj", s.replace(".cu", ".o")) for s in build.SOURCES]
    if not all(map(os.path.exists, objs)):
        build.build()
    so = str(tmp_path_factory.mktemp("host") / "libswig_no_device.so")
    cmd = [nvcc] + build.ARCH + ["-std=c++17", "-O1", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-I",
                                 build.INCLUDE, "-I", build.CSRC, "-cudart", "none", "-shared", "-Xlinker",
                                 "-Bsymbolic", "-o", so, os.path.join(ROOT, "tests", "fake_runtime.cu")] + objs
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    lib = ctypes.CDLL(so)
    for name, (res, args) in swig.SIGNATURES.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    lib.fake_get.restype = ctypes.c_longlong
    return lib


@pytest.fixture
def device(fake_lib, monkeypatch):
    monkeypatch.setattr(swig, "_lib", fake_lib)
    fake_lib.fake_set(b"sms", 152)
    fake_lib.fake_reset()
    return fake_lib


def _report(lib):
    buf = ctypes.create_string_buffer(1 << 16)
    lib.fake_report(buf, len(buf))
    return sorted(set(buf.value.decode().splitlines()))


def _context(i=0, nlive=200, nrep=20, het=False, **extra):
    wl = dataclasses.replace(si.config1(nlive=nlive), noise_seed=9100 + i, sampler_seed=9200 + i)
    ev, th = events.build_event(wl)
    ctx = swig.context_for_workload(wl, ev.data, ev.psds, ev.gmst)
    if het:
        extra.update(likelihood=swig.LIKE_HET, het_bins=300, het_fiducial=th)
    ctx.set_sampler(**{**dict(nlive=nlive, nrep=nrep, seed=1, precision=swig.PREC_MIXED), **extra})
    return ctx, th


@pytest.mark.parametrize("n_ev", [1, 2, 4])
@pytest.mark.parametrize("nrep", [20, 100, 160])
def test_campaign_counters_stay_in_their_buffer(device, n_ev, nrep):
    """A shared launch has a CTA per chain of all its events, up to the SMs: more
    than any event's rows of CTA counters."""
    ctxs = [_context(i, nlive=400, nrep=nrep)[0] for i in range(n_ev)]
    swig.run_batch(ctxs)
    assert not [r for r in _report(device) if "counters" in r or "past" in r]
    for c in ctxs:
        c.close()


def _hazards(lib):
    return [r for r in _report(lib) if "counters" not in r]


@pytest.mark.parametrize("kind", ["mixed", "fp64", "het", "het_time"])
def test_uploads_precede_the_kernels_that_read_them(device, kind):
    """Preparation, a batch on another stream and a run: no kernel is launched
    while a copy that it may read is under way, and no copy's host array goes
    before the copy is done."""
    extra = {"mixed": {}, "fp64": dict(precision=swig.PREC_FP64), "het": dict(het=True),
             "het_time": dict(het=True, tmarg_nodes=256)}[kind]
    ctx, th = _context(max_iter=4, **extra)
    if kind == "het_time":
        params = list(si.config1(nlive=200).params)
        params[11] = si.Param(params[11].kind, params[11].lo, params[11].hi, si.MODE_MARG)
        ctx.set_prior(params)
    theta, out = np.tile(th, (100, 1)), np.empty(100)
    device.fake_set(b"check streams", 1)
    # (host arrays for device pointers: no kernel runs)
    ctx.loglike_batch_dev(theta.ctypes.data, 100, out.ctypes.data, 0x1000)
    device.cudaStreamSynchronize(ctypes.c_void_p(0x1000))
    ctx.loglike_batch(theta)
    ctx.run()
    ctx.get_samples()
    assert not _hazards(device)
    ctx.close()


def test_uploads_of_a_campaign(device):
    ctxs = [_context(i)[0] for i in range(3)]
    swig.run_batch(ctxs)
    assert not _hazards(device)
    for c in ctxs:
        c.close()


def test_uploads_of_the_learned_proposal(device):
    ctx = swig.Context(0)
    rng = np.random.default_rng(0)
    params = ctx.mlp_init(1)
    x, t, u = rng.standard_normal((40, 13)), rng.standard_normal((40, 13)), rng.random((40, 5))
    ctx.mlp_forward(params, x)
    ctx.mlp_loss_grad(params, x, t, t, 13)
    ctx.mlp_targets(u)
    ctx.mlp_train(u, params, 2, lr=1e-3)
    assert not _hazards(device)
    ctx.close()
    ctx, _ = _context(proposal=swig.PROPOSAL_LEARNED, max_iter=4)
    ctx.run()
    assert not _hazards(device)
    ctx.close()


def test_uploads_of_an_injection(device):
    ctx, th = _context()
    ctx.inject(th, 1, target_snr=20.0)
    assert not _hazards(device)
    ctx.close()


def test_contexts_do_not_lower_each_others_shared_memory_limit(device):
    """The limit is the function's and contexts may run in several threads: calls
    of different sizes, types and grids never lower it."""
    def use(i, **kw):
        ctx, th = _context(i, max_iter=2, **kw)
        theta = np.tile(th, (400, 1))
        for n in (400, 1, 160):
            ctx.loglike_batch(theta[:n])
        ctx.run()
        ctx.close()

    for het in (True, False):
        use(0, het=het, nlive=2000)
        use(1, het=het, nlive=200)
    rng = np.random.default_rng(0)
    ctx = swig.Context(0)
    params = ctx.mlp_init(1)
    for n in (2000, 40):
        ctx.mlp_train(rng.random((n, 5)), params, 2, lr=1e-3)
    ctx.close()
    assert not _report(device)


@pytest.mark.parametrize("n", [1, 37, 300, 5000, 16384, 20000])
def test_scratch_of_a_batch_holds_its_strays(device, n):
    """Records, list, counts and partial sums of any batch lie in its scratch, also
    in the fixed one of the entry point that does not allocate."""
    ctx, th = _context()
    theta, out = np.tile(th, (n, 1)), np.empty(n)
    ctx.loglike_batch(theta)
    cap = n
    try:
        ctx.loglike_batch_noalloc(theta.ctypes.data, n, out.ctypes.data, 0x1000)
    except swig.SwigError as e:
        cap = int(str(e).split(" parameter vectors")[0].split()[-1])
        ctx.loglike_batch_noalloc(theta.ctypes.data, cap, out.ctypes.data, 0x1000)
    assert cap >= min(n, 100)
    assert not _report(device)
    ctx.close()


def test_a_context_per_event_reuses_the_mapped_memory(device):
    """Small host batches of contexts made one after another page-lock memory once,
    not in each one's first call; what is kept is bounded, and dropped where a device
    reset has freed it."""
    def once(ctx, th):
        ctx.loglike_batch(th[None])
        ctx.close()

    once(*_context())
    device.fake_reset()
    for i in range(5):
        once(*_context(i))
    assert device.fake_get(b"cudaHostAlloc") == 0 and device.fake_get(b"cudaFreeHost") == 0
    many = [_context(i % 3) for i in range(30)]
    for ctx, th in many:
        ctx.loglike_batch(th[None])
    for ctx, _ in many:
        ctx.close()
    assert device.fake_get(b"hosts") <= 16
    device.fake_set(b"forget hosts", 1)
    once(*_context())
    assert device.fake_get(b"hosts") == 1
    assert not _report(device)


@pytest.mark.parametrize("het", [False, True])
def test_small_batches_hold_no_scratch_of_the_fp64_path(device, het):
    """A new event's first call pays for what it allocates: the partial sums per slice
    of the FP64 path (256 vectors x 31 slices x 4 x 64 bytes) are not among it."""
    ctx, th = _context(het=het)
    ctx.loglike_batch(th[None])
    held = device.fake_get(b"bytes")
    ctx.close()
    assert held - device.fake_get(b"bytes") < 256 * 31 * 4 * 64
    assert not _report(device)


@pytest.mark.parametrize("kind", ["mixed", "fp64", "het"])
def test_a_long_batch_is_captured_after_a_batch_of_4096(device, kind):
    """Nothing is allocated or freed under capture: the batch is recorded in pieces
    that the scratch serves."""
    ctx, th = _context(**{"mixed": {}, "fp64": dict(precision=swig.PREC_FP64), "het": dict(het=True)}[kind])
    theta, out = np.tile(th, (20000, 1)), np.empty(20000)
    ctx.loglike_batch(theta[:4500])
    device.fake_reset()
    device.fake_set(b"capturing", 1)
    try:
        ctx.loglike_batch_dev(theta.ctypes.data, 20000, out.ctypes.data, 0x1000)
    finally:
        device.fake_set(b"capturing", 0)
    assert device.fake_get(b"cudaMalloc") == 0 and device.fake_get(b"cudaFree") == 0
    ctx.close()
