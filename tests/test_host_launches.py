"""What the host code asks of the device and in which order, on the CPU: the
library's own objects linked with a runtime that has no device
(fake_runtime.cu) and driven through the Python binding."""
import ctypes
import dataclasses
import os
import shutil
import subprocess

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
