"""The host side of the library (csrc/api.cu, csrc/serve.cu) on a simulated device (tests/hostsim): buffer sizes, lifetimes
of host and device memory and the order of launches are checked for the calls a user makes, without a GPU."""
import ctypes
import os
import shutil
import subprocess
import time

import numpy as np
import pytest

import workloads

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_27231_gb300", "csrc")
SIM = os.path.join(ROOT, "tests", "hostsim")


@pytest.fixture(scope="module")
def sim_lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    from paper_2605_27231_gb300 import build, sigw
    real = build.build()
    so = str(tmp_path_factory.mktemp("sim") / "libsim.so")
    src = [os.path.join(CSRC, f) for f in ("api.cu", "serve.cu", "plan.cpp")] + [os.path.join(SIM, "sim.cpp")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", SIM, "-I", CSRC, "-x", "c++",
                    *src, "-ldl", "-lpthread", "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.sim_init(real.encode())
    lib.sim_launches.restype = ctypes.c_long
    lib.sim_device_bytes.restype = ctypes.c_size_t
    lib.sim_faults.restype = ctypes.c_char_p
    return lib, so, sigw


@pytest.fixture
def sim(sim_lib, monkeypatch):
    """The package's binding on the simulated device; every test has to end without a fault."""
    lib, so, sigw = sim_lib
    monkeypatch.setattr(sigw, "LIB_PATH", so)
    monkeypatch.setattr(sigw, "_lib", None)
    lib.sim_faults()
    yield sigw
    assert lib.sim_faults().decode() == ""


def _run(p, batch=1, shells=(1,), **kw):
    p.generate(1e-2, 0.5, 10.0, seeds=list(range(1, batch + 1)), **kw)
    p.spectrum(list(shells))


KINDS = slice(1, 4)  # first, second and last inverse pass among the profile's kinds


def _launches(p, kinds=KINDS):
    r = p.profile_read()
    return [r[k]["launches"] for k in [k for k in r if isinstance(r[k], dict)][kinds]]


def _autotune(sim, p):
    sim.lib().sim_check_values(0)
    r = p.autotune()
    sim.lib().sim_check_values(1)
    return r


# ---- host memory that a queued copy may still read

def test_queued_uploads_keep_their_host_buffers(sim):
    """Synthesis parameters and shell lists of calls that return, or go on, before the stream was waited for."""
    import ctypes as C
    with sim.Plan(16, 1.0, precision=64, n_alpha=5, max_batch=3) as p:
        p.target_scan(np.geomspace(0.3, 2.5, 19), 1e-2, 0.5, 1.0, "local", 2.0, seed=3)
        _run(p, 3, (8, 2, 5, 2))
        p.generate(1e-2, 0.5, 10.0, "nonlocal", alpha_NL=1.0, seeds=(1, 2))
        p.spectrum_async(None, [3, 1])
        assert sim.lib().sigw_spectrum_async(p.handle, None, 0, None) == sim.OK  # all shells, captured
        p.generate(1e-2, 0.5, 10.0, "usr")
        p.spectrum_async(None, [1])
        p.synchronize()
        p.spectrum_jackknife([1, 4])


# ---- server

def _spec(N, seed):
    return workloads.Spec(N=N, L=1.0, A=1e-2, sigma=0.5, kstar=12.0, kind="gauss", seed=seed)


def test_express_slot_leaves_the_head_what_it_has_to_evict(sim):
    """A 64^3 request at the head of the queue fits once the idle 32^3 plan is evicted, and waits for the general slot, which
    is busy.  The express slot must not keep that plan busy with a later 32^3 request; it may run a 16^3 one, whose idle plan
    the head does not need."""
    o = dict(precision=32, n_alpha=5)
    fp = {N: sim.footprint(N, sim.default_opts(**o)) for N in (32, 64, 128)}
    with sim.Server(fp[128] + fp[64] + fp[32] // 2, max_slots=1, **o) as s:
        for N in (32, 16):
            s.wait(s.submit(_spec(N, 1)), timeout_s=60)
        sim.lib().sim_hold(128)
        try:
            busy = s.submit(_spec(128, 2))
            while s.stats()["queued"]:
                time.sleep(0.001)
            s.set_express(1, 32)
            head, small, free = s.submit(_spec(64, 3)), s.submit(_spec(32, 4)), s.submit(_spec(16, 5))
            s.wait(free, timeout_s=60)
            with pytest.raises(sim.SigwError) as e:
                s.wait(small, timeout_s=0.2)
            assert e.value.status == sim.ETIMEOUT
        finally:
            sim.lib().sim_hold(0)
        for t in (busy, head, small):
            s.wait(t, timeout_s=60)
        st = s.stats()
    assert st["completed"] == 6 and st["failed"] == 0 and st["plans_evicted"] >= 1


# ---- launches

@pytest.mark.parametrize("N,n_alpha", [(32, 1), (32, 3), (32, 9), (32, 15), (32, 16), (256, 7), (128, 17)])
def test_terms_that_fit_take_one_launch(sim, N, n_alpha):
    with sim.Plan(N, 1.0, precision=64 if N == 32 else 32, n_alpha=n_alpha) as p:
        p.generate(1e-2, 0.5, 10.0)
        p.profile(False)
        p.spectrum([1, N // 2])
        assert _launches(p) == [4, 4, 4]  # passes of two shells, two kernels


@pytest.mark.parametrize("n_alpha", [2, 3, 6, 9, 13, 15])
def test_autotuner_times_the_untuned_choice(sim, n_alpha):
    """A launch takes a millisecond here, so all terms at once, the untuned choice, are the fastest."""
    with sim.Plan(32, 1.0, precision=64, n_alpha=n_alpha) as p:
        _run(p)
        _, _, ms = _autotune(sim, p)
        assert ms == 2.0  # a launch of either pass
        p.profile(False)
        p.spectrum([1])
        assert _launches(p) == [2, 2, 2]


# ---- buffers

@pytest.mark.parametrize("alpha_batch", [50, 20])
def test_terms_tuned_on_another_plan_fit_this_plan(sim, alpha_batch):
    """A plan with its own (larger) terms per launch is tuned; a default plan of the same size keeps within its buffers."""
    with sim.Plan(16, 1.0, n_alpha=50, alpha_batch=alpha_batch) as p:
        _run(p)
        _autotune(sim, p)
        _run(p)
    with sim.Plan(16, 1.0, n_alpha=50) as q:
        _run(q)


# Device memory (bytes) that admitted a plan when its stages lay side by side, with one group of term pairs and one kernel at a
# time: (N, precision, n_alpha, alpha_batch, max_batch).  A server's budget is counted in these.
FOOTPRINT = {(8, 32, 50, 0, 1): 492324,
             (8, 64, 13, 1, 64): 15125080,
             (16, 32, 5, 0, 2): 1320216,
             (32, 64, 50, 0, 1): 51553448,
             (32, 32, 3, 1, 1): 3314516,
             (64, 32, 50, 0, 1): 205358500,
             (64, 32, 50, 0, 8): 1640890752,
             (64, 32, 50, 50, 1): 276661668,
             (64, 64, 51, 0, 2): 832923184,
             (64, 32, 3, 1, 64): 1649457072,
             (128, 32, 50, 0, 1): 1640377188,
             (128, 64, 50, 0, 1): 3277990664,
             (128, 32, 1, 50, 64): 11480740560,
             (256, 32, 50, 0, 4): 52421434288,
             (256, 32, 3, 1, 1): 1639170612,
             (512, 32, 50, 0, 1): 104955218404,
             (512, 64, 50, 0, 1): 209807398280,
             (512, 64, 1, 0, 1): 22984552168}


@pytest.mark.parametrize("key", FOOTPRINT)
def test_footprint_does_not_grow(sim, key):
    o = sim.default_opts(**dict(zip(("precision", "n_alpha", "alpha_batch", "max_batch"), key[1:])))
    assert sim.footprint(key[0], o) <= FOOTPRINT[key]
    before = sim.lib().sim_device_bytes()
    with sim.Plan(key[0], 1.0, o):
        assert sim.lib().sim_device_bytes() - before <= sim.footprint(key[0], o)


@pytest.mark.parametrize("N,precision,bits", [(8, 32, 0), (16, 64, 0), (32, 64, 0), (64, 32, 24), (64, 32, 0), (64, 64, 0),
                                              (128, 32, 26), (128, 64, 0), (256, 32, 26)])
@pytest.mark.parametrize("n_alpha,alpha_batch", [(1, 0), (2, 1), (3, 1), (5, 0), (13, 4), (50, 0), (51, 7), (50, 50), (300, 300)])
def test_every_stage_finds_what_the_one_before_left(sim, N, precision, bits, n_alpha, alpha_batch):
    """All buffers of the hot loop share one block: spectra, jackknife and the transforms' scratch over every plan form."""
    o = dict(precision=precision, n_alpha=n_alpha, n_modes=max(200, n_alpha), alpha_batch=alpha_batch, max_batch=3)
    shells = sorted({1, 2, N // 4, N // 2 - 1, N // 2})
    with sim.Plan(N, 1.0, **o) as p:
        for batch, choices in ((1, (None,)), (3, (None, 1, 2, 3, 10))):
            p.generate(1e-2, 0.5, 10.0, "nonlocal", alpha_NL=1.0, seeds=range(batch))
            for c in choices:
                if c is not None and c <= min(n_alpha, alpha_batch or 16):
                    p.set_tuning(c, bits)
                p.spectrum(shells)
            p.spectrum_jackknife(shells[:-1], M=2)
            p.spectrum([N // 2])
        _autotune(sim, p)
        p.spectrum(shells)
