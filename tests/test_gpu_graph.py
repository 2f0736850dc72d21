"""The captured all-shells graph (a null shell list at the C ABI; the binding's Plan.spectrum passes its list): the bits of
direct launches on capture, on replay, after a change of the batch, the box or the tuning, and after a wait that gave up."""
import ctypes

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_27231_gb300 import build, sigw
    build.build()
    sigw.lib()
    return sigw


def _graph(lib, p):
    out = np.zeros((p.batch, p.N // 2))
    st = lib.lib().sigw_spectrum(p.handle, None, 0, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), None, None, None)
    assert st == lib.OK, st
    return out


@pytest.mark.parametrize("N,precision,n_alpha", [(16, 64, 7), (32, 32, 50), (64, 32, 50), (128, 32, 21)])
def test_graph_gives_the_bits_of_direct_launches(lib, N, precision, n_alpha):
    spec = workloads.Spec(N=N, L=1.0, A=1e-2, sigma=0.5, kstar=(N // 8) * 2 * np.pi, kind="local", F_NL=2.0, seed=3)

    def same(p):
        direct = p.spectrum()["omega"]
        assert np.array_equal(_graph(lib, p), direct) and np.array_equal(_graph(lib, p), direct)
        return direct

    with lib.Plan(N, 1.0, precision=precision, n_alpha=n_alpha, max_batch=2) as p:
        p.generate_spec(spec, seeds=[3, 4])
        two = same(p)
        p.generate_spec(spec)
        assert np.array_equal(same(p)[0], two[0])
        p.set_tuning(4, 0)
        same(p)
        p.set_box(0.8)
        p.generate_spec(spec)
        clean = same(p)
        p.debug_wait_limit(1)
        assert lib.lib().sigw_spectrum(p.handle, None, 0, None, None, None, None) == lib.ETIMEOUT
        p.debug_wait_limit(0)
        assert np.array_equal(_graph(lib, p), clean)
