"""GPU parity where the last pair of terms has one member: every form of the second and the last pass at odd term counts,
in one launch and in several, alone and in a batch.  Up to 128^3 against the CPU FP64 oracle (FP64 1e-9, FP32 1e-4 relative
per shell, as everywhere on this path), above against the FP64 path."""
import numpy as np
import pytest

import workloads
from oracle import decomposition as odec
from oracle import sigw as osigw
from oracle import synth

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


def _spec(N):
    return workloads.Spec(N=N, L=1.0, A=1e-2, sigma=0.5, kstar=(N // 8) * 2 * np.pi, kind="local", F_NL=2.0, seed=47)


def _check(lib, N, precision, n_alpha, shells, ref, rtol):
    spec = _spec(N)
    with lib.Plan(N, 1.0, precision=precision, n_alpha=n_alpha, max_batch=2) as p:
        p.generate_spec(spec, seeds=[spec.seed, 5])
        both = p.spectrum(shells)["omega"]
        np.testing.assert_allclose(both[0], ref, rtol=rtol)
        p.generate_spec(spec)
        assert np.array_equal(p.spectrum(shells)["omega"][0], both[0])
        for choice in (1, 2, 4):  # several launches, the last one with the single term
            if choice <= n_alpha:
                for bits in ((0, 2, 8, 26) if precision == 32 else (0,)):
                    p.set_tuning(choice, bits)
                    np.testing.assert_allclose(p.spectrum(shells)["omega"][0], ref, rtol=rtol)


@pytest.mark.parametrize("N,precision,n_alpha", [(64, 64, 5), (128, 32, 1), (128, 32, 3), (128, 32, 13), (128, 64, 3)])
def test_odd_terms_match_oracle(lib, N, precision, n_alpha):
    shells = [3, N // 4]
    spec = _spec(N)
    Phi, _ = synth.phi_tilde(spec.N, spec.L, spec.A, spec.sigma, spec.kstar, spec.seed, spec.kind, spec.F_NL)
    ref = osigw.omega(Phi, spec.L, odec.build(n_alpha=n_alpha), shells=shells)["omega"]
    _check(lib, N, precision, n_alpha, shells, ref, 1e-9 if precision == 64 else 1e-4)


@pytest.mark.parametrize("N,n_alpha", [(256, 5), (512, 3)])
def test_odd_terms_match_double_precision(lib, N, n_alpha):
    shells = [5, N // 4]
    with lib.Plan(N, 1.0, precision=64, n_alpha=n_alpha) as p:
        p.generate_spec(_spec(N))
        ref = p.spectrum(shells)["omega"][0]
    _check(lib, N, 32, n_alpha, shells, ref, 1e-4)
