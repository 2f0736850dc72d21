"""The jackknife where its scratch shares the plan's memory with the first pass of both kernels (64^3 FP32, the fused pass),
where two kernels share its passes (up to 128^3), and where a small plan runs them one by one; against the oracle, with the
tolerances of the small lattices, and a realisation's bits alone and in a batch."""
import numpy as np
import pytest

import workloads
from oracle import decomposition as odec
from oracle import jackknife as ojk
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


@pytest.mark.parametrize("N,precision,n_alpha,alpha_batch", [(64, 32, 50, 0), (64, 64, 12, 0), (128, 32, 11, 0),
                                                             (64, 32, 3, 1), (16, 64, 1, 1), (16, 32, 50, 0)])
def test_jackknife_matches_oracle(lib, N, precision, n_alpha, alpha_batch):
    spec = workloads.Spec(N=N, L=1.0, A=2e-2, sigma=0.5, kstar=(N // 4) * 2 * np.pi, kind="local", F_NL=2.0, seed=21)
    shells = [2, N // 2 - 1]
    Phi, _ = synth.phi_tilde(spec.N, spec.L, spec.A, spec.sigma, spec.kstar, spec.seed, spec.kind, spec.F_NL)
    ref = ojk.jackknife(Phi, spec.L, odec.build(n_alpha=n_alpha), shells, M=4)
    with lib.Plan(N, 1.0, precision=precision, n_alpha=n_alpha, alpha_batch=alpha_batch, max_batch=2) as p:
        p.generate_spec(spec)
        got = p.spectrum_jackknife(shells)
        plain = p.spectrum(shells)
        p.generate_spec(spec, seeds=[4, spec.seed])
        both = p.spectrum_jackknife(shells)
    rm, rs = (1e-9, 1e-8) if precision == 64 else (1e-4, 2e-3)
    for k in ("omega", "PA", "PB"):
        np.testing.assert_allclose(got[k][0], ref[k], rtol=rm)
        np.testing.assert_allclose(got["sigma_" + k][0], ref["sigma_" + k], rtol=rs)
        np.testing.assert_allclose(got[k][0], plain[k][0], rtol=1e-12 if precision == 64 else 1e-5)
        assert np.array_equal(both[k][1], got[k][0]) and np.array_equal(both["sigma_" + k][1], got["sigma_" + k][0])
