"""GPU parity of the launch forms for small lattices against the CPU FP64 oracle: the fused second and last pass
(FP32, N = 64) and the last pass whose term pairs are split into groups (N <= 32), at term counts where the split is
uneven (one term, an odd last pair, fewer pairs than groups), in batches, and at the first, an inner and the Nyquist
shell.  Tolerances as everywhere on this path: FP32 1e-4, FP64 1e-9 relative per shell; a realisation has the same
bits alone and in a batch."""
import numpy as np
import pytest

import workloads
from oracle import decomposition as odec
from oracle import sigw as osigw
from oracle import synth

pytestmark = pytest.mark.gpu

RTOL = {64: 1e-9, 32: 1e-4}


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_27231_gb300 import build, sigw
    build.build()
    sigw.lib()
    return sigw


@pytest.mark.parametrize("N,precision", [(64, 32), (32, 32), (32, 64), (16, 64), (8, 32)])
@pytest.mark.parametrize("n_alpha", [1, 2, 5, 13])
def test_split_terms_match_oracle(lib, N, precision, n_alpha):
    spec = workloads.Spec(N=N, L=1.0, A=1e-2, sigma=0.5, kstar=(N // 8 if N > 8 else 2) * 2 * np.pi, kind="local",
                          F_NL=2.0, seed=41)
    shells = [1, N // 4 + 1, N // 2]
    Phi, _ = synth.phi_tilde(spec.N, spec.L, spec.A, spec.sigma, spec.kstar, spec.seed, spec.kind, spec.F_NL)
    ref = osigw.omega(Phi, spec.L, odec.build(n_alpha=n_alpha), shells=shells)
    with lib.Plan(N, spec.L, precision=precision, n_alpha=n_alpha, max_batch=3) as p:
        p.generate_spec(spec)
        alone = p.spectrum(shells)
        p.generate_spec(spec, seeds=[7, spec.seed, 9])
        batched = p.spectrum(shells)
    for key in ("omega", "PA", "PB"):
        np.testing.assert_allclose(alone[key][0], ref[key], rtol=RTOL[precision])
        assert np.array_equal(batched[key][1], alone[key][0])
    assert np.array_equal(alone["Nk"][0], ref["Nk"])


def test_fused_pass_matches_three_passes(lib):
    """N = 64, FP32, all shells: the untuned choice (bits 24: both transforms of the first pass side by side, second and
    last pass fused), and each of its two parts alone, against the three passes (bits 0)."""
    spec = workloads.Spec(N=64, L=1.0, A=1e-2, sigma=0.5, kstar=8 * 2 * np.pi, kind="usr", seed=43)
    with lib.Plan(64, 1.0, precision=32, n_alpha=21) as p:
        p.generate_spec(spec)
        fused = p.spectrum()["omega"][0]
        p.set_tuning(16, 0)
        three = p.spectrum()["omega"][0]
        p.set_tuning(16, 24)
        assert np.array_equal(p.spectrum()["omega"][0], fused)
        for bits in (8, 16):
            p.set_tuning(16, bits)
            np.testing.assert_allclose(p.spectrum()["omega"][0], three, rtol=2e-5)
    np.testing.assert_allclose(fused, three, rtol=2e-5)  # two FP32 evaluations of the same sums


def test_scan_of_more_targets_than_shells(lib):
    """A scan whose targets do not fit one read-back (N = 8 holds four results): the values of one-target scans, and a
    bad target in the middle is refused after the ones before it were written."""
    k = np.geomspace(0.3, 2.5, 11)
    with lib.Plan(8, 1.0, precision=64, n_alpha=5) as p:
        scan = p.target_scan(k, 1e-2, 0.5, 1.0, "local", 2.0, seed=3)
        one = [p.target_scan([x], 1e-2, 0.5, 1.0, "local", 2.0, seed=3) for x in k]
        assert p.L == one[-1]["L"][0]
        with pytest.raises(lib.SigwError) as e:
            p.target_scan([0.5, -1.0, 2.0], 1e-2, 0.5, 1.0)
        assert e.value.status == lib.EINVAL
    for key in ("omega", "L", "n_c"):
        assert np.array_equal(scan[key], np.concatenate([o[key] for o in one]))
