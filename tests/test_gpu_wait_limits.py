"""The bounded waits of every pass that waits for bulk copies: with a one-cycle limit they give up while every copy still
lands, the error names each pass that gave up, and with the default limit the plan gives the bits it gave before."""
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


# the second pass with a field per CTA (up to 32^3), with its stash in shared memory (FP64, and FP32 at 64^3), with its stash in
# tensor memory; the last pass with its accumulators in registers (radix 8 and 16) and in tensor memory; both in one kernel
@pytest.mark.parametrize("N,precision,bits,passes", [
    (8, 32, 0, ("second", "last")), (32, 32, 0, ("second", "last")), (32, 64, 0, ("second", "last")),
    (64, 64, 0, ("second", "last")), (64, 32, 0, ("second", "last")), (64, 32, 24, ("fused second and last",)),
    (128, 32, 2, ("second", "last")), (128, 32, 26, ("second", "last")), (256, 32, 26, ("second", "last"))])
@pytest.mark.parametrize("n_alpha", [6, 7])
def test_waits_that_give_up_are_named_and_recoverable(lib, N, precision, bits, passes, n_alpha):
    spec = workloads.Spec(N=N, L=1.0, A=1e-2, sigma=0.5, kstar=max(2, N // 8) * 2 * np.pi, kind="local", F_NL=2.0, seed=31)
    shells = [2, N // 4, N // 2]
    with lib.Plan(N, 1.0, precision=precision, n_alpha=n_alpha) as p:
        p.set_tuning(n_alpha, bits)
        p.generate_spec(spec)
        clean = p.spectrum(shells)["omega"][0]
        p.debug_wait_limit(1)
        with pytest.raises(lib.SigwError) as e:
            p.spectrum(shells)
        assert e.value.status == lib.ETIMEOUT
        assert "(inverse passes: %s)" % ", ".join(passes) in str(e.value)
        p.debug_wait_limit(0)
        assert np.array_equal(p.spectrum(shells)["omega"][0], clean)
