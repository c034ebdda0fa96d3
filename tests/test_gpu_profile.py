"""Kernel-class counts and times of a cell: every class of an iteration is
reported, the error reduction included, although it has no launch of its own."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", [0, 1])
def test_reduction_is_counted_and_timed(precision):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_10774_gb300 as M
    rve = M.Rve(M.Context(0), W.workload_centered_sphere(ref_kind="midrange", tol=1e-6), precision=precision)
    for profile in (False, True):  # the loop decided on the device, then on the host
        rve.reset()
        rve.profile(profile)
        rve.profile_read(reset=True)
        assert rve.run(2) == 0
        prof = rve.profile_read()
        its = rve.iterations
        assert prof["pass_a"][1] == its and prof["reduce"][1] == its
        assert (prof["reduce"][0] > 0.0) == profile
        # a few microseconds of pass A's some twenty
        assert 0.0 <= prof["reduce"][0] < (prof["pass_a"][0] if profile else 1e-9)
    rve.close()
