"""The ion-target-only stepper (one warp per track) against the oracle, over
the window sizes, frozen margins and summation widths it accepts.

Windows smaller than a warp's pass, with remainders and larger than every
summation width; with a frozen layer (listed but never kicked) and without;
surface and bulk targets.  First steps of each track: 1e-4 A in the mixed form
(as for the other traces) and 1e-9 A in the FP64 form, where 100 steps grow a
rounding of 1e-15 A by less than a million in a thermal crystal.
"""
import numpy as np
import pytest

from paper_0810_4737_gb300.workloads import workload

pytestmark = pytest.mark.gpu

STEPS = 100


@pytest.fixture(scope="module")
def R():
    from paper_0810_4737_gb300 import build, reed
    build.build()
    return reed


@pytest.mark.parametrize("name,n,margin", [("b1kev_si_0k_zbl", 2, 0), ("b1kev_si_0k_zbl", 3, 1),
                                           ("b1kev_si_0k_zbl", 4, 1), ("b1kev_si_0k_zbl", 5, 0),
                                           ("u85kev_uo2_300k_recoil", 3, 0), ("u85kev_uo2_300k_recoil", 4, 1)])
@pytest.mark.parametrize("threads", [32, 64, 256])
@pytest.mark.parametrize("prec", [0, 1])
def test_windows_and_summation_widths(R, O, name, n, margin, threads, prec):
    w = workload(name, n=n, margin=margin, sigma=0.076, thresholds=[], s_loc=0.1)
    p = O.params(w)
    with R.Reed(w) as ctx:
        ctx.run(n_ions=3, seed=11, precision=prec, threads=threads, trace_tracks=3, trace_steps=STEPS, step_cap=STEPS)
        traj, anchors = ctx.trace(3, STEPS)
        rec = ctx.records()
    assert sorted(rec["id"]) == [0, 1, 2] and np.all(rec["steps"] == STEPS)
    for t in range(3):
        ref, ref_anchors = O.trace(p, 11, t, STEPS)
        k = ref.shape[0]
        assert k == STEPS
        np.testing.assert_allclose(traj[t, :, :3], ref[:, :3], rtol=0, atol=1e-9 if prec else 1e-4)
        assert np.array_equal(anchors[t], ref_anchors)


def test_density_of_atoms_without_a_force(R, O):
    """A correction exp(c) that underflows in FP32 leaves the pair terms zero and
    the local density as it is: atoms that the ion has left behind must not stay
    in it.  (Long density range and a steep taper, so that an atom's weight is
    still large when it leaves the cutoff.)  The drag on a straight flight through
    20 A: velocities to 1e-5, some hundred FP32 roundings; the drag changes them
    by more than 1e-2."""
    w = workload("b1kev_si_0k_zbl", sigma=0.076, spline_c=[-2000.0] * 6, s_loc=1.0, lam_loc=5.0, rt=4.9, s_e=20.0)
    p = O.params(w)
    steps = 400
    with R.Reed(w) as ctx:
        ctx.run(n_ions=2, seed=11, trace_tracks=2, trace_steps=steps, step_cap=steps)
        traj, _ = ctx.trace(2, steps)
    for t in range(2):
        ref, _ = O.trace(p, 11, t, steps)
        assert abs(ref[-1, 6] / ref[0, 6] - 1) > 1e-2
        np.testing.assert_allclose(traj[t, :, 4:7], ref[:, 4:7], rtol=1e-5, atol=0)
