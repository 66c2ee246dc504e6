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


def _sorted_run(R, w, n, **kw):
    with R.Reed(w) as ctx:
        ctx.run(n_ions=n, seed=7, record_capacity=20000, **kw)
        rec = ctx.records()
        st = ctx.stats()
        damage = ctx.damage_map() if ctx.w["damage_n"] else None
    return rec[np.argsort(rec["id"], kind="stable")], st, damage


@pytest.mark.parametrize("threads", [128, 256])
@pytest.mark.parametrize("name,over", [
    ("b1kev_si_0k_zbl", dict(sigma=0.076, s_loc=0.2, damage_n=16)),
    ("b1kev_si_0k_zbl", dict(n=2, sigma=0.076, rc=4.0, rt=3.5)),
    ("b1kev_si_0k_zbl", dict(n=4, margin=1, sigma=0.076, spline_c=[0.1, -0.1, 0.2, 0.1, 0.0, -0.1])),
    ("u85kev_uo2_300k_recoil", dict(n=3)),
    ("kr85mev_uo2_300k_recoil", dict(n=3))])
def test_a_block_follows_few_tracks(R, name, over, threads):
    """A width of 128 or 256 puts a block of threads on each track while there
    are two tracks per SM (128) or all run at once (256: three blocks per SM),
    and one warp beyond: the tracks are the same, bit for bit, on the two sides of
    the line on 152 SMs."""
    w = workload(name, thresholds=[], step_cap=500, **over)
    line = 304 if threads == 128 else 456
    rec, st, dam = _sorted_run(R, w, line, threads=threads)
    ref, st1, _ = _sorted_run(R, w, line + 1, threads=threads)
    assert st["ctas_per_sm"] < st1["ctas_per_sm"]   # (a block each; one warp each)
    assert rec.tobytes() == ref[:line].tobytes()
    one, st0, _ = _sorted_run(R, w, 1, threads=threads, first_id=line)
    assert one.tobytes() == ref[line:].tobytes()
    for k in ("steps", "pair_evals", "atom_updates", "shifts", "stopped", "truncated", "backscattered"):
        assert st[k] + st0[k] == st1[k], k
    if dam is not None:
        with R.Reed(dict(w)) as ctx:
            ctx.run(n_ions=line, seed=7, threads=64)
            other = ctx.damage_map()   # another width: other roundings, the same tracks to statistics
        assert abs(dam[0].sum() + dam[1] - other[0].sum() - other[1]) < 0.05 * (other[0].sum() + other[1])


def test_a_block_makes_clones(R):
    """Large windows leave room for few tracks per SM, and a width of 256 puts a
    block on each there, cloning depths or not."""
    w = workload("u85kev_uo2_300k_recoil", n=5, energy=2000.0, thresholds=[2.0, 5.0], step_cap=600)
    rec, st, _ = _sorted_run(R, w, 60, threads=256)
    assert st["ctas_per_sm"] * 256 <= 2048
    assert st["clones"] > 60 and st["dropped_clones"] == 0 and st["tracks"] == 60 + st["clones"] == len(rec)
    assert np.sum(np.ldexp(1.0, -rec["level"].astype(int))) == 60
    again, _, _ = _sorted_run(R, w, 60, threads=256)
    assert again.tobytes() == rec.tobytes()
    # a few primaries with cloning depths by blocks, and among many by one warp each
    w = workload("u85kev_uo2_300k_recoil", n=3, energy=2000.0, thresholds=[2.0, 5.0], step_cap=600)
    a, sa, _ = _sorted_run(R, w, 20, threads=256)
    b, sb, _ = _sorted_run(R, w, 200, threads=256)
    assert sa["ctas_per_sm"] < sb["ctas_per_sm"] and sa["clones"] > 20
    assert a.tobytes() == b[b["primary"] < 20].tobytes()
