"""Tracks with target-target forces whose CTA has another number of threads
than threads_per_track: the sums over atoms are then taken by virtual threads.

First steps of each track against the oracle (1e-4 A mixed, 1e-9 A FP64: 50
steps grow a rounding of 1e-15 A by far less than a million), with frozen atoms
(their pair terms are summed after those of the integrated ones) and without,
for widths below, at and above the CTA's own.
"""
import numpy as np
import pytest

from paper_0810_4737_gb300.workloads import workload

pytestmark = pytest.mark.gpu

STEPS = 50


@pytest.fixture(scope="module")
def R():
    from paper_0810_4737_gb300 import build, reed
    build.build()
    return reed


@pytest.mark.parametrize("name,n,margin,threads", [("as10kev_si_300k_tersoff", 4, 1, (32, 128, 256)),
                                                   ("as10kev_si_300k_tersoff", 3, 0, (64, 256)),
                                                   ("ar30kev_ceo2_300k_buck", 3, 0, (32, 256, 512)),
                                                   ("ar30kev_ceo2_300k_buck", 4, 1, (64, 512))])
@pytest.mark.parametrize("prec", [0, 1])
def test_widths(R, O, name, n, margin, threads, prec):
    w = workload(name, n=n, margin=margin, s_loc=0.1)
    p = O.params(w)
    ref = [O.trace(p, 5, t, STEPS) for t in range(2)]
    for width in threads:
        with R.Reed(w) as ctx:
            ctx.run(n_ions=2, seed=5, precision=prec, threads=width, trace_tracks=2, trace_steps=STEPS, step_cap=STEPS,
                    damage=False)
            traj, anchors = ctx.trace(2, STEPS)
            st = ctx.stats()
        assert st["threads_per_track"] == width and st["steps"] == 2 * STEPS
        for t in range(2):
            np.testing.assert_allclose(traj[t, :, :3], ref[t][0][:, :3], rtol=0, atol=1e-9 if prec else 1e-4)
            assert np.array_equal(anchors[t], ref[t][1])


@pytest.mark.parametrize("name,n,margin,threads,tracks", [("as10kev_si_300k_tersoff", 3, 1, (32, 64, 128), 300),
                                                          ("as10kev_si_300k_tersoff", 2, 0, (32, 128), 300),
                                                          ("ar30kev_ceo2_300k_buck", 3, 1, (32, 64, 128), 700)])
def test_narrow_ctas_of_many_fp64_tracks(R, name, n, margin, threads, tracks):
    """More FP64 tracks than wide CTAs fit get CTAs as narrow as their sums: more
    per SM, and the same bits as the few that get wide ones.  (200 steps, past the
    surface: the window's integrated atoms lie above it before.)"""
    w = workload(name, n=n, margin=margin, thresholds=[], step_cap=200, damage_n=0)
    for width in threads:
        recs, per_sm = [], []
        for k in (tracks, 5):
            with R.Reed(w) as ctx:
                ctx.run(n_ions=k, seed=5, precision=1, threads=width)
                rec = ctx.records()
                st = ctx.stats()
            recs.append(rec[np.argsort(rec["id"], kind="stable")])
            per_sm.append(st["ctas_per_sm"])
            assert st["tracks"] == k and st["steps"] == rec["steps"].sum() and st["pair_evals"] > 0 and st["bond_evals"] > 0
        assert per_sm[0] > per_sm[1]
        assert recs[0][:5].tobytes() == recs[1].tobytes()
