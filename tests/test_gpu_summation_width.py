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
