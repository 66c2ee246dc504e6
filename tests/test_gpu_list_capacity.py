"""Rows of the Tersoff list table: a cascade that makes more frozen atoms needed
than a perfect window has, plus a quarter, must not fail the run.

Primary 122730 (seed 0) of the 10 keV As batch throws enough atoms into the
frozen layer to need two rows more than that estimate; the table has the shared
memory that its launch leaves unused.
"""
import numpy as np
import pytest

from paper_0810_4737_gb300.workloads import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_0810_4737_gb300 import build, reed
    build.build()
    return reed


def test_a_cascade_in_the_frozen_layer(R):
    w = workload("as10kev_si_300k_tersoff")
    recs = []
    # a team of SMs, and the batch kernel (chosen because of a depth that no track reaches)
    for thresholds in ([], [1e6]):
        with R.Reed(w) as ctx:
            ctx.run(n_ions=1, seed=0, first_id=122730, thresholds=thresholds)
            recs.append(ctx.records())
            st = ctx.stats()
        assert st["bond_cap_overflow"] == st["nb_overflow"] == 0
        assert len(recs[-1]) == 1 and recs[-1]["status"][0] == R.STOPPED
    assert recs[0].tobytes() == recs[1].tobytes()


@pytest.mark.parametrize("n,margin", [(3, 1), (4, 1), (5, 1), (5, 2), (6, 2)])
@pytest.mark.parametrize("prec", [0, 1])
def test_lists_of_other_windows(R, n, margin, prec):
    """Exact lists (self-check) whatever room the table finds."""
    w = workload("as10kev_si_300k_tersoff", n=n, margin=margin, thresholds=[], energy=500.0, step_cap=150)
    with R.Reed(w) as ctx:
        try:
            ctx.run(n_ions=6, seed=4, precision=prec, nl_check=True)
        except R.ReedError as e:
            assert e.code == R.E_SMEM and prec == 1 and n == 6   # (a window that FP64 has no room for)
            return
        st = ctx.stats()
    assert st["tracks"] == 6 and st["steps"] <= 900 and st["nl_check_errors"] == 0
    assert st["bond_cap_overflow"] == st["nb_overflow"] == 0
