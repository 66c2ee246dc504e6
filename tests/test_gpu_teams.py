"""Tersoff tracks followed by a team of SMs against the same tracks by one CTA
each (a cloning depth that no track reaches selects the batch launch): what only
the leader of a team may do, and what a team's members write into one another's
windows.
"""
import numpy as np
import pytest

from paper_0810_4737_gb300.workloads import workload

pytestmark = pytest.mark.gpu

COUNTERS = ("primaries", "tracks", "steps", "pair_evals", "bond_evals", "triplets", "atom_updates", "shifts", "rebuilds",
            "list_refreshes", "nb_spilled", "centre_class", "stopped", "backscattered", "truncated")


@pytest.fixture(scope="module")
def R():
    from paper_0810_4737_gb300 import build, reed
    build.build()
    return reed


def _run(R, w, n, prec, thresholds, **kw):
    with R.Reed(w) as ctx:
        ctx.run(n_ions=n, precision=prec, thresholds=thresholds, **kw)
        rec = ctx.records()
        st = ctx.stats()
        damage = ctx.damage_map() if ctx.w["damage_n"] else None
    return rec[np.argsort(rec["id"], kind="stable")], st, damage


def _both(R, w, n, prec, **kw):
    team, st, dam = _run(R, w, n, prec, [], **kw)
    one, st1, dam1 = _run(R, w, n, prec, [1e6], **kw)
    assert st["grid"] in (2 * n, 4 * n) and st1["grid"] % 152 == 0   # both shapes were launched
    assert team.tobytes() == one.tobytes()
    for k in COUNTERS:
        assert st[k] == st1[k], k
    return st, dam, dam1


@pytest.mark.parametrize("prec,n,steps", [(0, 1, 1500), (0, 7, 600), (0, 39, 400), (1, 5, 300)])
def test_damage_and_counters(R, prec, n, steps):
    """Each atom's energy is deposited once, by the leader (a map's sums differ by
    the order of the atomics: 1e-12 of a voxel with up to some thousand
    deposits)."""
    w = workload("as10kev_si_300k_tersoff", energy=2000.0, step_cap=steps, damage_n=32)
    st, dam, one = _both(R, w, n, prec, seed=11)
    assert st["shifts"] > 0 and one[0].sum() > 0
    np.testing.assert_allclose(dam[0], one[0], rtol=1e-12, atol=0)
    np.testing.assert_allclose(dam[1], one[1], rtol=1e-12, atol=1e-300)


@pytest.mark.parametrize("prec", [0, 1])
def test_overflow_rows_of_every_member(R, prec):
    """Lists of more than twelve entries: their forces go into overflow rows of
    each member's block.  (A skin of 0.82 A reaches the nearest of the thermally
    displaced second neighbours: some three atoms of a window have more than
    twelve within 3.82 A.)"""
    w = workload("as10kev_si_300k_tersoff", energy=500.0, step_cap=250)
    st, _, _ = _both(R, w, 6, prec, seed=11, nl_skin=0.82)
    assert st["nb_spilled"] > 0


def test_overflow_rows_in_a_cascade(R):
    """A whole 10 keV track whose cascade fills overflow rows between window
    moves."""
    w = workload("as10kev_si_300k_tersoff")
    st, _, _ = _both(R, w, 1, 0, seed=0, first_id=2083)
    assert st["nb_spilled"] > 0
