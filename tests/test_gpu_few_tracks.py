"""A run with no more tracks than SMs (or other processors' worth of CTAs) is
launched in another shape than a large batch: every track must come out the
same, bit for bit, for each number of tracks around the places where the shape
changes.
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


def _records(R, w, n, prec, **kw):
    with R.Reed(w) as ctx:
        ctx.run(n_ions=n, seed=11, precision=prec, **kw)
        rec = ctx.records()
        st = ctx.stats()
        damage = ctx.damage_map() if ctx.w["damage_n"] else None
    return rec[np.argsort(rec["id"], kind="stable")], st, damage


@pytest.mark.parametrize("name,prec,steps,few", [
    ("as10kev_si_300k_tersoff", 0, 400, (1, 5, 76, 152, 153, 304)),
    ("as10kev_si_300k_tersoff", 1, 120, (1, 5, 20, 39, 77, 152)),
    ("ar30kev_ceo2_300k_buck", 0, 150, (1, 5, 39, 77, 152)),
    ("ar30kev_ceo2_300k_buck", 1, 40, (1, 5, 77)),
    ("b1kev_si_0k_zbl", 0, 500, (1, 5, 153)),
    ("b1kev_si_0k_zbl", 1, 200, (1, 153))])
def test_tracks_do_not_depend_on_the_launch_shape(R, name, prec, steps, few):
    w = workload(name, thresholds=[], step_cap=steps)
    ref, _, _ = _records(R, w, 330, prec)
    for n in few:
        rec, st, _ = _records(R, w, n, prec)
        assert st["tracks"] == st["primaries"] == n
        assert rec.tobytes() == ref[:n].tobytes(), n


def test_low_energy_tracks_to_their_end(R):
    """Whole tracks with window moves, cascades and list refreshes."""
    w = workload("as10kev_si_300k_tersoff", thresholds=[], energy=300.0)
    ref, _, _ = _records(R, w, 200, 0)
    rec, _, _ = _records(R, w, 9, 0)
    assert rec.tobytes() == ref[:9].tobytes()
    w = workload("as10kev_si_300k_tersoff", thresholds=[], energy=60.0)
    ref, _, _ = _records(R, w, 160, 1)
    rec, _, _ = _records(R, w, 9, 1)
    assert rec.tobytes() == ref[:9].tobytes()


def test_damage_of_a_single_track_is_deposited_once(R):
    w = workload("ar30kev_ceo2_300k_buck", thresholds=[], energy=1000.0, step_cap=400)
    a, _, da = _records(R, w, 1, 0)
    b, _, db = _records(R, w, 1, 0, ctas_per_sm=1)
    assert a.tobytes() == b.tobytes() and np.allclose(da[0], db[0], rtol=1e-12, atol=0)


def test_first_epoch_of_an_adaptive_run(R):
    """Launched inside a captured graph, without cloning and with few tracks."""
    w = workload("as10kev_si_300k_tersoff", energy=500.0, thresholds=[], step_cap=600)
    ref, _, _ = _records(R, w, 20, 0)
    w = workload("as10kev_si_300k_tersoff", energy=500.0, thresholds=[15.0, 30.0], step_cap=600)
    rec, st, _ = _records(R, w, 50, 0, adaptive=True, n_initial=20, epoch_size=30, record_capacity=4000)
    assert st["primaries"] == 50
    assert rec[:20].tobytes() == ref.tobytes()


@pytest.mark.parametrize("name,prec,thresholds,grids", [
    # Tersoff: clusters of SMs on a few tracks, then a CTA for each, then two per SM
    ("as10kev_si_300k_tersoff", 0, [], {1: (2, 4, 8), 31: (2, 4), 63: (2,), 64: (1,), 152: (1,), 304: (1,)}),
    ("as10kev_si_300k_tersoff", 1, [], {1: (2, 4, 8), 31: (2, 4), 63: (2,), 64: (1,), 152: (1,)}),
    ("ar30kev_ceo2_300k_buck", 0, [], {1: (1,), 152: (1,)}),
    ("b1kev_si_0k_zbl", 0, [], {1: (1,), 153: (1,)}),
    # with a cloning depth every CTA that fits is launched
    ("as10kev_si_300k_tersoff", 0, [1e6], {5: None}),
    ("b1kev_si_0k_zbl", 0, [1e6], {5: None})])
def test_statistics_tell_the_ctas_launched(R, name, prec, thresholds, grids):
    """(On 152 SMs, the count that the lines between the shapes are tested for.)"""
    w = workload(name, thresholds=thresholds, step_cap=20)
    for n, per_track in grids.items():
        _, st, _ = _records(R, w, n, prec)
        if per_track is None:
            assert st["grid"] == 152 * st["ctas_per_sm"]
        else:
            assert st["grid"] % n == 0 and st["grid"] // n in per_track, (n, st["grid"])
    if name.startswith("as10kev") and prec == 0 and not thresholds:
        _, st, _ = _records(R, w, 305, prec)
        assert st["grid"] == 304


def test_a_team_has_four_sms_at_most(R):
    w = workload("as10kev_si_300k_tersoff", thresholds=[], step_cap=20)
    for prec in (0, 1):
        for n in (1, 7, 15, 31):
            _, st, _ = _records(R, w, n, prec)
            assert st["grid"] == 4 * n


@pytest.mark.parametrize("n,margin,prec,team", [
    (2, 0, 0, False), (3, 0, 0, False), (3, 1, 0, False), (4, 1, 0, False), (5, 2, 0, False), (5, 1, 0, True),
    (6, 1, 0, True), (3, 0, 1, True), (4, 1, 1, False), (5, 1, 1, True)])
def test_teams_where_there_are_many_centres(R, n, margin, prec, team):
    """Small windows, and in the mixed form windows without a frozen layer, get no
    teams; the tracks are those of the batch launch (which a cloning depth out of
    reach selects) in every shape."""
    w = workload("as10kev_si_300k_tersoff", n=n, margin=margin, thresholds=[], energy=300.0, step_cap=120 if prec else 300)
    rec, st, _ = _records(R, w, 7, prec)
    assert st["grid"] == (28 if team else 7)
    ref, st1, _ = _records(R, dict(w, thresholds=[1e6]), 7, prec)
    assert st1["grid"] % 152 == 0
    assert rec.tobytes() == ref.tobytes()
    for k in ("steps", "pair_evals", "bond_evals", "triplets", "atom_updates", "shifts"):
        assert st[k] == st1[k], k
