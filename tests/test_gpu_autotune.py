"""The autotuner times launches that differ: CTAs per SM only where they change
the launch of the trial tracks, and the occupancy maximum is kept as no limit."""
import pytest

from paper_0810_4737_gb300.workloads import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_0810_4737_gb300 import build, reed
    build.build()
    return reed


def test_fewer_tracks_than_half_the_gpu_holds(R):
    """600 one-warp tracks are the same launch at 16, 12 and 8 CTAs per SM."""
    w = workload("b1kev_si_0k_zbl", sigma=0.076, rot=(0.0, 45.0))
    with R.Reed(w) as ctx:
        tab = ctx.autotune(n_trial=600, seed=11, step_cap=100)
        assert [t for t, _, _ in tab] == [32, 64, 128, 256]
        # ... and a run that fills the GPU gets every CTA that fits
        ctx.run(n_ions=3000, seed=2)
        st = ctx.stats()
        with R.Reed(w) as other:
            other.run(n_ions=3000, seed=2, threads=st["threads_per_track"])
            most = other.stats()
    assert (st["ctas_per_sm"], st["grid"]) == (most["ctas_per_sm"], most["grid"])


def test_more_tracks_than_the_gpu_holds(R):
    w = workload("b1kev_si_0k_zbl", sigma=0.076, rot=(0.0, 45.0))
    with R.Reed(w) as ctx:
        tab = ctx.autotune(n_trial=3000, seed=11, step_cap=50)
    by = {}
    for t, c, v in tab:
        assert v > 0
        by.setdefault(t, []).append(c)
    assert sorted(by) == [32, 64, 128, 256]
    for c in by.values():
        assert len(set(c)) == len(c) == 3 and c[0] == max(c)


def test_tersoff_trials(R):
    """Two tracks fit on an SM: one per SM is another launch for more tracks than
    SMs only."""
    w = workload("as10kev_si_300k_tersoff", thresholds=[])
    with R.Reed(w) as ctx:
        few = ctx.autotune(n_trial=40, seed=11, step_cap=20)
        many = ctx.autotune(n_trial=320, seed=11, step_cap=20)
    assert [c for _, c, _ in few] == [2] * 4
    assert sorted((t, c) for t, c, _ in many) == [(t, c) for t in (32, 64, 128, 256) for c in (1, 2)]
