"""A track's roundings are written out where the compiler could fuse a sum in
more than one way, so that its bits are those of every earlier kernel.

Depth and time of five FP64 As tracks after 800 steps (several window moves), as
the stepper gave them before the ion's update was rewritten.  A rounding of
1e-16 in the ion's place in the window, taken at each move, is some 1e-14 A by
then, far below every physical tolerance: only the bits can tell.
"""
import numpy as np
import pytest

from paper_0810_4737_gb300.workloads import workload

pytestmark = pytest.mark.gpu

Z = ["0x1.160de81d2e442p+5", "0x1.15fdeb42c0beap+5", "0x1.afb87285cfc81p+4", "0x1.0e477bd86bddbp+5",
     "0x1.0fa3b0beb3d4ap+5"]
T = ["0x1.3fde0c769c946p+1", "0x1.4884f4a881429p+1", "0x1.80b9040c6d9f1p+1", "0x1.73e343ea75b03p+1",
     "0x1.55359ed229579p+1"]


def test_fp64_tracks_across_window_moves():
    from paper_0810_4737_gb300 import build, reed as R
    build.build()
    w = workload("as10kev_si_300k_tersoff", step_cap=800)
    with R.Reed(w) as ctx:
        ctx.run(n_ions=5, seed=3, precision=R.PREC_FP64)
        rec = ctx.records()
        assert ctx.stats()["shifts"] > 5
    rec = rec[np.argsort(rec["id"])]
    assert [float(x).hex() for x in rec["z"]] == Z
    assert [float(x).hex() for x in rec["t"]] == T
