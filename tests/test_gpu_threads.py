"""Contexts on several host threads: the same kernels with windows of different
sizes, launched at the same time, and every run the same as alone."""
import threading

import numpy as np
import pytest

from paper_0810_4737_gb300.workloads import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_0810_4737_gb300 import build, reed
    build.build()
    return reed


@pytest.mark.parametrize("name,windows,repeats", [("as10kev_si_300k_tersoff", (3, 5, 5, 4), 60),
                                                  ("b1kev_si_0k_zbl", (3, 6, 4, 5), 60),
                                                  ("ar30kev_ceo2_300k_buck", (3, 4, 3, 4), 30)])
def test_windows_of_several_sizes(R, name, windows, repeats):
    """(A run that finds its kernel's limit of shared memory lowered by another
    thread fails with REED_E_CUDA.)"""
    def run(n, first):
        w = workload(name, n=n, margin=1 if name.startswith("as") else 0, sigma=0.076, thresholds=[], step_cap=5,
                     damage_n=0)
        with R.Reed(w) as ctx:
            for k in range(first, first + (repeats if first else 1)):
                ctx.reset()
                ctx.run(n_ions=4, seed=9)
                rec = ctx.records()
        return np.sort(rec, order="id").tobytes()

    alone = [run(n, 0) for n in windows]
    got, errors = [None] * len(windows), []

    def work(i):
        try:
            got[i] = run(windows[i], 1)
        except Exception as e:   # reported below
            errors.append((windows[i], e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(windows))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert got == alone
