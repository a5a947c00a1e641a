"""pepo_launch_count counts every kernel of a launcher that enqueues several.

One BP sweep on the initial state in FP32: the Grams take one launch per band of F
that chi_max reaches (24, 32, 48, 64, 128), and a leg contraction one per 512 items.
"""
import pytest

import paper_2606_30985_gb300 as pkg

pytestmark = pytest.mark.gpu


def sweep_launches(n, Lx, Ly, chi_max):
    cfg = pkg.Config(Lx=Lx, Ly=Ly, J=1.0, h=1.0, dt=0.05, order=1, obs=(0, 0), chi_max=chi_max, precision="fp32", bp_max_sweeps=1)
    eng = pkg.Engine([cfg] * n)
    try:
        before = eng.launches()
        eng.bp_converge()
        return eng.launches() - before
    finally:
        eng.close()


def test_gram_bands_are_counted():
    base = sweep_launches(1, 3, 1, 24)
    for extra, chi_max in enumerate((25, 33, 49, 65), start=1):
        assert sweep_launches(1, 3, 1, chi_max) == base + extra


def test_launches_of_more_than_512_items_are_counted():
    # 16 sites an instance: 512 and 528 items on the first and second legs, fewer on the others
    assert sweep_launches(33, 4, 4, 2) == sweep_launches(32, 4, 4, 2) + 2
