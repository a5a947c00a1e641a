"""The exact Gram of FP32 storage finds the rank of rank-deficient FP32 data.

Every row of the absorbed matrix cv of a bond's two sites is a power of two times one
of three rows with full mantissas, and every message is the identity, so that in
FP32 cv has rank 3 exactly and its product with the gate's four Schmidt factors rank
12.  With eps_cut = 0 the bond keeps every direction that the factors found, so one
taken from the Gram's rounding shows as a thirteenth.  No tolerance: the rank cut of
1e-14 of the squares stands above the 3e-15 at which the pivots of such Grams end when
every entry is 1e-15 of the paired columns' norms off (twice the Gram's error).
"""
import numpy as np
import pytest

import paper_2606_30985_gb300 as pkg
from workloads.synthetic import bond_list, site_legs, site_tensor

pytestmark = pytest.mark.gpu


def low_rank_site(chi, nenv, seed):
    rng = np.random.default_rng(seed)
    base = rng.standard_normal((3, 4 * chi)).astype(np.float32)
    rows = chi ** nenv
    pick = rng.integers(0, 3, rows)
    pick[:3] = [0, 1, 2]
    scale = np.ldexp(rng.choice([-1.0, 1.0], rows), rng.integers(-3, 1, rows)).astype(np.float32)
    return (base[pick] * scale[:, None]).reshape((chi,) * nenv + (chi, 4))


# rows of cv: 64 (a single run of the Gram, n = 256), 256 and 1024 (several splits)
@pytest.mark.parametrize("Ly,chi", [(2, 64), (3, 16), (3, 32)])
@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
@pytest.mark.parametrize("n_thresh", [10 ** 9, 0])
def test_rank_of_rank_deficient_data(Ly, chi, precision, n_thresh):
    Lx, y = 2, 1 if Ly == 3 else 0
    cfg = pkg.Config(Lx=Lx, Ly=Ly, J=1.0, h=2.0, dt=0.05, order=2, obs=(0, 0), chi_max=chi, eps_cut=0.0,
                     precision=precision, qr_n_thresh=n_thresh, qr_ratio_thresh=0.0)
    nb = len(bond_list(Lx, Ly))
    lam = np.full((nb, chi), chi ** -0.5)
    msgs = np.tile(np.eye(chi), (nb, 2, 1, 1))
    eng = pkg.Engine(cfg)
    try:
        eng.set_bonds(0, np.full(nb, chi, dtype=np.int32), lam, msgs)
        for v in range(Lx * Ly):
            legs = site_legs(Lx, Ly, v)
            if v // Lx == y:
                # legs U, D, then the horizontal one, which colour 0 cuts
                t = low_rank_site(chi, len(legs) - 1, [chi, v])
            else:
                t = site_tensor(Lx, Ly, chi, 5, v, np.float32)
            eng.set_site(0, v, t)
        eng.qr_branch_counts()
        eng.trotter_colour(0)
        assert len(eng.spectrum(0, y)) == 12
        count = eng.qr_branch_counts()
        assert count["householder" if n_thresh else "cholesky_fallback"] >= 2
    finally:
        eng.close()
