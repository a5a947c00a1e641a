"""The branches of Eq. 10 in FP32 storage, each shown to be the one that ran.

Complements test_gpu_factor_paths.py: there every site may be handed back by the trust
test, and the scales are compared on one branch only.  Horizontal bonds of dimension 2
between vertical ones of 16 give the first colour absorbed matrices of 16 rows and 8
columns, none of them rank-deficient, so that Cholesky-QR keeps every site.  One colour
against FP64 on the same data: the bound of that file, 1e-5 of the norm.
"""
import numpy as np
import pytest

import paper_2606_30985_gb300 as pkg
from workloads.synthetic import bond_list, site_legs, spectrum

pytestmark = pytest.mark.gpu


def one_colour(precision, n_thresh, scale):
    Lx = Ly = 2
    cm = 16
    chi = np.array([2, 2, 16, 16], dtype=np.int32)
    nb = len(bond_list(Lx, Ly))
    lam, msgs = np.zeros((nb, cm)), np.zeros((nb, 2, cm, cm))
    for b in range(nb):
        lam[b, : chi[b]] = spectrum(chi[b])
        for d in range(2):
            msgs[b, d, : chi[b], : chi[b]] = np.diag(spectrum(chi[b]))
    cfg = pkg.Config(Lx=Lx, Ly=Ly, J=1.0, h=2.0, dt=0.05, order=2, obs=(0, 0), chi_max=cm, precision=precision,
                     qr_n_thresh=n_thresh, qr_ratio_thresh=0.0)
    eng = pkg.Engine(cfg)
    try:
        eng.set_bonds(0, chi, lam, msgs)
        for v in range(4):
            dims = [chi[b] for _, b in site_legs(Lx, Ly, v)]
            t = np.random.default_rng([7, v]).standard_normal(dims + [4]).astype(np.float32)
            eng.set_site(0, v, scale * t.astype(np.float64))
        eng.qr_branch_counts()
        eng.trotter_colour(0)
        return [eng.spectrum(0, b) for b in range(2)], eng.qr_branch_counts()
    finally:
        eng.close()


@pytest.mark.parametrize("scale", [1e-14, 1.0, 1e14])
@pytest.mark.parametrize("n_thresh,branch", [(0, "cholesky"), (10 ** 9, "householder")])
def test_each_branch_at_each_scale(n_thresh, branch, scale):
    ref, _ = one_colour("fp64", 10 ** 9, 1.0)
    got, count = one_colour("fp32", n_thresh, scale)
    assert count == {"householder": 0, "cholesky": 0, "cholesky_fallback": 0, branch: 4}
    for a, b in zip(got, ref):
        assert len(a) == len(b) and np.max(np.abs(a - b)) < 1e-5


@pytest.mark.parametrize("precision,rows,tol", [("fp64", 512, 1e-12), ("fp32", 2048, 1e-6)])
def test_splits_that_differ_change_only_rounding(precision, rows, tol):
    # chi 16 on an interior site sums 4 chi^3 products: several splits of `rows` each,
    # in both engines, and not as many
    cfg = pkg.Config(Lx=4, Ly=4, J=1.0, h=1.5, dt=0.05, order=2, obs=(1, 1), chi_max=16, precision=precision)
    out = []
    for tuning in (None, {"gram_leg_splits": 3, "gram_rows_splits": 5}):
        eng = pkg.Engine(cfg, tuning=tuning)
        try:
            recs = eng.run(5)
            chi = [len(eng.spectrum(0, b)) for b in range(eng.num_bonds(0))]
            out.append((np.array([r["C"] for r in recs]), min(eng.get_tuning()["gram_leg_splits"], 4 * max(chi) ** 3 // rows)))
        finally:
            eng.close()
    (Ca, sa), (Cb, sb) = out
    assert sa > sb > 1
    assert np.max(np.abs(Ca - Cb)) < tol
