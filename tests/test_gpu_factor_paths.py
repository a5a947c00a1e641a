"""The FP32 factor paths of the bond update at the edges of their tiles.

One Trotter step from a seeded saturated state, FP32 storage against the FP64
mode on the same data, with every site sent to the Householder side of Eq. 10 (in
FP32 storage: the exact Gram) or every site to Cholesky-QR.  Tolerance: the FP32
tensors carry u = 6e-8 per entry and a bond's spectrum moves by at most the
perturbation of its two-site tensor (Weyl), which four updates of sums over two
absorbed sites build up to well under 100 u of the norm; 1e-5 is the bound that the
FP32 parity tests hold.
"""
import numpy as np
import pytest

import paper_2606_30985_gb300 as pkg
from workloads.synthetic import bond_data, site_tensor

pytestmark = pytest.mark.gpu


def spectra(Lx, Ly, chi, precision, n_thresh, scale=1.0):
    cfg = pkg.Config(Lx=Lx, Ly=Ly, J=1.0, h=2.0, dt=0.05, order=2, obs=(0, 0), chi_max=chi, precision=precision,
                     qr_n_thresh=n_thresh, qr_ratio_thresh=0.0)
    eng = pkg.Engine(cfg)
    try:
        bd = bond_data(Lx, Ly, chi)
        eng.set_bonds(0, bd["chi"], bd["lam"], bd["msgs"])
        for v in range(Lx * Ly):
            eng.set_site(0, v, scale * site_tensor(Lx, Ly, chi, 5, v, np.float32, obs=(0, 0)).astype(np.float64))
        eng.trotter_step(1)
        return [eng.spectrum(0, b) for b in range(eng.num_bonds(0))], eng.qr_branch_counts()
    finally:
        eng.close()


# n = 4 chi columns around the 64-wide tiles of the Gram, rows (chi^2, chi^3) around
# its 64-row runs, its splits and the shared-memory limit of the factor
@pytest.mark.parametrize("Lx,Ly,chi", [(2, 2, 1), (3, 3, 3), (3, 3, 16), (3, 3, 17), (2, 4, 33), (2, 2, 41), (4, 1, 128)])
@pytest.mark.parametrize("n_thresh", [10 ** 9, 0])
def test_fp32_factor_paths_match_fp64(Lx, Ly, chi, n_thresh):
    ref, _ = spectra(Lx, Ly, chi, "fp64", 10 ** 9)
    got, count = spectra(Lx, Ly, chi, "fp32", n_thresh)
    assert (count["householder"] > 0) == (n_thresh > 0)
    for a, b in zip(got, ref):
        k = min(len(a), len(b))
        assert np.max(np.abs(a[:k] - b[:k])) < 1e-5
        assert max(np.max(a[k:], initial=0.0), np.max(b[k:], initial=0.0)) < 1e-5


@pytest.mark.parametrize("scale", [1e-14, 1e14])
def test_fp32_factor_is_scale_free(scale):
    # a column's magnitude is divided out before its squares are summed in FP32
    ref, _ = spectra(3, 3, 9, "fp32", 10 ** 9)
    got, _ = spectra(3, 3, 9, "fp32", 10 ** 9, scale)
    for a, b in zip(got, ref):
        assert len(a) == len(b) and np.max(np.abs(a - b)) < 1e-5


def test_nan_site_in_a_tensor_core_step_is_flagged():
    # a NaN coefficient makes its bonds' messages NaN, whose factors have rank 0: the
    # later colours' contractions then have an output leg of size 0
    cfg = pkg.Config(Lx=3, Ly=3, J=1.0, h=2.0, dt=0.05, order=2, obs=(1, 1), chi_max=8, precision="tf32x3")
    eng = pkg.Engine(cfg)
    try:
        eng.trotter_step(2)
        t, _ = eng.site(0, 4)
        t.reshape(-1)[0] = np.nan
        eng.set_site(0, 4, t)
        eng.trotter_step(2)
        eng.bp_converge()
        _, D = eng.correlator()
        assert D[0]["flags"] & 2
    finally:
        eng.close()
