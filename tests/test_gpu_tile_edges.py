"""Two BP sweeps at the edges of the tiles of the contraction kernels, against the oracle.

The leg contractions and Grams choose their tiles, and the message eigenproblem its
lanes, from the live bond dimensions.  A chain puts one large dimension on every
bond; a 3x3 grid mixes dimensions, and several of them within one launch.

Tolerance, relative to a message's Frobenius norm: a message is a sum of squares
(no cancellation) of tensors that passed at most three leg contractions, each with
a relative error of a few u = 6e-8 (FP32) or 2^-21 = 5e-7 (three TF32 products),
plus the same from the eigenbasis's orthogonality, twice for two sweeps: below 20 x
5e-7 = 1e-5.  FP64: eigenvalues of a message are floored at 1e-12 of the largest,
which moves a message by at most that; 1e-10.
"""
import numpy as np
import pytest

import paper_2606_30985_gb300 as pkg
from oracle import bp as obp
from oracle.pepo import from_pauli
from workloads.synthetic import bond_list, site_legs, spectrum

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-5, "tf32x3": 1e-5}


def sweep_both(Lx, Ly, chi, chi_max, precision):
    nb = len(bond_list(Lx, Ly))
    rng = np.random.default_rng([Lx, Ly, nb, int(np.sum(chi))])
    lam, msgs = np.zeros((nb, chi_max)), np.zeros((nb, 2, chi_max, chi_max))
    for b in range(nb):
        lam[b, : chi[b]] = spectrum(chi[b])
        for d in range(2):
            msgs[b, d, : chi[b], : chi[b]] = np.diag(spectrum(chi[b]))
    sites = []
    for v in range(Lx * Ly):
        dims = [chi[b] for _, b in site_legs(Lx, Ly, v)]
        t = rng.standard_normal(dims + [4])
        for k, (_, b) in enumerate(site_legs(Lx, Ly, v)):
            t *= np.sqrt(spectrum(chi[b])).reshape([-1 if i == k else 1 for i in range(t.ndim)])
        sites.append(t.astype(np.float32).astype(np.float64))
    cfg = pkg.Config(Lx=Lx, Ly=Ly, J=1.0, h=2.0, dt=0.05, order=2, obs=(0, 0), chi_max=chi_max, precision=precision,
                     bp_alpha=0.7, bp_tol=1e-300, bp_max_sweeps=2)
    eng = pkg.Engine(cfg)
    try:
        eng.set_bonds(0, np.asarray(chi, dtype=np.int32), lam, msgs)
        for v, t in enumerate(sites):
            eng.set_site(0, v, t)
        eng.bp_converge()
        got = eng.get_messages(0).reshape(nb, 2, chi_max, chi_max)
    finally:
        eng.close()
    net = from_pauli(Lx, Ly, (0, 0), "Z", sites, chi, msgs)
    obp.bp_double(net, 0.7, 1e-300, 2)
    worst = 0.0
    for b, (u, v) in enumerate(bond_list(Lx, Ly)):
        for d, key in enumerate([(u, v), (v, u)]):
            ref = net.M[key].real
            worst = max(worst, np.linalg.norm(got[b, d, : chi[b], : chi[b]] - ref) / np.linalg.norm(ref))
    return worst


@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32x3"])
@pytest.mark.parametrize("chi", [1, 8, 9, 16, 17, 24, 25, 32, 33, 48, 49, 64, 65, 97, 128])
def test_chain_of_equal_bonds(chi, precision):
    assert sweep_both(3, 1, [chi] * 2, chi, precision) < TOL[precision]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32x3"])
@pytest.mark.parametrize("chi", [[3, 17, 1, 9, 8, 5, 16, 25, 12, 4, 7, 2], [33, 2, 7, 16, 1, 26, 5, 9, 3, 24, 8, 10]])
def test_grid_of_mixed_bonds(chi, precision):
    assert sweep_both(3, 3, chi, 40, precision) < TOL[precision]
