"""An expired pipeline wait drops the flags of the aborted call only.

The kernels behind an aborted one raise flags on its unwritten results; a flag that
an earlier call raised on any instance of the context is still reported after the
error.
"""
import numpy as np
import pytest

import paper_2606_30985_gb300 as pkg

pytestmark = pytest.mark.gpu


def test_earlier_flags_survive_an_expired_wait():
    import torch
    cfg = dict(Lx=3, Ly=3, J=1.0, h=1.0, dt=0.05, order=1, chi_max=8, precision="tf32x3")
    eng = pkg.Engine([pkg.Config(**cfg), pkg.Config(**cfg)])

    def layer():
        eng.trotter_step(1)
        eng.bp_converge()
        return [d["flags"] & 2 for d in eng.correlator()[1]]

    try:
        eng.trotter_step(2)
        snaps = [torch.empty(eng.state_bytes(i), dtype=torch.uint8, device="cuda:0") for i in range(2)]
        for i, s in enumerate(snaps):
            eng.save_state(s, i)
        t, _ = eng.site(0, 4)
        t = np.array(t)
        t.flat[0] = np.nan
        eng.set_site(0, 4, t)
        assert layer() == [2, 0]                 # a non-finite coefficient on instance 0
        for i, s in enumerate(snaps):
            eng.load_state(s, i)
        eng.set_wait_limit(1e-9)
        with pytest.raises(pkg.PepoError, match="wait limit"):
            for _ in range(3):
                layer()
        eng.set_wait_limit(4.0)
        for i, s in enumerate(snaps):
            eng.load_state(s, i)
        assert layer() == [2, 0]
    finally:
        eng.close()
