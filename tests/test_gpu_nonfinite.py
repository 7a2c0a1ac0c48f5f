"""A NaN or an infinity in an orbital, or an FP32 overflow, reaches E_x and V_x phi as one on every path,
whatever the passes of the edge are: 30 runtime geometry, 36 and 64 plane passes, 54 one stage at a time."""
import numpy as np
import pytest
import torch

from paper_2309_00651_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [30, 36, 54, 64])
@pytest.mark.parametrize("n_orb", [3, 11])
@pytest.mark.parametrize("what", ["nan", "inf", "overflow"])
def test_not_finite_stays_not_finite(n, n_orb, what):
    from paper_2309_00651_gb300 import hfx
    phi = torch.from_numpy(np.random.default_rng(n).standard_normal((n_orb, n, n, n))).cuda()
    if what == "overflow":
        phi[1] *= 1e25  # the pair (1, 1) is infinite in FP32
    else:
        phi[1, 2, 3, 4] = float(what)
    pairs = torch.from_numpy(I.all_pairs(n_orb)).cuda()
    ex = hfx.Exchange(np.diag([n / 4.0] * 3), (n, n, n), precision="fp32")
    E, V = ex.apply(phi, pairs)
    E_only, _ = ex.apply(phi, pairs, energy_only=True)
    ex.sync_status()
    ex.close()
    assert not np.isfinite(E.item()) and not np.isfinite(E_only.item())
    assert not bool(torch.isfinite(V[1]).any())
    assert not bool(torch.isfinite(V[0]).any())  # from the pair (0, 1)
