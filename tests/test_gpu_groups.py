"""Batches that share a launch of the forward and x passes: the same transforms, added into V_x phi in the
same order, as with one launch each (a small transform budget), so V is the same bit for bit."""
import numpy as np
import pytest
import torch

from paper_2309_00651_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_orb", [(48, 48), (64, 26), (72, 20)])
def test_shared_launches_change_nothing(n, n_orb, monkeypatch):
    from paper_2309_00651_gb300 import hfx
    phi = torch.from_numpy(np.random.default_rng(n).standard_normal((n_orb, n, n, n))).cuda()
    pairs = torch.from_numpy(I.all_pairs(n_orb)).cuda()
    res = []
    for mb in ("2048", "40"):
        monkeypatch.setenv("HFX_BATCH_MB", mb)
        ex = hfx.Exchange(np.diag([n / 4.0] * 3), (n, n, n), precision="fp32")
        E, V = ex.apply(phi, pairs)
        ex.sync_status()
        res.append((E.item(), V))
        ex.close()
    assert res[0][0] == res[1][0]
    assert torch.equal(res[0][1], res[1][1])
