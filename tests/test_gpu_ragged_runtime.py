"""The runtime-geometry dense accumulate pass on ragged last blocks, against the generic pass (a block size
without a dense kernel leaves every block pair to it)."""
import numpy as np
import pytest
import torch

from paper_2309_00651_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-6), ("fp64", 1e-12)])
@pytest.mark.parametrize("grid", [(20, 16, 24), (30, 36, 18), (24, 24, 24)])
@pytest.mark.parametrize("block,n_orb", [("8", 9), ("8", 15), ("8", 26), ("4", 7), ("4", 13)])
def test_against_the_generic_pass(precision, tol, grid, block, n_orb, monkeypatch):
    from paper_2309_00651_gb300 import hfx
    rng = np.random.default_rng(sum(grid) + n_orb)
    phi = torch.from_numpy(rng.standard_normal((n_orb,) + grid)).cuda()
    pairs = I.all_pairs(n_orb)
    pairs = torch.from_numpy(np.ascontiguousarray(pairs[rng.random(len(pairs)) < 0.85])).cuda()
    res = []
    for b in (block, "5"):
        monkeypatch.setenv("HFX_BLOCK", b)
        ex = hfx.Exchange(np.diag([g / 3.0 for g in grid]), grid, precision=precision)
        V0 = torch.full_like(phi, 0.25)
        E, V = ex.apply(phi, pairs, accumulate=True, vxphi=V0)
        ex.sync_status()
        res.append((E.item(), V))
        ex.close()
    (Ea, Va), (Eb, Vb) = res
    assert abs(Ea - Eb) <= tol * abs(Eb)
    assert float(torch.linalg.norm(Va - Vb)) <= tol * float(torch.linalg.norm(Vb))
