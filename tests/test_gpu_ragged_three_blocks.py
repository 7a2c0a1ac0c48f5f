"""Three orbital blocks with a ragged last one on runtime-geometry grids, on both sides of the size from which
the dense pass takes the ragged block's pairs, against the generic pass alone (a block size without a dense
kernel)."""
import numpy as np
import pytest
import torch

from paper_2309_00651_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-6), ("fp64", 1e-12)])
@pytest.mark.parametrize("grid", [(8, 8, 8), (10, 12, 8), (18, 18, 24), (20, 20, 20), (30, 18, 16)])
@pytest.mark.parametrize("block,n_orb", [("8", 17), ("8", 20), ("8", 23), ("4", 9), ("4", 11)])
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
        E, V = ex.apply(phi, pairs)
        ex.sync_status()
        res.append((E.item(), V))
        ex.close()
    (Ea, Va), (Eb, Vb) = res
    assert abs(Ea - Eb) <= tol * abs(Eb)
    assert float(torch.linalg.norm(Va - Vb)) <= tol * float(torch.linalg.norm(Vb))
