"""The compile-time forward and x passes of every edge against the FP64 path of the same library (itself
within 1e-8 of the oracle), with couples that hold no pair, one pair and two."""
import numpy as np
import pytest
import torch

from paper_2309_00651_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 48, 64, 72, 80, 96, 128])
@pytest.mark.parametrize("n_orb,share", [(8, 1.0), (3, 1.0), (10, 0.4)])
def test_edges_against_the_fp64_path(n, n_orb, share):
    from paper_2309_00651_gb300 import hfx
    L = n / 4.0
    raw = I.gaussian_orbitals(n_orb, L, n, 40.0, 1.2, seed=n + n_orb)
    phi = torch.from_numpy(raw).cuda()
    pairs = I.all_pairs(n_orb)
    if share < 1.0:
        pairs = pairs[np.sort(np.random.default_rng(n).permutation(len(pairs))[: int(share * len(pairs))])]
    pairs = torch.from_numpy(np.ascontiguousarray(pairs)).cuda()
    res = {}
    for prec in ("fp64", "fp32"):
        ex = hfx.Exchange(np.diag([L] * 3), (n, n, n), precision=prec)
        E, V = ex.apply(phi, pairs)
        E_only, _ = ex.apply(phi, pairs, energy_only=True)
        ex.sync_status()
        assert abs(E_only.item() - E.item()) <= 1e-12 * abs(E.item())
        res[prec] = (E.item(), V)
        ex.close()
    (E64, V64), (E32, V32) = res["fp64"], res["fp32"]
    # the mixed path's stated error: 1e-6 relative, in E and in the norm of V
    assert abs(E32 - E64) <= 1e-6 * abs(E64)
    assert float(torch.linalg.norm(V32 - V64)) <= 1e-6 * float(torch.linalg.norm(V64))
