"""The TMA dense accumulate pass on ragged last blocks and on block pairs with few or no listed pairs,
against the generic pass (HFX_DENSE_TMA=0 leaves ragged blocks to it) on the same inputs."""
import numpy as np
import pytest
import torch

from paper_2309_00651_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_orb", [(32, 9), (32, 15), (48, 17), (72, 23), (80, 12), (96, 11)])
@pytest.mark.parametrize("lists", ["all", "rows", "few"])
def test_against_the_generic_pass(n, n_orb, lists, monkeypatch):
    from paper_2309_00651_gb300 import hfx
    rng = np.random.default_rng(n * 100 + n_orb)
    phi = torch.from_numpy(rng.standard_normal((n_orb, n, n, n))).cuda()
    pairs = I.all_pairs(n_orb)
    if lists == "rows":    # whole orbitals without partners outside their own block: rows of couples without pairs
        off = pairs[:, 0] // 8 != pairs[:, 1] // 8
        pairs = pairs[~off | ((pairs[:, 0] % 3 != 0) & (pairs[:, 1] % 4 != 1))]
    elif lists == "few":   # a handful of pairs: most block pairs empty
        pairs = pairs[np.sort(rng.permutation(len(pairs))[:4])]
    pairs = torch.from_numpy(np.ascontiguousarray(pairs)).cuda()
    res = []
    for tma in ("1", "0"):
        monkeypatch.setenv("HFX_DENSE_TMA", tma)
        ex = hfx.Exchange(np.diag([n / 4.0] * 3), (n, n, n), precision="fp32")
        ex.ensure_workspace(n_orb, len(pairs))
        ex._ws.fill_(0xFF)  # NaN in every transform that no pass writes
        hfx.hfx_set_workspace(ex.ctx, ex._ws)
        E, V = ex.apply(phi, pairs)
        ex.sync_status()
        res.append((E.item(), V))
        ex.close()
    (Ea, Va), (Eb, Vb) = res
    # which two pairs share a transform differs, and with it the rounding: the path's stated 1e-6
    assert abs(Ea - Eb) <= 1e-6 * abs(Eb)
    assert float(torch.linalg.norm(Va - Vb)) <= 1e-6 * float(torch.linalg.norm(Vb))
