"""The residual update of the SCDM localisation at orbital counts around the groups of rows it takes at once
(64, 32, 16 and 8 in FP32, 8, 4, 2 and 1 in FP64), on a grid of one round and, for FP32, one of several:
picks against the FP64 residual norms, Q and Phi against the oracle's for those picks, and the same bits
when the call is replayed from a CUDA graph."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ace_oracle as A  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-8, "fp32": 1e-6}  # of the ACE and SCDM parity tests


@pytest.mark.parametrize("precision,n_orb,n", [("fp32", k, 16) for k in (1, 7, 8, 15, 17, 31, 33, 63, 65, 71, 97, 127)]
                         + [("fp64", k, 16) for k in (1, 3, 7, 9, 15)] + [("fp32", 47, 72)])
def test_rows_left_over(precision, n_orb, n):
    from paper_2309_00651_gb300 import hfx
    L = n / 3.9
    phi = np.random.default_rng(n_orb).standard_normal((n_orb, n, n, n))
    q, _ = np.linalg.qr(phi.reshape(n_orb, -1).T)
    phi = np.ascontiguousarray(q.T).reshape(phi.shape) * np.sqrt(n ** 3 / L ** 3)
    phid = torch.from_numpy(phi).cuda()
    ex = hfx.Exchange(np.diag([L] * 3), (n, n, n), precision=precision)
    piv, Q, Phi = ex.scdm_localise(phid)
    ex.sync_status()
    pivots = piv.cpu().numpy()
    if precision == "fp64":
        assert np.array_equal(pivots, A.scdm_pivots(phi)[0])
    else:
        assert A.scdm_pivot_slack(phi, pivots).min() >= 1 - 1e-4
    _, Q0, Phi0 = A.scdm_localise(phi, pivots)
    for got, want in ((Q, Q0), (Phi, Phi0)):
        assert np.linalg.norm(got.cpu().numpy() - want) < 10 * TOL[precision] * np.linalg.norm(want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        again = ex.scdm_localise(phid)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(again, (piv, Q, Phi)))
    ex.close()
