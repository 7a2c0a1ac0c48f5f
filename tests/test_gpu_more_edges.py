"""Every edge with compile-time passes against the runtime-geometry passes that took it before
(HFX_NO_CT=1), and the batched call's two forms against one call each."""
import numpy as np
import pytest
import torch

from paper_2309_00651_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [36, 40, 50, 54, 60, 100, 108, 120])
@pytest.mark.parametrize("n_orb,f32", [(9, False), (16, True), (4, True)])
def test_edge_against_runtime_geometry(n, n_orb, f32, monkeypatch):
    from paper_2309_00651_gb300 import hfx
    rng = np.random.default_rng(n)
    phi = torch.from_numpy(rng.standard_normal((n_orb, n, n, n))).cuda()
    phi = phi.float() if f32 else phi
    pairs = I.all_pairs(n_orb)
    pairs = torch.from_numpy(np.ascontiguousarray(pairs[rng.random(len(pairs)) < 0.8])).cuda()
    res = []
    for no_ct in ("0", "1"):
        monkeypatch.setenv("HFX_NO_CT", no_ct)
        ex = hfx.Exchange(np.diag([n / 4.0] * 3), (n, n, n), precision="fp32")
        E, V = ex.apply(phi, pairs)
        E_only, _ = ex.apply(phi, pairs, energy_only=True)
        ex.sync_status()
        assert abs(E_only.item() - E.item()) <= 1e-12 * abs(E.item())
        res.append((E.item(), V))
        ex.close()
    (Ea, Va), (Eb, Vb) = res
    # both are within the path's stated 1e-6 of the exact result
    assert abs(Ea - Eb) <= 2e-6 * abs(Eb)
    assert float(torch.linalg.norm(Va - Vb)) <= 2e-6 * float(torch.linalg.norm(Vb))


@pytest.mark.parametrize("sizes,precision", [(((9, 32), (12, 60), (20, 48), (5, 24)), "fp32"),   # forked streams
                                             (((9, 24), (3, 18)), "fp64"),
                                             (((12, 32), (9, 48)), "mixed_tc"),
                                             (((4, 24), (1, 30), (3, 32), (2, 36)), "fp32"),     # one persistent launch
                                             (((3, 10), (2, 12)), "fp64")])
def test_batched_forms(sizes, precision):
    from paper_2309_00651_gb300 import hfx
    exs, args, ref = [], [], []
    for k, (n_orb, n) in enumerate(sizes):
        phi = torch.from_numpy(np.random.default_rng(k).standard_normal((n_orb, n, n, n))).cuda()
        pairs = torch.from_numpy(I.all_pairs(n_orb)).cuda()
        ex = hfx.Exchange(np.diag([n / 4.0] * 3), (n, n, n), precision=precision)
        ex.ensure_workspace(n_orb, len(pairs))
        # a batched call runs MIXED_TC problems with the FP32 forward pass
        one = hfx.Exchange(np.diag([n / 4.0] * 3), (n, n, n), precision="fp32" if precision == "mixed_tc" else precision)
        E, V = one.apply(phi, pairs)
        ref.append((E.item(), V))
        one.close()
        exs.append(ex)
        args.append((phi, pairs, torch.zeros(1, dtype=torch.float64, device="cuda"), torch.empty_like(phi), 0))
    for _ in range(2):
        hfx.hfx_apply_batched([e.ctx for e in exs], args)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        hfx.hfx_apply_batched([e.ctx for e in exs], args)
    for a in args:
        a[2].zero_()
        a[3].zero_()
    g.replay()
    torch.cuda.synchronize()
    tol = 1e-12 if precision == "fp64" else 2e-6
    for ex, a, (E, V) in zip(exs, args, ref):
        ex.sync_status()
        assert abs(a[2].item() - E) <= tol * abs(E)
        assert float(torch.linalg.norm(a[3] - V)) <= tol * float(torch.linalg.norm(V))
        ex.close()
