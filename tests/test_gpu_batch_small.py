"""hfx_apply_batched where every problem is small enough for the one persistent launch: the flags, an empty
list, capture, and the calls after a wait that ran out, against one call each.  (The problems of
test_gpu_batch.py are larger and run on forked streams, but for its stalled call.)"""
import os
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2309_00651_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOL = {"fp32": 1e-6, "fp64": 1e-8}  # of the batched call's other tests
SIZES = {"fp32": [(4, 24), (3, 18), (2, 30), (1, 32)], "fp64": [(3, 10), (2, 12), (2, 8), (1, 16)]}


def small(precision):
    """The rule that sends a batch to the persistent launch, on this file's sizes."""
    with open(os.path.join(ROOT, "paper_2309_00651_gb300", "csrc", "hfx_api.cu")) as f:
        fp64, fp32 = re.search(r"work > \(ctxs\[k\]->prec == HFX_PREC_FP64 \? (\S+) : (\S+)\)\) return false", f.read()).groups()
    most = float(fp64 if precision == "fp64" else fp32)
    return all(o <= 8 and 0.5 * o * (o + 1) * n ** 3 <= most for o, n in SIZES[precision])


def setup(precision):
    from paper_2309_00651_gb300 import hfx
    assert small(precision)
    exs, phis, lists = [], [], []
    for k, (n_orb, n) in enumerate(SIZES[precision]):
        phis.append(torch.from_numpy(np.random.default_rng(k).standard_normal((n_orb, n, n, n))).cuda())
        lists.append(torch.from_numpy(I.all_pairs(n_orb)).cuda())
        exs.append(hfx.Exchange(np.diag([n / 4.0] * 3), (n, n, n), precision=precision))
        exs[-1].ensure_workspace(n_orb, len(lists[-1]))
    return exs, phis, lists


def run(call, exs, phis, lists, flags):
    from paper_2309_00651_gb300 import hfx
    E = [torch.full((1,), 0.5, dtype=torch.float64, device="cuda") for _ in phis]
    V = [torch.full_like(p, 0.25) for p in phis]
    call([e.ctx for e in exs], [(p, q, e, None if f & hfx.HFX_ENERGY_ONLY else v, f)
                                for p, q, e, v, f in zip(phis, lists, E, V, flags)])
    for e in exs:
        e.sync_status()
    return E, V


def agree(got, want, tol):
    for a, b in zip(got[0] + got[1], want[0] + want[1]):
        assert float(torch.linalg.norm(a - b)) <= tol * float(torch.linalg.norm(b))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shift", range(4))
def test_flags_and_an_empty_list(precision, shift):
    from paper_2309_00651_gb300 import hfx
    exs, phis, lists = setup(precision)
    flags = np.roll([0, hfx.HFX_ENERGY_ONLY, hfx.HFX_ACCUMULATE, 0], shift).tolist()
    lists[(3 + shift) % 4] = lists[(3 + shift) % 4][:0]
    got, want = (run(f, exs, phis, lists, flags) for f in (hfx.hfx_apply_batched, hfx.hfx_apply_sequential))
    agree(got, want, TOL[precision])
    empty, energy = (3 + shift) % 4, (1 + shift) % 4
    assert got[0][empty].item() == 0.0 and not bool(got[1][empty].any()) and bool((got[1][energy] == 0.25).all())
    for e in exs:
        e.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_after_a_wait_that_ran_out_and_from_a_graph(precision):
    from paper_2309_00651_gb300 import hfx
    exs, phis, lists = setup(precision)
    ctxs = [e.ctx for e in exs]
    want = run(hfx.hfx_apply_sequential, exs, phis, lists, [0] * 4)
    hfx.hfx_set_wait_budget(ctxs[0], 200000)  # about 0.1 ms
    hfx.hfx_apply_batched(ctxs[:1], [(phis[0], lists[0], want[0][0].clone(), torch.empty_like(phis[0]), hfx.HFX_TEST_STALL)])
    with pytest.raises(hfx.HFXError) as err:
        exs[0].sync_status()
    assert err.value.status == -6
    hfx.hfx_set_wait_budget(ctxs[0], 0)
    got = run(hfx.hfx_apply_batched, exs, phis, lists, [0] * 4)
    agree(got, want, TOL[precision])
    E, V = [torch.empty_like(e) for e in got[0]], [torch.empty_like(v) for v in got[1]]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hfx.hfx_apply_batched(ctxs, list(zip(phis, lists, E, V, [0] * 4)))
    for _ in range(2):
        for t in E + V:
            t.fill_(7.0)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(E + V, got[0] + got[1]))
    for e in exs:
        e.close()
