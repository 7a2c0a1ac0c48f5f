"""A workspace that holds batches of 1 GiB with launches of their own, but not what hfx_workspace_bytes asks
for: hfx_apply, the batched call and Exchange take it and give the same result; a smaller one is refused."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2309_00651_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def problem(n, n_orb):
    phi = torch.from_numpy(np.random.default_rng(n).standard_normal((n_orb, n, n, n))).cuda()
    return phi, torch.from_numpy(I.all_pairs(n_orb)).cuda(), np.diag([n / 4.0] * 3)


def room(ex, nbytes):
    from paper_2309_00651_gb300 import hfx
    ex._ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    hfx.hfx_set_workspace(ex.ctx, ex._ws)


@pytest.mark.parametrize("n,n_orb", [(64, 26), (72, 33)])
def test_least_workspace(n, n_orb):
    from paper_2309_00651_gb300 import hfx
    phi, pairs, box = problem(n, n_orb)
    ex = hfx.Exchange(box, (n, n, n), precision="fp32")
    full, least = (f(ex.ctx, n_orb, len(pairs)) for f in (hfx.hfx_workspace_bytes, hfx.hfx_workspace_bytes_least))
    assert least < full
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    V = torch.empty_like(phi)
    out = []
    for nbytes in (full, full - 256, least + 4096, least):
        room(ex, nbytes)
        for call in (lambda a: hfx.hfx_apply(ex.ctx, *a), lambda a: hfx.hfx_apply_batched([ex.ctx], [a + (0,)])):
            E.zero_()
            V.zero_()
            call((phi, pairs, E, V))
            ex.sync_status()
            out.append((E.item(), V.clone()))
    # the same transforms, added into V in the same order
    assert all(e == out[0][0] and torch.equal(v, out[0][1]) for e, v in out)
    room(ex, least - 256)
    with pytest.raises(hfx.HFXError) as err:
        hfx.hfx_apply(ex.ctx, phi, pairs, E, V)
    assert err.value.status == -3
    ex.close()


def test_exchange_without_memory_for_more(monkeypatch):
    from paper_2309_00651_gb300 import hfx
    phi, pairs, box = problem(64, 26)
    ex = hfx.Exchange(box, (64, 64, 64), precision="fp32")
    want = ex.apply(phi, pairs)
    full, least = (f(ex.ctx, 26, len(pairs)) for f in (hfx.hfx_workspace_bytes, hfx.hfx_workspace_bytes_least))
    ex._ws = None
    real, asked = torch.empty, []

    def empty(*a, **k):
        if k.get("dtype") == torch.uint8:
            asked.append(a[0])
            if a[0] > least:
                raise torch.cuda.OutOfMemoryError("no room")
        return real(*a, **k)

    monkeypatch.setattr(torch, "empty", empty)
    for _ in range(2):
        E, V = ex.apply(phi, pairs)
        ex.sync_status()
        assert E.item() == want[0].item() and torch.equal(V, want[1])
    assert asked == [full, least]  # it is not asked for again on the next call
    ex.close()
