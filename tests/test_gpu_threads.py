"""hfx_workspace_bytes only reads the context: it may be called from other threads while a call for a new
orbital count adds that count's schedule."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2309_00651_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def test_workspace_bytes_beside_new_schedules():
    from paper_2309_00651_gb300 import hfx
    n, counts = 16, list(range(1, 41))
    box = np.diag([4.0] * 3)
    ex = hfx.Exchange(box, (n, n, n), precision="fp32")
    want = {k: hfx.hfx_workspace_bytes(ex.ctx, k, 1) for k in counts}
    ex.ensure_workspace(counts[-1], 1)
    phi = torch.randn((counts[-1], n, n, n), dtype=torch.float64, device="cuda")
    wrong, stop = [], threading.Event()

    def ask(seed):
        order = np.random.default_rng(seed).permutation(counts)
        while not stop.is_set():
            for k in order:
                if hfx.hfx_workspace_bytes(ex.ctx, int(k), 1) != want[int(k)]:
                    wrong.append(int(k))
                    return

    threads = [threading.Thread(target=ask, args=(s,)) for s in range(8)]
    for t in threads:
        t.start()
    try:
        for k in counts[::-1]:
            ex.apply(phi[:k].contiguous(), torch.from_numpy(I.all_pairs(k)).cuda())
    finally:
        stop.set()
        for t in threads:
            t.join()
    ex.sync_status()
    ex.close()
    assert not wrong
