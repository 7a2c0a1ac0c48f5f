"""Update A at every chain length with a kernel of its own (1 to 6), the lengths around them, and degrees of
freedom in each range of threads per block (32 to 256, by steps of 152 x 32), against the FP64 oracle with the
tolerance of test_gpu_sinr.py."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sinr_oracle as S  # noqa: E402

pytestmark = pytest.mark.gpu

KT = 0.0019
Q1, Q2 = KT * 40.0 ** 2, KT * 45.0 ** 2


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b))


@pytest.mark.parametrize("L,n", [(L, 1000) for L in (2, 3, 5, 6, 7)]
                         + [(L, n) for L in (2, 6) for n in (1, 31, 33, 4864, 4865, 10007, 38913, 50001)])
def test_update_a(L, n):
    from paper_2309_00651_gb300 import hfx
    rng = np.random.default_rng(L * 100000 + n)
    M, V = rng.uniform(1000.0, 30000.0, n), rng.standard_normal(n) * 1e-3
    v1, v2 = rng.standard_normal((n, L)) * math.sqrt(KT / Q1), rng.standard_normal((n, L)) * math.sqrt(KT / Q2)
    f = np.sqrt(L * KT / S.constraint(M, V, v1, Q1, L))
    V, v1 = V * f, v1 * f[:, None]
    got = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (V, v1, v2)]
    hfx.hfx_sinr_update_n({"kT": KT, "Q1": Q1, "Q2": Q2, "gamma": 0.01, "L": L}, 30.0, torch.from_numpy(M).cuda(), *got,
                          n_res=2, n_sy=3)
    want = S.update_n_half_step(V, v1, v2, M, KT, Q1, Q2, L, 30.0, n_res=2, n_sy=3)
    assert all(rel(a, b) < 1e-12 for a, b in zip(got, want))
