"""The plane energies of the compile-time FP32 passes carry FP32 rounding inside one butterfly only.

A density that is 1 at the origin and 0 elsewhere has F(G) = 1 exactly (every butterfly adds zeros to ones
and every twiddle it meets is 1), so E_x is -(alpha/2) (Omega/N^2) sum_G v(G) with v rounded to FP32 and no
error but that of the sum.  One butterfly of the last x stage, of radix r, adds the r terms of the x
frequencies k, k + n/r, ... in that order in FP32; all other sums keep at least 2^-48 of what they add, 20
times a plane, so E agrees with those chains summed in FP64 to 20 2^-48 < 1e-13, and the bound here leaves
room for single entries of v that the two sides round differently (2^-24 of one of about N / 10 terms)."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BOUND = 1e-11


def chained_sum(n, L, r):
    m = np.fft.fftfreq(n, 1.0 / n) * (2.0 * math.pi / L)
    gg = m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2
    gg[0, 0, 0] = np.inf
    v = (4.0 * math.pi / gg).astype(np.float32).reshape(r, n // r, n, n)
    chain = v[0].copy()
    for f in range(1, r):
        chain += v[f]
    return float(chain.sum(dtype=np.float64))


@pytest.mark.parametrize("n,r", [(n, 4) for n in (32, 36, 40, 48, 60, 64, 72, 80, 96, 100, 108, 120, 128)]
                         + [(50, 5), (54, 9), (90, 9)])
@pytest.mark.parametrize("energy_only", [False, True])
def test_only_butterflies_round(n, r, energy_only):
    from paper_2309_00651_gb300 import hfx
    phi = torch.zeros((1, n, n, n), dtype=torch.float64, device="cuda")
    phi[0, 0, 0, 0] = 1.0
    pairs = torch.zeros((1, 2), dtype=torch.int32, device="cuda")
    for L in (n / 4.0, n / 2.7):
        ex = hfx.Exchange(np.diag([L] * 3), (n, n, n), precision="fp32", alpha=0.25)
        E, _ = ex.apply(phi, pairs, energy_only=energy_only)
        ex.sync_status()
        ex.close()
        want = -0.125 * L ** 3 / float(n) ** 6 * chained_sum(n, L, r)
        assert abs(E.item() - want) <= BOUND * abs(want), (L, (E.item() - want) / want)
