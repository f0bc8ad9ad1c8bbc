"""FP64 energies of D_0 with Cholesky vectors on which an order of summation or a way of
rounding shows: E = 1/2 sum_g (2 sum_j L_jj)^2 - sum_g sum_jl L_jl^2 over the occupied
block, in exact rational arithmetic."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _energy(L, n):
    import torch

    from paper_2406_08314_gb300 import msd
    from paper_2406_08314_gb300.synth import System
    M = L.shape[1]
    occ = np.arange(n, dtype=np.int32)[None]
    s = System(M, n, n, np.zeros((2, M, M)), 0.0, L, np.ones(1), occ, occ)
    phi = torch.eye(M, n, dtype=torch.complex128, device="cuda")[None].contiguous()
    ctx = msd.Context(s, "fp64")
    e = complex(ctx.local_energy(phi, phi).cpu().numpy()[0])
    ctx.close()
    want = Fraction(0)
    for g in L[:, :n, :n]:
        q = [[Fraction(float(x)) for x in r] for r in g]
        want += 2 * sum(q[j][j] for j in range(n)) ** 2 - sum(x * x for r in q for x in r)
    assert e.imag == 0.0
    return e.real, want


def test_sum_over_vectors():
    # one vector of 1 and seven of 2^-27, 32 vectors apart: sum of squares 1 + 7 2^-54
    L = np.zeros((256, 4, 4))
    L[::32, 0, 0] = 2.0 ** -27
    L[0, 0, 0] = 1.0
    e, want = _energy(L, 1)
    # eight partial sums added in pairs: three roundings of half an ulp
    assert abs(Fraction(e) - want) <= Fraction(3, 2) * Fraction(1, 2 ** 52), float(Fraction(e) - want)


def test_ties_round_to_even():
    # 1 and values just below 1/4 whose last two of 55 bits are 10: ties at 53
    rng = np.random.default_rng(0)
    n = 32
    m = np.triu(rng.integers(2 ** 53 - 2 ** 50, 2 ** 53, (n, n)) // 4 * 4 + 2)
    x = (m + np.triu(m, 1).T).astype(float) * 2.0 ** -55
    x *= np.where((np.add.outer(np.arange(n), np.arange(n)) // 2) % 2, -1.0, 1.0)
    x[0, 0] = 1.0
    L = np.zeros((1, 40, 40))
    L[0, :n, :n] = x
    e, want = _energy(L, n)
    # the sum of squares and of the traces' square to half an ulp each, their differences: two
    # ulps; 2^10 ties of one sign are four
    assert abs(Fraction(e) - want) <= 2 * Fraction(float(np.spacing(abs(float(want))))), float(Fraction(e) - want)
