"""FP64 force bias and density matrix at walkers whose ratios vanish: the cofactors do
not. At phi = D_0 the mixed Green's function is D_0 D_0^T plus one entry +-c_I / c_0 per
single excitation; evaluate, force_bias, rdm1 agree with it and with one another."""
import numpy as np
import pytest

import exact_msd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_act,n,pairs", [
    (8, 4, [(1, 0, 9), (0, 1, 9), (2, 1, 40), (2, 2, 60), (4, 2, 5)]),
    (12, 6, [(1, 0, 3), (0, 1, 3), (2, 0, 3), (3, 2, 9), (5, 1, 3), (6, 0, 1), (4, 4, 9)]),
])
def test_at_the_reference(n_act, n, pairs):
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, G = 15, 10
    s = synth.make_system(3, M, n, n, 0, n_act, 6, 4, 0.7, G)
    s = exact_msd.with_strings(s, n, n_act, pairs, np.random.default_rng(3))
    g = np.zeros((2, M, M))
    g[:, np.arange(n), np.arange(n)] = 1.0
    ref = set(range(n))
    for c, oa, ob in zip(s.coeff, s.occ_a, s.occ_b):
        ex = [(i, sorted(ref - set(o)), sorted(set(o) - ref)) for i, o in enumerate((oa, ob)) if set(o) != ref]
        if len(ex) == 1 and len(ex[0][1]) == 1:
            i, (h,), (p,) = ex[0]
            g[i, p, h] += c / s.coeff[0] * (-1) ** (n - 1 - h)
    assert np.count_nonzero(g) > 2 * n
    want = np.einsum("gpq,spq->g", s.L, g)
    phi = torch.eye(M, n, dtype=torch.complex128, device="cuda").repeat(3, 1, 1)
    ctx = msd.Context(s, "fp64")
    _, v, _ = ctx.evaluate(phi, phi)
    f = ctx.force_bias(phi, phi)
    rdm = ctx.rdm1(phi, phi).cpu().numpy()
    ctx.close()
    # sums of at most 2 M^2 products of order one
    assert np.abs(rdm - g).max() <= 1e-13 * np.abs(g).max()
    assert np.abs(f.cpu().numpy() - want).max() <= 1e-13 * np.abs(s.L).sum((1, 2)).max() * np.abs(g).max()
    assert torch.equal(v, f)
