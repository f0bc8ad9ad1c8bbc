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


def _cofactor_form(s, phi):
    """G_T per spin of one walker [1; T] from determinants of the strings' sub-blocks:
    G - G Cm G / R + Cm G / R, Cm[p][h] = sum_I c_I r_other dr / dG[h][p]."""
    M, n = phi[0].shape
    hp = [exact_msd.levels(o) for o in (s.occ_a, s.occ_b)]
    r = np.ones((2, s.n_det), complex)
    cof = []
    for i in (0, 1):
        out = np.zeros((s.n_det, M, M), complex)
        for I, (h, p) in enumerate(hp[i]):
            k = len(h)
            if not k:
                continue
            sign = (-1) ** (sum(n - 1 - x for x in h) - k * (k - 1) // 2)
            a = phi[i][p][:, h].T                                      # G[h][p] = T[p][h]
            r[i, I] = sign * np.linalg.det(a)
            for x in range(k):
                for y in range(k):
                    b = np.delete(np.delete(a, x, 0), y, 1)
                    out[I, p[y], h[x]] = sign * (-1) ** (x + y) * (np.linalg.det(b) if k > 1 else 1.0)
        cof.append(out)
    R = (s.coeff * r[0] * r[1]).sum()
    res = []
    for i in (0, 1):
        cm = np.tensordot(s.coeff * r[1 - i], cof[i], 1) / R           # [p][h]
        g = np.zeros((M, M), complex)
        g[:n] = phi[i].T
        y = cm @ g
        res.append(g - g @ y + y)
    return np.stack(res)


@pytest.mark.parametrize("entries", [{(5, 1): 0.5}, {(5, 1): 7.0}, {(5, 1): 7.0, (6, 2): -3.0 + 2j, (7, 3): 0.25}])
def test_beside_large_entries(entries):
    """Active blocks with a few entries, some above 1, and zeros: most ratios vanish."""
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, n = 9, 4
    s = synth.make_system(3, M, n, n, 0, 8, 6, 4, 0.7, 10)
    s = exact_msd.with_strings(s, n, 8, [(1, 0, 9), (0, 1, 9), (2, 1, 40), (2, 2, 60), (3, 1, 30), (4, 0, 1), (0, 4, 1)],
                               np.random.default_rng(3))
    phi = np.eye(M, n, dtype=complex)
    for (p, h), x in entries.items():
        phi[p, h] = x
    want = _cofactor_form(s, [phi, phi])
    d = torch.from_numpy(np.ascontiguousarray(phi[None])).cuda()
    ctx = msd.Context(s, "fp64")
    rdm = ctx.rdm1(d, d).cpu().numpy()[0]
    _, v, _ = ctx.evaluate(d, d)
    f = ctx.force_bias(d, d)
    ctx.close()
    # a few hundred products of entries up to 7, FP64
    assert np.abs(rdm - want).max() <= 1e-12 * np.abs(want).max()
    assert torch.equal(v, f)
