"""Ratios of every determinant by the expansions over shared minors, levels 0 to
6 per spin, with all, some or none of the smaller strings in the trial, and at
walker counts around the tiles of 32: against numpy determinants in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_act,n_o,n_det,n_w", [
    (8, 4, 4900, 33),      # the complete space: every sub-minor is a string of the trial
    (12, 6, 2500, 3),      # levels up to 6, some sub-minors missing
    (12, 6, 40, 1),        # sparse: expansions over 2 x 2 minors only
    (7, 1, 20, 70),        # a single active electron: level 1 alone
])
def test_ratios_against_determinants(n_act, n_o, n_det, n_w):
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, n = 15, n_o + 1
    n_det = min(n_det, sum(synth.math.comb(n_o, k) * synth.math.comb(n_act - n_o, k) for k in range(7)) ** 2)
    s = synth.make_system(n_act + n_det, M, n, n, 1, n_act, n_det, 12, 1.0, 8)
    w = synth.make_walkers(np.random.default_rng(5), M, n, n, n_w, noise=0.4)
    want = np.ones((n_w, n_det), complex)
    for occ, phi in ((s.occ_a, w.phi_a), (s.occ_b, w.phi_b)):
        want *= np.linalg.det(phi[:, occ]) / np.linalg.det(phi[:, occ[0]])[:, None]
    da, db = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
    for prec in ("fp64", "mixed"):
        ctx = msd.Context(s, prec)
        r = ctx.det_ratios(da, db).cpu().numpy()
        _, total = ctx.overlap(da, db, ratio_sum=True)
        # FP64 rounding of minors of entries of order one, a few hundred products
        assert np.all(np.abs(r - want) <= 1e-12 * np.abs(want).max(axis=1, keepdims=True)), prec
        assert np.allclose(total.cpu().numpy(), want @ s.coeff, rtol=0, atol=1e-12 * np.abs(want).max() * np.abs(s.coeff).sum())
        ctx.close()
