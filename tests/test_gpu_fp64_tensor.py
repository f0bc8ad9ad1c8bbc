"""FP64 contractions on the tensor cores at tile edges and remainders: force
bias, energy and one propagation step of FP64 contexts against the oracles. The
rows, the walkers' columns and the contraction lengths straddle the 128 x 64 tile,
the 32-element k-block and the 384-step chunk."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [  # M, n_alpha, n_beta, n_core, n_act, n_chol, n_w
    (33, 5, 4, 1, 9, 130, 1),        # K = 33: one element past a k-block; 1 walker
    (40, 7, 7, 2, 11, 127, 5),
    (64, 9, 8, 3, 12, 385, 3),       # n_chol one past a chunk
    (47, 4, 3, 0, 8, 200, 33),       # 2 x 33 columns: two past a tile
    (80, 33, 32, 29, 8, 60, 2),      # epilogue: N = 32 in fixed point, N = 33 in FP64
    (70, 18, 17, 14, 8, 96, 5),      # reference product: alpha on the tensor cores, beta not
]


@pytest.mark.parametrize("M,na,nb,nc,nact,G,nw", CASES)
def test_fp64_contractions_against_oracle(M, na, nb, nc, nact, G, nw):
    import torch

    import oracle
    from oracle import prop_oracle
    from paper_2406_08314_gb300 import msd, synth
    s = synth.make_system(M + G, M, na, nb, nc, nact, 40, 4, 1.2, G, decay=G / 6.0)
    w = synth.make_walkers(np.random.default_rng(G), M, na, nb, nw)
    ref = oracle.msd(s, w.phi_a, w.phi_b, per_det=True)
    scale_e = np.sum(np.abs(s.coeff * ref["det_ovlp"] * ref["det_e"]), axis=1) / np.abs(ref["ovlp"])
    da, db = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
    ctx = msd.Context(s, "fp64")
    o, v, e = (t.cpu().numpy() for t in ctx.evaluate(da, db))
    assert np.all(np.abs(v - ref["vbias"]) <= 1e-12 * np.abs(ref["vbias"]).max())
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-10 * scale_e)
    x = np.random.default_rng(1).standard_normal((nw, G))
    ra, rb, rw, rS = prop_oracle.step(s, w.phi_a, w.phi_b, np.ones(nw), x, 0.01, orthonormalize=True)
    wt = torch.ones(nw, dtype=torch.float64, device="cuda")
    S = ctx.propagate(da, db, wt, torch.from_numpy(x).cuda(), 0.01, 6, True)
    assert np.allclose(S.cpu().numpy(), rS, rtol=1e-10, atol=0)
    assert np.allclose(wt.cpu().numpy(), rw, rtol=1e-10, atol=0)
    assert np.abs(da.cpu().numpy() - ra).max() <= 1e-12 and np.abs(db.cpu().numpy() - rb).max() <= 1e-12
    ctx.close()
