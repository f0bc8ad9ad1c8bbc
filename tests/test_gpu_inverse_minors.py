"""FP64 inverse minors as cofactors over determinants: energies and force bias
against the oracle for trials that hold all, some or none of the sub-minors, whose
sub-minors are too many (the LU path), levels 1 to 6, unequal spins, walker counts
around a warp, several walker chunks, and a walker whose ratios all vanish (singular
minors: entries 0, as in the other forms)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _high_only(s, n_act, n_o, n_str, seed):
    """The trial's determinants replaced by disjointly drawn 6-fold alpha ones."""
    rng = np.random.default_rng(seed)
    occ = np.tile(np.arange(s.n_alpha, dtype=np.int32), (n_str + 1, 1))
    for row in occ[1:]:
        row[rng.choice(n_o, 6, replace=False)] = n_o + rng.choice(n_act - n_o, 6, replace=False)
    s.occ_a = np.unique(np.sort(occ, axis=1), axis=0)
    s.occ_b = np.tile(np.arange(s.n_beta, dtype=np.int32), (len(s.occ_a), 1))
    s.coeff = np.ones(len(s.occ_a)) / len(s.occ_a)
    return s


@pytest.mark.parametrize("n_act,n_o,extra,n_det,n_w", [
    (8, 4, 1, 400, 33),     # complete low levels
    (12, 6, 0, 300, 3),     # levels up to 6, sub-minors outside the trial
    (12, 6, 2, 12, 1),      # a handful of high determinants
    (6, 1, 0, 6, 5),        # level 1 alone
    (20, 10, 0, 0, 2),      # 30 6-fold strings: too many sub-minors
])
def test_energy_and_force_bias(n_act, n_o, extra, n_det, n_w):
    import torch

    import oracle
    from paper_2406_08314_gb300 import msd, synth
    M, nb = (22, n_o) if n_det == 0 else (15, n_o)
    na = min(nb + extra, n_act)
    s = synth.make_system(7 + n_det, M, na, nb, 0, n_act, max(n_det, 6), 12, 0.7, 10)
    if n_det == 0:
        s = _high_only(s, n_act, n_o, 30, 3)
    w = synth.make_walkers(np.random.default_rng(2), M, na, nb, n_w, noise=0.4)
    ref = oracle.msd(s, w.phi_a, w.phi_b, energy=True, vbias=True, per_det=True)
    da, db = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
    ctx = msd.Context(s, "fp64")
    # scales of the determinant sums, as in the parity tests
    r = s.coeff * ref["det_ovlp"]
    canc = np.sum(np.abs(r), axis=1) / np.abs(ref["ovlp"])
    scale_e = np.sum(np.abs(r * ref["det_e"]), axis=1) / np.abs(ref["ovlp"]) + canc * np.abs(ref["e_loc"])
    for limit in (0, 300 * 1024):           # one chunk, several
        ctx.set_workspace_limit(limit)
        e = ctx.local_energy(da, db).cpu().numpy()
        o, v, e2 = (t.cpu().numpy() for t in ctx.evaluate(da, db))
        assert np.all(np.abs(e - ref["e_loc"]) <= 1e-10 * scale_e)
        assert np.all(np.abs(e2 - ref["e_loc"]) <= 1e-10 * scale_e)
        assert np.allclose(o, ref["ovlp"], rtol=1e-10 * canc.max(), atol=0)
        assert np.all(np.abs(v - ref["vbias"]) <= 1e-10 * canc[:, None] * np.abs(ref["vbias"]).max())
    ctx.close()


def test_vanishing_ratios():
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, n = 15, 4
    s = synth.make_system(3, M, n, n, 0, 8, 300, 12, 0.7, 10)
    phi = torch.eye(M, n, dtype=torch.complex128, device="cuda").repeat(3, 1, 1)
    e = {}
    for prec in ("fp64", "mixed"):
        ctx = msd.Context(s, prec)
        o, v, e[prec] = (t.cpu().numpy() for t in ctx.evaluate(phi, phi))
        assert np.all(np.isfinite(v)) and np.allclose(o, s.coeff[0], rtol=1e-14)
        ctx.close()
    # single-determinant energy; FP32 contractions of at most M n_chol products each
    assert np.allclose(e["fp64"], e["mixed"], rtol=1e-5, atol=0)
