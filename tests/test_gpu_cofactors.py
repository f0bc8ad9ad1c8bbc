"""FP64 cofactors by reverse differentiation of the minors' expansions: force bias
and density matrix against the oracle for trials that hold all, some or none of the
sub-minors, levels up to 6 per spin, unequal spins, walker counts around a warp, and
several walker chunks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_act,n_o,extra,n_det,n_w", [
    (8, 4, 1, 400, 33),     # complete low levels
    (12, 6, 0, 300, 3),     # levels up to 6, sub-minors outside the trial
    (12, 6, 2, 12, 1),      # a handful of high determinants
    (6, 1, 0, 6, 5),        # level 1 alone
])
def test_force_bias_and_density(n_act, n_o, extra, n_det, n_w):
    import torch

    import oracle
    from paper_2406_08314_gb300 import msd, synth
    M, nb = 15, n_o
    na = min(nb + extra, n_act)
    s = synth.make_system(7 + n_det, M, na, nb, 0, n_act, n_det, 12, 0.7, 10)
    w = synth.make_walkers(np.random.default_rng(2), M, na, nb, n_w, noise=0.4)
    ref = oracle.msd(s, w.phi_a, w.phi_b, energy=False, green=True, per_det=True)
    da, db = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
    ctx = msd.Context(s, "fp64")
    # cancellation scale of the determinant sums, as in the parity tests
    canc = np.sum(np.abs(s.coeff * ref["det_ovlp"]), axis=1) / np.abs(ref["ovlp"])
    for limit in (0, 200 * 1024):           # one chunk, several
        ctx.set_workspace_limit(limit)
        v, o = (t.cpu().numpy() for t in ctx.force_bias(da, db, ovlp=True))
        g = ctx.rdm1(da, db).cpu().numpy()
        assert np.allclose(o, ref["ovlp"], rtol=1e-10 * canc.max(), atol=0)
        assert np.all(np.abs(v - ref["vbias"]) <= 1e-10 * canc[:, None] * np.abs(ref["vbias"]).max())
        assert np.all(np.abs(g - ref["G_T"]) <= 1e-10 * canc[:, None, None, None] * np.abs(ref["G_T"]).max())
    ctx.close()
