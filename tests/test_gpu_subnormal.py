"""FP64 force bias of Cholesky vectors whose entries are all subnormal numbers: the
contraction on the tensor cores keeps them as the FP64 units do."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_subnormal_rows():
    import torch

    import oracle
    from paper_2406_08314_gb300 import msd, synth
    M, n, G = 40, 7, 100                        # n_chol Kd = 100 x 960: on the tensor cores
    s = synth.make_system(9, M, n, n, 2, 11, 40, 4, 1.2, G, decay=1e3)
    w = synth.make_walkers(np.random.default_rng(0), M, n, n, 3)
    ref = oracle.msd(s, w.phi_a, w.phi_b, energy=False)["vbias"]
    tiny = 2.0 ** -1030
    L = s.L.copy()
    L[G // 2:] *= tiny
    assert np.abs(L[G // 2:]).max() < np.finfo(float).tiny
    s.L = L
    ctx = msd.Context(s, "fp64")
    v = ctx.force_bias(torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()).cpu().numpy()
    ctx.close()
    assert np.abs(v[:, :G // 2] - ref[:, :G // 2]).max() <= 1e-12 * np.abs(ref).max()
    # M^2 entries rounded to 2^-1074 each, at 2^-1030 of the vectors' scale
    assert np.abs(v[:, G // 2:] * 2.0 ** 1000 - ref[:, G // 2:] * 2.0 ** -30).max() <= 2.0 ** -30 * M * M * 2.0 ** -44
