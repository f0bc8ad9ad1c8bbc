"""More walkers in one chunk than a grid's second dimension holds (65535): features, whose
reference product runs on the tensor cores for one spin."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_features_of_65600_walkers():
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, na, nb, nw, rep = 61, 20, 4, 8, 8200          # (M - N) N^2 = 16400, 912
    s = synth.make_system(5, M, na, nb, 3, 20, 6, 2, 1.0, 12)
    w = synth.make_walkers(np.random.default_rng(1), M, na, nb, nw)
    few = [torch.from_numpy(x).cuda() for x in (w.phi_a, w.phi_b)]
    many = [x.repeat(rep, 1, 1) for x in few]
    ctx = msd.Context(s, "fp64")
    want = ctx.features_rows(*few)
    ctx.set_workspace_limit(64 << 30)
    got = ctx.features_rows(*many)
    assert ctx.info("walker_chunk") == nw * rep
    ctx.close()
    assert torch.equal(got.reshape(rep, nw, -1), want.expand(rep, -1, -1))
