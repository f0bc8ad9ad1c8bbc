"""A walker with a singular reference block is flagged and leaves zero rows of G, whichever
way the reference product runs (by size: alpha on the tensor cores, beta not), and leaves
the other walkers alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_rows_of_a_singular_walker_are_zero():
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, na, nb, nw = 64, 20, 18, 4        # (M - N) N^2 = 17600, 14904
    s = synth.make_system(5, M, na, nb, 15, 12, 20, 3, 0.7, 12)
    w = synth.make_walkers(np.random.default_rng(1), M, na, nb, nw)
    good = [torch.from_numpy(x).cuda() for x in (w.phi_a, w.phi_b)]
    bad = [x.clone() for x in good]
    bad[0][1, :na, 3] = 0                # alpha of walker 1, beta of walker 2
    bad[1][2, :nb, 5] = 0
    ctx = msd.Context(s, "fp64")
    want = ctx.features_rows(*good)
    with pytest.raises(msd.MSDError) as err:
        ctx.features_rows(*bad)
    assert err.value.name == "MSD_ERR_REF_SINGULAR"
    ctx.set_sync(False)
    f = ctx.features_rows(*bad)
    torch.cuda.synchronize()
    ctx.close()
    cut = 2 * na * M
    assert torch.equal(f[0], want[0]) and torch.equal(f[3], want[3])
    assert not f[1, :cut].any() and torch.equal(f[1, cut:], want[1, cut:])
    assert not f[2, cut:2 * (na + nb) * M].any() and torch.equal(f[2, :cut], want[2, :cut])
