"""The workspace limit: a propagation step's own buffers stay within the half of it that
they are sized for, the splits' partial results of a long contraction included."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_propagation_stays_within_its_share():
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, n, G, nw = 40, 6, 780, 60                # 25 k-blocks: V in two splits
    s = synth.make_system(4, M, n, n, 2, 8, 20, 3, 1.0, G)
    w = synth.make_walkers(np.random.default_rng(1), M, n, n, nw)
    pa, pb = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
    ctx = msd.Context(s, "mixed")               # the force bias in FP32: V alone is split
    limit = 4 << 20
    ctx.set_workspace_limit(limit)
    ctx.force_bias(pa, pb)
    ctx.overlap(pa, pb)
    before = ctx.info("workspace_bytes")
    wt = torch.ones(nw, dtype=torch.float64, device="cuda")
    x = torch.from_numpy(np.random.default_rng(2).standard_normal((nw, G))).cuda()
    ctx.propagate(pa, pb, wt, x, 0.01)
    # the fields, coefficients and overlaps of all walkers, and 256 bytes of rounding per buffer
    per_walker = 16 * nw * (2 * G + 3)
    assert ctx.info("workspace_bytes") - before <= limit // 2 + per_walker + 64 * 256
    ctx.close()
