"""Same-spin energies of strings whose inverse minors have large columns and rows (holes
and particles that the walker mixes only weakly: 1 / amplitude) beside ordinary ones,
FP64 mode, levels 1 to 6, per system and batched, against 60-digit arithmetic. A
determinant's term stays of order one as the amplitude goes to zero."""
import numpy as np
import pytest

import exact_msd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hole,part", [(1, 1), (1e-2, 1), (1, 1e-2), (1e-4, 1), (1e-8, 1), (1, 1e-8), (1e-5, 1e-5),
                                       (1e-12, 1), (1, 1e-16), (1e-16, 1)])
def test_string_energies(hole, part):
    import torch

    from paper_2406_08314_gb300 import msd, synth
    n, n_act = 6, 12
    s = synth.make_system(3, n_act + 1, n, n, 0, n_act, 6, 12, 0.7, 8)
    s = exact_msd.with_strings(s, n, n_act, [(1, 0, 2), (2, 0, 6), (3, 0, 6), (4, 0, 6), (5, 0, 6), (6, 0, 1), (0, 2, 3), (2, 2, 3)],
                               np.random.default_rng(1))
    rng = np.random.default_rng(7)
    walkers = []
    for _ in (0, 1):
        t = rng.standard_normal((2, n_act + 1 - n, n)) + 1j * rng.standard_normal((2, n_act + 1 - n, n))
        t[:, :, 1] *= hole
        t[:, 2] *= part
        walkers.append(np.concatenate([np.broadcast_to(np.eye(n), (2, n, n)), 0.5 * t], 1))
    ref = exact_msd.msd(s, *walkers)
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in walkers]
    # FP64 rounding of sums of at most 225 products a string over the sum of the
    # determinants' magnitudes, three orders of slack
    scale = np.sum(np.abs(s.coeff * ref["det_ovlp"] * ref["det_e"]), 1) / np.abs(ref["ovlp"])
    ctx = msd.Context(s, "fp64")
    e = ctx.local_energy(*dev).cpu().numpy()
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * scale)
    batch = msd.Batch([ctx])
    eb = batch.evaluate([tuple(dev)])[0][2].cpu().numpy()
    assert np.all(np.abs(eb - ref["e_loc"]) <= 1e-12 * scale)
    batch.close()
    ctx.close()
