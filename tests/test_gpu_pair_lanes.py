"""FP64 per-determinant energy terms by groups of lanes: the largest opposite-spin Gram
matrix (112 x 112 active pairs: fewer warps per block), more determinants of one level
pair than a block takes, counts that no group size divides, and level pairs up to
(4, 4), against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _trial(s, n_o, n_act, pairs, seed):
    """s with `count` random determinants of every (level_a, level_b, count)."""
    rng = np.random.default_rng(seed)
    occ = {(tuple(range(n_o)), tuple(range(n_o))): 1.0}

    def string(k):
        keep = np.delete(np.arange(n_o), rng.choice(n_o, k, replace=False))
        return tuple(sorted(np.concatenate([keep, n_o + rng.choice(n_act - n_o, k, replace=False)]).tolist()))

    for ka, kb, count in pairs:
        for _ in range(count):
            occ.setdefault((string(ka), string(kb)), rng.normal() / np.sqrt(count))
    s.occ_a = np.array([a for a, _ in occ], np.int32)
    s.occ_b = np.array([b for _, b in occ], np.int32)
    s.coeff = np.array(list(occ.values()))
    return s


@pytest.mark.parametrize("n_o,n_act,pairs,n_w", [
    (8, 22, [(1, 1, 40), (2, 4, 61), (3, 3, 47), (2, 0, 9), (0, 3, 9)], 2),
    (5, 10, [(1, 2, 30), (2, 2, 2100), (3, 3, 2011), (4, 2, 1), (1, 5, 3)], 3),
    (6, 12, [(4, 4, 33), (3, 5, 11), (6, 2, 7), (1, 6, 5), (6, 6, 4), (2, 1, 31)], 33),
])
def test_energy(n_o, n_act, pairs, n_w):
    import torch

    import oracle
    from paper_2406_08314_gb300 import msd, synth
    M = n_act + 2
    s = synth.make_system(11, M, n_o, n_o, 0, n_act, 6, 12, 0.7, 10)
    s = _trial(s, n_o, n_act, pairs, 5)
    w = synth.make_walkers(np.random.default_rng(4), M, n_o, n_o, n_w, noise=0.4)
    ref = oracle.msd(s, w.phi_a, w.phi_b, energy=True, vbias=False, per_det=True)
    da, db = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
    scale = np.sum(np.abs(s.coeff * ref["det_ovlp"] * ref["det_e"]), axis=1) / np.abs(ref["ovlp"])
    ctx = msd.Context(s, "fp64")
    e = ctx.local_energy(da, db).cpu().numpy()
    one = ctx.local_energy(da[:1].contiguous(), db[:1].contiguous()).cpu().numpy()
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-10 * scale)   # the parity tests' bound
    assert np.abs(one[0] - e[0]) <= 1e-12 * scale[0]
    ctx.close()


def test_one_launch_and_separate_launches_agree():
    """Few walkers take every level pair in one launch, many a launch per pair: the
    same value for the same walker."""
    import torch

    from paper_2406_08314_gb300 import msd, synth
    n_o, n_act, n_w = 5, 10, 200
    s = synth.make_system(11, n_act + 2, n_o, n_o, 0, n_act, 6, 12, 0.7, 10)
    s = _trial(s, n_o, n_act, [(1, 1, 25), (1, 2, 30), (2, 2, 400), (3, 3, 500), (2, 4, 50), (4, 2, 31), (1, 5, 3)], 5)
    w = synth.make_walkers(np.random.default_rng(4), n_act + 2, n_o, n_o, n_w, noise=0.4)
    da, db = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
    for precision in ("fp64", "mixed"):
        ctx = msd.Context(s, precision)
        e = ctx.local_energy(da, db)
        few = ctx.local_energy(da[:3].contiguous(), db[:3].contiguous())
        assert torch.equal(e[:3], few), precision
        ctx.close()
