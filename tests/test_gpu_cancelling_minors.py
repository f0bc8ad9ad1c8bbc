"""Walkers that overlap the reference little: the Green's function's active block is a
large part of low rank plus one of order one, and the minors from level 3 on are sums
that cancel. Ratios, overlaps, density matrix, force bias and energy against 60-digit
arithmetic, within what a pivoted LU of every minor may be off."""
import numpy as np
import pytest

import exact_msd

pytestmark = pytest.mark.gpu

N, N_ACT = 7, 14
PAIRS = [(0, 1, 3), (1, 0, 3), (2, 0, 5), (3, 0, 6), (4, 0, 6), (5, 0, 6), (6, 0, 6), (0, 4, 4), (0, 6, 3)]


def _system(seed, complete):
    from paper_2406_08314_gb300 import synth
    s = synth.make_system(seed, N_ACT + 1, N, N, 0, N_ACT, 6, 12, 0.7, 6)
    pairs = PAIRS if not complete else PAIRS + [(2, 3, 4), (3, 0, 250), (4, 0, 250), (5, 0, 60)]
    return exact_msd.with_strings(s, N, N_ACT, pairs, np.random.default_rng(seed))


def _walkers(rank, size, n_w, seed):
    """phi = [1; T]: G of the active block is T^T to the last bit."""
    rng = np.random.default_rng(seed)

    def c(*shape):
        return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)

    out = []
    for _ in (0, 1):
        m = N_ACT + 1 - N
        t = 0.5 * c(n_w, m, N)
        if rank:
            t += size * (c(n_w, m, rank) @ c(n_w, rank, N)) / 2
        out.append(np.ascontiguousarray(np.concatenate([np.broadcast_to(np.eye(N), (n_w, N, N)), t], 1)))
    return out


def _ratios(s, walkers):
    """Exact ratios of the two spins' strings and their LU bounds, [w][det] each."""
    r = [[], []]
    for occ, phi in ((s.occ_a, walkers[0]), (s.occ_b, walkers[1])):
        hp = exact_msd.levels(occ)
        for w in range(phi.shape[0]):
            done, row = {}, []
            for h, p in hp:
                if (key := (tuple(h), tuple(p))) not in done:
                    if h:
                        sign = (-1) ** (sum(N - 1 - x for x in h) - len(h) * (len(h) - 1) // 2)
                        d, b = exact_msd.minor(phi[w][p][:, h])
                        done[key] = (sign * d, b)
                    else:
                        done[key] = (1.0 + 0j, 0.0)
                row.append(done[key])
            r[occ is s.occ_b].append(row)
    return [(np.array([[x[0] for x in q] for q in z]), np.array([[x[1] for x in q] for q in z])) for z in r]


CASES = [(0, 0.0), (1, 3.0), (1, 30.0), (1, 1e3), (1, 1e4), (2, 30.0), (2, 1e3), (2, 1e4)]


@pytest.mark.parametrize("complete", [False, True])
@pytest.mark.parametrize("rank,size", CASES)
def test_ratios(rank, size, complete):
    import torch

    from paper_2406_08314_gb300 import msd
    s, w = _system(2, complete), _walkers(rank, size, 2, 9)
    (ra, ba), (rb, bb) = _ratios(s, w)
    want, tol = ra * rb, ba * np.abs(rb) + bb * np.abs(ra) + 1e-15 * np.abs(ra * rb)
    dev = [torch.from_numpy(x).cuda() for x in w]
    total, tt = want @ s.coeff, tol @ np.abs(s.coeff) + 1e-14 * np.abs(want) @ np.abs(s.coeff)
    for prec in ("fp64", "mixed"):
        ctx = msd.Context(s, prec)
        r = ctx.det_ratios(*dev).cpu().numpy()
        assert np.all(np.abs(r - want) <= tol), prec
        assert np.all(np.abs(ctx.overlap(*dev).cpu().numpy() - total) <= tt), prec
        o = torch.empty(2, dtype=torch.complex128, device="cuda")
        ctx.overlap_noalloc(*dev, o)
        assert np.all(np.abs(o.cpu().numpy() - total) <= tt), prec
        ctx.close()


@pytest.mark.parametrize("rank,size", CASES)
def test_observables(rank, size):
    import torch

    from paper_2406_08314_gb300 import msd
    s, w = _system(2, False), _walkers(rank, size, 1, 9)
    ref = exact_msd.msd(s, *w)
    # a determinant's relative error as of the LU bounds of its two strings (their
    # inverses are off by no more), its Green's function and energy weighted with it;
    # FP64 sums of terms as large as the reference's and the determinants' own
    (ra, ba), (rb, bb) = _ratios(s, w)
    rel = 4 * (ba / np.abs(ra) + bb / np.abs(rb)) + 1e-14
    f = np.abs(s.coeff * ref["det_ovlp"]) / np.abs(ref["ovlp"])[:, None]
    g = np.abs(ref["det_g"]).max(axis=(2, 3, 4))
    tol_g = np.sum(f * rel * (g + g[:, :1]), 1)
    lam = np.abs(s.L).sum(axis=(1, 2)).max()
    big = np.abs(ref["det_e"]) + np.abs(ref["det_e"][:, :1]) + lam ** 2 * (g + g[:, :1]) ** 2
    tol_e = np.sum(f * rel * big, 1)
    dev = [torch.from_numpy(x).cuda() for x in w]
    ctx = msd.Context(s, "fp64")
    rdm = ctx.rdm1(*dev).cpu().numpy()
    assert np.all(np.abs(rdm - ref["G_T"]).max((1, 2, 3)) <= tol_g)
    _, v, e = (t.cpu().numpy() for t in ctx.evaluate(*dev))
    for x in (v, ctx.force_bias(*dev).cpu().numpy()):
        assert np.all(np.abs(x - ref["vbias"]).max(1) <= tol_g * lam)
    assert np.all(np.abs(e - ref["e_loc"]) <= tol_e)
    ctx.close()


@pytest.mark.parametrize("size", [1e-2, 1e-4, 1e-6])
def test_energy_of_blocks_near_rank_one(size):
    """Active blocks with entries below 1, of rank one but for a part of 0.1 size: minors from
    level 2 on are small, inverse minors large."""
    import torch

    from paper_2406_08314_gb300 import msd
    s, n_w = _system(2, False), 4
    rng = np.random.default_rng(5)

    def c(*shape):
        return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)

    walkers = []
    for _ in (0, 1):
        t = c(n_w, N_ACT + 1 - N, 1) @ c(n_w, 1, N)
        t *= 0.9 / np.maximum(np.abs(t.real), np.abs(t.imag)).max((1, 2), keepdims=True)
        t += 0.1 * size * c(*t.shape)
        walkers.append(np.ascontiguousarray(np.concatenate([np.broadcast_to(np.eye(N), (n_w, N, N)), t], 1)))
    ref = exact_msd.msd(s, *walkers)
    ctx = msd.Context(s, "fp64")
    e = ctx.local_energy(*[torch.from_numpy(x).cuda() for x in walkers]).cpu().numpy()
    ctx.close()
    # an inverse of condition k = 10 / size is off by u k of its entries, and a string's energy is
    # ratio x inverse x inverse, of the size of k for level 2 and its sums of up to 64 terms
    assert np.all(np.abs(e - ref["e_loc"]) <= 64 * 2.0 ** -53 * 10 / size * np.abs(ref["e_loc"]))
