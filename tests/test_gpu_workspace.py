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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_that_fits_its_results(precision):
    """All walkers of a batch share one chunk: a limit that holds their stages' results is
    enough, the tensor-core products' and expansions' scratch goes over them in pieces."""
    from collections import Counter

    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, n, G, nw = 64, 20, 120, 40
    s = synth.make_system(2, M, n, n, 14, 12, 300, 4, 1.0, G)
    w = synth.make_walkers(np.random.default_rng(3), M, n, n, nw)
    pair = tuple(torch.from_numpy(x).cuda() for x in (w.phi_a, w.phi_b))
    ref, ctxs = msd.Context(s, precision), [msd.Context(s, precision) for _ in (0, 1)]
    want = ref.evaluate(*pair)
    # complex numbers per walker: G's rows, active block, ratios, weights and inverse minors; partial
    # sums; G_T; per vector V0, exchange and the Lambda and Xi rows; Gram matrices; F (FP64)
    # or the split rows and partial products (mixed)
    X, NC, level, tot = 36, n + 6, [], 0
    for occ in (s.occ_a, s.occ_b):
        level.append([len(set(o.tolist()) - set(range(n))) for o in occ])
        strings = Counter({tuple(o.tolist()): k for o, k in zip(occ, level[-1])}.values())
        n_str = sum(strings.values())
        tot += n * M + 1 + X + 2 * n_str + (n_str + 1) // 2 + sum(c * (k * k + k % 2) for k, c in strings.items())
        tot += sum(-(-c // 1024) for c in strings.values()) + (-(-n_str // 32) if occ is s.occ_a else 0)
        tot += NC * M + X + G * (2 + 2 * X) + 3 * X + 1
    tot += sum(-(-c // 2048) for c in Counter(zip(*level)).values()) + 11 + 3 * X * X
    if precision == "fp64":
        tot += 2 * n * G * NC
    else:
        K = 64 * 14                    # N (M - N) padded to 64, one spin; and its partial results
        tot += (20 * K + 8 * G + 2 * (2 * 16 * ((880 + G + 63) // 64 * 2 + 2) + 16 * G) + 8 * 64 * 112 + 128 * G + 8 * 2 * NC * M) // 16
    limit = 16 * tot * nw
    for c in ctxs:
        c.set_workspace_limit(limit)
    batch = msd.Batch(ctxs)
    for o, v, e in batch.evaluate([pair, pair]):
        assert torch.equal(o, want[0])
        assert torch.allclose(v, want[1], rtol=1e-13 if precision == "fp64" else 1e-5, atol=0)
        assert torch.allclose(e, want[2], rtol=1e-12 if precision == "fp64" else 1e-6, atol=0)
    for c in ctxs:
        assert c.info("walker_chunk") == nw
    batch.close()
    for c in [ref, *ctxs]:
        c.close()


def test_constants_are_built_once_their_memory_can_be_had():
    """A propagation step beside which the tensor-core form of the Cholesky vectors does not
    fit runs without it; the next one, with memory free again, takes it."""
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, n, G, nw = 64, 6, 1500, 4                 # 64 x 64 rows of 1500: 47 MB, in FP64 form 96 MB
    s = synth.make_system(4, M, n, n, 2, 8, 20, 3, 1.0, G)
    w = synth.make_walkers(np.random.default_rng(1), M, n, n, nw)
    x = torch.from_numpy(np.random.default_rng(2).standard_normal((nw, G))).cuda()
    ctx = msd.Context(s, "fp64")

    def step():
        pa, pb = torch.from_numpy(w.phi_a).cuda(), torch.from_numpy(w.phi_b).cuda()
        wt = torch.ones(nw, dtype=torch.float64, device="cuda")
        before = msd.launch_count()
        ctx.propagate(pa, pb, wt, x, 0.01)
        return msd.launch_count() - before, pa, pb, wt

    step()
    launches, pa, pb, _ = step()
    again = msd.Context(s, "fp64")
    ctx.close()
    ctx = again
    # everything a step needs but the propagator's constants
    ctx.force_bias(pa, pb)
    ctx.overlap(pa, pb)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hog = torch.empty(free - (90 << 20), dtype=torch.uint8, device="cuda")
    step()                                       # its first launches on the side
    few = step()
    del hog
    torch.cuda.empty_cache()
    step()
    many = step()
    ctx.close()
    assert few[0] < launches and many[0] == launches
    for a, b in zip(few[1:], many[1:]):
        assert torch.allclose(a, b, rtol=1e-10, atol=1e-12)
