"""Every quantity but the overlap is invariant under a scaling of the walker's columns,
as it is under any phi -> phi R (walkers propagated without re-orthonormalisation have
columns of different norms). One spin's reference product runs on the
tensor cores, the other's does not."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [0, 10, 30, 50])
def test_column_scale(bits):
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, na, nb, nw = 64, 20, 18, 3        # (M - N) N^2 = 17600, 14904
    s = synth.make_system(5, M, na, nb, 15, 12, 80, 4, 0.7, 40)
    w = synth.make_walkers(np.random.default_rng(1), M, na, nb, nw, noise=0.4)
    rng = np.random.default_rng(bits)
    scaled = [phi * 2.0 ** -rng.permutation(np.round(np.linspace(0, bits, phi.shape[2]))) for phi in (w.phi_a, w.phi_b)]
    base = [torch.from_numpy(x).cuda() for x in (w.phi_a, w.phi_b)]
    other = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in scaled]
    # powers of two scale FP64 exactly but for the pivots' reciprocals (an ulp each):
    # FP64 rounding; mixed: the same through FP32 inputs, the parity bounds
    for prec, tol, tol_v in (("fp64", 1e-12, 1e-12), ("mixed", 2e-6, 1e-4)):
        ctx = msd.Context(s, prec)
        want, got = [], []
        for out, phi in ((want, base), (got, other)):
            _, v, e = ctx.evaluate(*phi)
            out += [x.cpu().numpy() for x in (e, v, ctx.det_ratios(*phi), ctx.rdm1(*phi))]
        ctx.close()
        canc = np.abs(want[2] * s.coeff).sum(1) / np.abs((want[2] * s.coeff).sum(1))
        scale_e = canc * np.abs(want[0]).max()
        assert np.all(np.abs(got[0] - want[0]) <= tol * scale_e), prec
        for a, b, t in ((got[1], want[1], tol_v), (got[2], want[2], 1e-12), (got[3], want[3], tol_v)):
            assert np.abs(a - b).max() <= t * canc.max() * np.abs(b).max(), prec
