"""An expired device wait in the FP64 contractions on the tensor cores: with a budget of
0 a wait is one poll, the kernel stops its pipeline and returns, the call reports
MSD_ERR_TIMEOUT, and the context then gives the values it gave before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["local_energy", "force_bias"])
def test_expired_wait_and_recovery(call):
    import torch

    from paper_2406_08314_gb300 import msd, synth
    M, n, G, nw = 64, 20, 120, 40               # reference product, F, Gram matrices and force bias
    s = synth.make_system(2, M, n, n, 14, 12, 60, 4, 1.0, G)
    w = synth.make_walkers(np.random.default_rng(3), M, n, n, nw)
    dev = [torch.from_numpy(x).cuda() for x in (w.phi_a, w.phi_b)]
    ctx = msd.Context(s, "fp64")
    fn = getattr(ctx, call)
    first = fn(*dev)
    ctx.set_wait_budget(0)
    codes = set()
    for _ in range(3):
        try:
            fn(*dev)
            codes.add("ok")
        except msd.MSDError as e:
            codes.add(e.name)
    assert "MSD_ERR_TIMEOUT" in codes and codes <= {"ok", "MSD_ERR_TIMEOUT"}, codes
    ctx.set_wait_budget(2_000_000_000)
    assert torch.equal(fn(*dev), first)
    ctx.close()
