"""A batch whose recorded graph has become stale: after a set-up call on one of its contexts
that fails, the batch reports that the trial is missing instead of replaying, and after a
valid one it gives the values of the new trial."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_failed_trial(precision):
    import torch

    from paper_2406_08314_gb300 import msd, synth
    s, w = synth.config_system("small", seed=0)
    other, _ = synth.config_system("small", seed=1)
    pair = tuple(torch.from_numpy(x).cuda() for x in (w.phi_a, w.phi_b))
    ctx, one = msd.Context(s, precision), msd.Context(s, precision)
    batch = msd.Batch([ctx])
    outs = batch.outputs([pair])
    batch.evaluate([pair], outs)
    assert batch.graph_ready()
    bad = s.occ_a.copy()
    bad[3] = bad[3, ::-1]
    with pytest.raises(msd.MSDError):
        ctx.set_trial(s.coeff, bad, s.occ_b)
    with pytest.raises(msd.MSDError) as err:
        batch.evaluate([pair], outs)
    assert err.value.name == "MSD_ERR_STATE"
    ctx.set_trial(other.coeff, other.occ_a, other.occ_b)
    one.set_trial(other.coeff, other.occ_a, other.occ_b)
    one.set_pair_form(0)
    for _ in (0, 1):
        o, v, e = batch.evaluate([pair], outs)[0]
    want = one.evaluate(*pair)
    assert torch.equal(o, want[0]) and torch.equal(v, want[1])
    # the batched kernel sums the same terms, in another order in FP64
    assert np.allclose(e.cpu().numpy(), want[2].cpu().numpy(), rtol=1e-12, atol=0)
    batch.close()
    ctx.close()
    one.close()
