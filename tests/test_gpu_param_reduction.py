"""The sum of the parameter gradients over the batch, at the edges of its blocks of 32 elements
(5 per neuron) and of its split of the batch."""
import numpy as np
import pytest
import torch

from paper_2311_11390_gb300 import synth

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B", [1, 2, 3, 31, 32, 33, 70])
@pytest.mark.parametrize("N", [1, 6, 7, 64])
def test_batch_sum_of_parameter_gradients(B, N):
    """Against the float64 sum of one-element calls: each of those is rounded once (2^-24), the
    batch's double-single sum once more.  The window length is fixed, so that both run the same
    backward kernel (its default depends on B N)."""
    from paper_2311_11390_gb300 import alif
    w = synth.population(seed=B, B=B, N=N, T=96)
    p = w.params
    table = alif.neuron_table(p.tau_mem, p.tau_adapt, p.theta0, p.d, p.R, w.dt, w.arp)
    I = torch.from_numpy(w.I).cuda()
    out = alif.forward(I, table)
    gS = torch.randn(I.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    before = alif.backward_window(256)
    gp = alif.backward(I, table, out["spikes"], gS, ckpt=out["ckpt"])[2].double().cpu().numpy()
    one = np.stack([alif.backward(I[b:b + 1], table, out["spikes"][b:b + 1], gS[b:b + 1], ckpt=out["ckpt"][b:b + 1])[2]
                    .double().cpu().numpy() for b in range(B)])
    alif.backward_window(before)
    u = 2.0 ** -24
    assert (np.abs(gp - one.sum(0)) <= u * (1 + 1e-6) * (np.abs(one).sum(0) + np.abs(one.sum(0)))).all()
