"""The event projection of an odd number of neurons (one per thread) over large products: rasters judged dense as a
whole, with dense tiles only, and sparse, against float64 within (k + 1) 2^-24 of the sum of magnitudes."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("what", ["dense", "tiles", "sparse"])
@pytest.mark.parametrize("B, Nin, N, T", [(40, 700, 1023, 900), (31, 1000, 515, 1401)])
def test_odd_neurons(B, Nin, N, T, what):
    from paper_2311_11390_gb300 import alif
    assert alif.lib().syn_project_events_workspace_size(B, Nin, N, T) > 0
    g = torch.Generator(device="cuda").manual_seed(N)
    S = (torch.rand((B, Nin, T), device="cuda", generator=g) < (0.1 if what == "dense" else 0.002)).float()
    if what == "tiles":
        S[1, :200, 256:700], S[B - 1, :, T - 3:] = 1.0, 1.0
    W, bias = torch.randn((N, Nin), device="cuda", generator=g), torch.randn(N, device="cuda", generator=g)
    I = alif.syn_project_events(alif.pack_spikes(S), alif.transpose_weights(W), bias, Nin=Nin, T=T)
    assert alif.device_status() == 0
    for b in range(B):
        want = W.double() @ S[b].double() + bias.double()[:, None]
        mag = W.double().abs() @ S[b].double() + bias.double().abs()[:, None]
        assert ((I[b].double() - want).abs() <= (S[b].double().sum(0) + 1) * 2.0 ** -24 * mag).all()
