"""The event projection where the chunks of a raster are many for its neurons: one to a few hundred neurons
(not a multiple of 4 or of 32), few and many inputs, partial words, an input that always spikes.  Bound: k
active inputs are summed within (k + 1) 2^-24 (|bias| + sum |W| S)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B, Nin, N, T", [(12, 33, 1, 1000), (13, 64, 3, 1001), (20, 100, 65, 700), (9, 1000, 130, 1999),
                                          (40, 7, 300, 515), (25, 1, 128, 800)])
@pytest.mark.parametrize("rate", [0.002, 0.05])
def test_small_event_projection_by_lists(B, Nin, N, T, rate):
    from paper_2311_11390_gb300 import alif
    assert alif.lib().syn_project_events_workspace_size(B, Nin, N, T) > 0
    g = torch.Generator(device="cuda").manual_seed(Nin + T)
    S = (torch.rand((B, Nin, T), device="cuda", generator=g) < rate).float()
    S[:, 0] = 1.0
    W = torch.randn((N, Nin), device="cuda", generator=g)
    bias = torch.randn((N,), device="cuda", generator=g)
    I = alif.syn_project_events(alif.pack_spikes(S), alif.transpose_weights(W), bias, Nin=Nin, T=T)
    assert alif.device_status() == 0
    want = torch.einsum("ij,bjt->bit", W.double(), S.double()) + bias.double()[:, None]
    size = torch.einsum("ij,bjt->bit", W.double().abs(), S.double()) + bias.double().abs()[:, None]
    k = S.double().sum(1, keepdim=True)
    assert ((I.double() - want).abs() <= (k + 1) * 2.0 ** -24 * size).all()
