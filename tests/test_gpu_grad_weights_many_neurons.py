"""Weight and bias gradients of more neurons than 65535 tiles of 32 hold: each sum has a few terms, compared with
float64 within (terms) 2^-24 of the sum of their magnitudes."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("Nin", [1, 33])
def test_more_than_65535_tiles(Nin):
    from paper_2311_11390_gb300 import alif
    N, T = 2097153, 20
    assert alif.lib().syn_project_backward_lists_size(1, Nin, N, T) > 0
    g = torch.Generator(device="cuda").manual_seed(Nin)
    S = (torch.rand((1, Nin, T), device="cuda", generator=g) < 0.3).float()
    G = torch.randn((1, N, T), device="cuda", generator=g)
    gW, _, gb = alif.syn_project_backward(alif.pack_spikes(S), G, Nin=Nin)
    assert alif.device_status() == 0
    want, size = G[0].double() @ S[0].double().T, G[0].double().abs() @ S[0].double().T
    assert ((gW.double() - want).abs() <= T * 2.0 ** -24 * size).all()
    assert ((gb.double() - G[0].double().sum(1)).abs() <= T * 2.0 ** -24 * G[0].double().abs().sum(1)).all()
