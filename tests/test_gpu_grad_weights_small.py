"""Weight and bias gradients by lists where one batch element's steps are long or the neurons' tiles many for
the product: few inputs and neurons, several batch elements, partial words and windows.  Bounds as for the
other sizes: a sum of m FP32 terms within m 2^-24 of the sum of their magnitudes (m: at most the spikes of an
input over the call and the partials joined)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B, Nin, N, T", [(1, 1, 1, 6000), (1, 40, 33, 16001), (2, 300, 17, 6145), (40, 64, 65, 7000),
                                          (3, 1024, 130, 18500), (130, 33, 257, 900)])
@pytest.mark.parametrize("rate", [0.002, 0.03])
def test_small_weight_gradients_by_lists(B, Nin, N, T, rate):
    from paper_2311_11390_gb300 import alif
    assert alif.lib().syn_project_backward_lists_size(B, Nin, N, T) > 0
    g = torch.Generator(device="cuda").manual_seed(Nin + T)
    S = (torch.rand((B, Nin, T), device="cuda", generator=g) < rate).float()
    G = torch.randn((B, N, T), device="cuda", generator=g)
    gW, _, gb = alif.syn_project_backward(alif.pack_spikes(S), G, Nin=Nin)
    assert alif.device_status() == 0
    want = torch.einsum("bit,bjt->ij", G.double(), S.double())
    size = torch.einsum("bit,bjt->ij", G.double().abs(), S.double())
    m = S.double().sum((0, 2)) + B * ((T + 511) // 512) + 64
    assert ((gW.double() - want).abs() <= m * 2.0 ** -24 * size + 1e-30).all()
    g64 = G.double()
    assert ((gb.double() - g64.sum((0, 2))).abs() <= (T + B + 100) * 2.0 ** -24 * g64.abs().sum((0, 2)) + 1e-30).all()
