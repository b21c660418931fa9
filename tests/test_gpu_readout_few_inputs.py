"""The readout's outputs from few inputs (a thread per output) and around the lines to a warp per output: within
(terms + 2) 2^-24 of the sum of their magnitudes."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B, K, C", [(1, 1, 1), (300, 3, 75), (130, 12, 7), (130, 13, 7), (2000, 16, 5), (1000, 24, 11), (1000, 25, 11)])
@pytest.mark.parametrize("with_bias", [True, False])
def test_few_inputs(B, K, C, with_bias):
    from paper_2311_11390_gb300 import alif
    T, u = 100, 2.0 ** -24
    g = torch.Generator(device="cuda").manual_seed(K)
    S = (torch.rand((B, K, T), device="cuda", generator=g) < 0.1).float()
    W = torch.randn((C, K), device="cuda", generator=g)
    bias = torch.randn((C,), device="cuda", generator=g) if with_bias else None
    w, w_sum = alif.readout_weights(T, 1.0, 20.0, "cuda")
    o, n = alif.readout_forward(alif.pack_spikes(S), T, W, bias, w, w_sum)
    b64 = bias.double() * w_sum if with_bias else torch.zeros(C, dtype=torch.float64, device="cuda")
    size = n.double() @ W.double().abs().T + b64.abs()
    assert ((o.double() - (n.double() @ W.double().T + b64)).abs() <= (K + 4) * u * size).all()
