"""The readout and its gradient over rows of more than 128 words, few enough that a row's gradient is written in
several parts: whole and partial words, rows on and off the 16-byte grid, parts of 512 steps and more.  Bounds as
for the other shapes: a sum of m FP32 terms within (m + 2) 2^-24 of the sum of their magnitudes."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B, K, C, T", [(1, 1, 2, 513), (1, 1, 11, 1024), (2, 3, 20, 20000), (1, 5, 10, 20003), (3, 129, 7, 9998),
                                        (61, 79, 3, 5004), (8, 608, 2, 4100)])
def test_long_rows(B, K, C, T):
    from paper_2311_11390_gb300 import alif
    g = torch.Generator(device="cuda").manual_seed(T)
    S = (torch.rand((B, K, T), device="cuda", generator=g) < 0.05).float()
    W, bias = torch.randn((C, K), device="cuda", generator=g), torch.randn((C,), device="cuda", generator=g)
    w, w_sum = alif.readout_weights(T, 0.1, 20.0, "cuda")
    u = 2.0 ** -24
    o, n = alif.readout_forward(alif.pack_spikes(S), T, W, bias, w, w_sum)
    nr = (S.double() * w.double()).sum(-1)
    assert ((n.double() - nr).abs() <= (T + 2) * u * nr).all()
    size = nr @ W.double().abs().T + bias.double().abs() * w_sum
    assert ((o.double() - (nr @ W.double().T + bias.double() * w_sum)).abs() <= (T + K + 6) * u * size).all()
    go = torch.randn((B, C), device="cuda", generator=g)
    gS, gW, gb = alif.readout_backward(W, w, w_sum, n, go, T)
    h = go.double() @ W.double()
    assert ((gS.double() - h[..., None] * w.double()).abs()
            <= (C + 3) * u * (go.double().abs() @ W.double().abs())[..., None] * w.double() + 1e-40).all()
    assert ((gW.double() - go.double().T @ n.double()).abs() <= (B + 2) * u * (go.double().abs().T @ n.double()) + 1e-40).all()
    only, _, _ = alif.readout_backward(W, w, w_sum, n, go, T, want_W=False, want_bias=False)
    assert torch.equal(only, gS)
