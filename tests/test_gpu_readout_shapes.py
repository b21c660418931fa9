"""The readout, its gradients and the loss where their warps' and blocks' shares change: one to a few
outputs, inputs and batch elements around 32, partial words.  Bounds: each sum of m FP32 terms within
(m + 2) 2^-24 of the sum of their magnitudes; the loss within 2^-24 (3 R + C + 16) and its gradient
2^-24 (R + C + 24) / B for logits R apart (expf and logf within 2 ulp)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B, K, C, T", [(1, 1, 1, 1), (31, 33, 20, 33), (32, 31, 33, 64), (33, 256, 10, 1001),
                                        (130, 64, 35, 100), (2, 500, 64, 1027)])
def test_readout_shapes(B, K, C, T):
    from paper_2311_11390_gb300 import alif
    g = torch.Generator(device="cuda").manual_seed(B + K)
    S = (torch.rand((B, K, T), device="cuda", generator=g) < 0.1).float()
    W = torch.randn((C, K), device="cuda", generator=g)
    bias = torch.randn((C,), device="cuda", generator=g)
    y = torch.randint(0, C, (B,), device="cuda", generator=g, dtype=torch.int32)
    w, w_sum = alif.readout_weights(T, 1.0, 20.0, "cuda")
    u = 2.0 ** -24
    o, n = alif.readout_forward(alif.pack_spikes(S), T, W, bias, w, w_sum)
    nr = (S.double() * w.double()).sum(-1)
    assert ((n.double() - nr).abs() <= (T + 2) * u * nr).all()
    size = nr @ W.double().abs().T + bias.double().abs() * w_sum
    assert ((o.double() - (nr @ W.double().T + bias.double() * w_sum)).abs() <= (T + K + 6) * u * size).all()
    loss, go = alif.cross_entropy(o, y)
    lr = torch.nn.functional.cross_entropy(o.double(), y.long())
    R = float((o.max(1).values - o.min(1).values).max())
    assert abs(float(loss) - float(lr)) <= u * (3 * R + C + 16) + u * abs(float(lr))
    gr = (torch.softmax(o.double(), 1) - torch.nn.functional.one_hot(y.long(), C)) / B
    assert ((go.double() - gr).abs() <= u * (R + C + 24) / B).all()
    gS, gW, gb = alif.readout_backward(W, w, w_sum, n, go, T)
    h = go.double() @ W.double()
    assert ((gS.double() - h[..., None] * w.double()).abs()
            <= (C + 3) * u * (go.double().abs() @ W.double().abs())[..., None] * w.double() + 1e-40).all()
    assert ((gW.double() - go.double().T @ n.double()).abs() <= (B + 2) * u * (go.double().abs().T @ n.double()) + 1e-40).all()
    assert ((gb.double() - go.double().sum(0) * w_sum).abs() <= (B + 3) * u * go.double().abs().sum(0) * w_sum + 1e-40).all()
