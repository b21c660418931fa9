"""Weight gradients where single 512-step units hold more spikes than their lists: those units are walked, the
others keep their lists, and every weight's additions are the same in the same order -- so that bits can be
compared: with a raster without the burst (dL/dI zero there) and with one whose unit does fit."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


def _grad(S, G):
    from paper_2311_11390_gb300 import alif
    assert alif.lib().syn_project_backward_lists_size(S.shape[0], S.shape[1], G.shape[1], S.shape[2]) > 0
    gW, _, gb = alif.syn_project_backward(alif.pack_spikes(S), G, Nin=S.shape[1])
    assert alif.device_status() == 0
    return gW, gb


@cuda
@pytest.mark.parametrize("Nin, N, T", [(64, 35, 16384), (515, 64, 16200), (1024, 65, 16001)])
@pytest.mark.parametrize("unit", ["first", "last"])
def test_unit_over_capacity(Nin, N, T, unit):
    B = 40
    g = torch.Generator(device="cuda").manual_seed(Nin)
    S = (torch.rand((B, Nin, T), device="cuda", generator=g) < 0.004).float()
    G = torch.randn((B, N, T), device="cuda", generator=g)
    b, t = (0, 0) if unit == "first" else (B - 1, (T - 1) // 512 * 512)
    burst = S.clone()
    burst[b, :, t:t + 512] = 1.0
    burst[b, 3::4, t:t + 512] = S[b, 3::4, t:t + 512]  # every fourth input as it was
    gW, gb = _grad(burst, G)
    rest, _ = _grad(S, G)
    assert torch.equal(gW[:, 3::4], rest[:, 3::4])  # its sums from the walk are those from the list
    want, mag = (sum(f(G[k].double()) @ burst[k].double().T for k in range(B)) for f in (lambda x: x, torch.abs))
    m = burst.double().sum((0, 2)) + B * ((T + 511) // 512) + 64
    assert ((gW.double() - want).abs() <= m * 2.0 ** -24 * mag + 1e-30).all()
    G[b, :, t:t + 512] = 0.0
    assert torch.equal(_grad(burst, G)[0], _grad(S, G)[0])  # the other units keep their lists
