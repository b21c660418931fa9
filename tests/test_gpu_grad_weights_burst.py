"""Weight and bias gradients of rasters that are sparse but for single 512-step units, whose lists do not fit,
over more CTAs of the lists kernel than run at a time: the blocks that start after such a unit was found take
the same decisions as those before it.  Bounds: a sum of m FP32 terms within m 2^-24 of the sum of their
magnitudes (m: an input's spikes and the partials joined)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("bursts", [((0, 0),), ((0, 3), (5, 700), (63, 16383))], ids=["first", "several"])
@pytest.mark.parametrize("Nin", [64, 515])
def test_units_over_capacity_in_several_waves(bursts, Nin):
    from paper_2311_11390_gb300 import alif
    B, N, T = 64, 35, 16384  # 1024 CTAs of two units; two fit an SM
    assert alif.lib().syn_project_backward_lists_size(B, Nin, N, T) > 0
    g = torch.Generator(device="cuda").manual_seed(Nin)
    S = (torch.rand((B, Nin, T), device="cuda", generator=g) < 0.002).float()
    for b, t in bursts:  # every input in every step: more than 2047 rows of 8 spikes
        S[b, :, t // 512 * 512:t // 512 * 512 + 512] = 1.0
    G = torch.randn((B, N, T), device="cuda", generator=g)
    words = alif.pack_spikes(S)
    gW, _, gb = alif.syn_project_backward(words, G, Nin=Nin)
    for _ in range(3):
        again = alif.syn_project_backward(words, G, Nin=Nin)
        assert torch.equal(gW, again[0]) and torch.equal(gb, again[2])
    assert alif.device_status() == 0
    want, size = (sum(f(G[b].double()) @ S[b].double().T for b in range(B)) for f in (lambda x: x, torch.abs))
    m = S.double().sum((0, 2)) + B * (T // 512) + 64
    assert ((gW.double() - want).abs() <= m * 2.0 ** -24 * size + 1e-30).all()
    g64 = G.double()
    assert ((gb.double() - g64.sum((0, 2))).abs() <= (T + B + 100) * 2.0 ** -24 * g64.abs().sum((0, 2)) + 1e-30).all()
