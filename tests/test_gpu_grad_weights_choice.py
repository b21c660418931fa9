"""Weight gradients of few neurons: which sizes take the lists (where both ways were timed), and one tile of neurons
over more ranges of units than 64, against float64 within (terms) 2^-24 of the sum of their magnitudes."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("size, lists", [((152, 60, 12, 7000), False), ((249, 186, 16, 4105), False), ((76, 256, 32, 6100), False),
                                         ((38, 700, 64, 6144), False), ((600, 120, 15, 2000), True), ((337, 18, 4, 3366), True),
                                         ((174, 342, 24, 3694), True), ((1, 40, 33, 16001), True)])
def test_choice(size, lists):
    from paper_2311_11390_gb300 import alif
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("timed on 152 SMs")
    assert (alif.lib().syn_project_backward_lists_size(*size) > 0) == lists


@cuda
def test_one_tile_over_many_ranges():
    from paper_2311_11390_gb300 import alif
    B, Nin, N, T = 600, 120, 15, 2000
    assert alif.lib().syn_project_backward_lists_size(B, Nin, N, T) > 0
    g = torch.Generator(device="cuda").manual_seed(5)
    S = (torch.rand((B, Nin, T), device="cuda", generator=g) < 0.01).float()
    G = torch.randn((B, N, T), device="cuda", generator=g)
    gW, _, gb = alif.syn_project_backward(alif.pack_spikes(S), G, Nin=Nin)
    assert alif.device_status() == 0
    want, mag = (sum(f(G[b].double()) @ S[b].double().T for b in range(B)) for f in (lambda x: x, torch.abs))
    m = S.double().sum((0, 2)) + B * 4 + 152
    assert ((gW.double() - want).abs() <= m * 2.0 ** -24 * mag + 1e-30).all()
    g64 = G.double()
    assert ((gb.double() - g64.sum((0, 2))).abs() <= (T + B + 200) * 2.0 ** -24 * g64.abs().sum((0, 2)) + 1e-30).all()
