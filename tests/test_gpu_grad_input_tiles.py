"""The projection's input gradient at the edges of its tiles: 128 inputs per accumulator, two of them per
tile, 128 steps, slabs of 64 neurons, rows that are not 16-byte aligned.  The bound is the kernel's own:
sum_i |W_ij| |G_i| (3 * 2^-16 + (3 N + 2) 2^-24)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B, Nin, N, T", [(1, 1, 1, 1), (2, 127, 63, 127), (2, 128, 64, 128), (3, 129, 65, 129),
                                          (1, 255, 31, 255), (2, 256, 33, 256), (2, 257, 96, 130), (1, 384, 128, 36),
                                          (1, 385, 191, 1001), (170, 40, 32, 33)])
def test_input_gradient_at_tile_edges(B, Nin, N, T):
    from paper_2311_11390_gb300 import alif
    g = torch.Generator(device="cuda").manual_seed(Nin + T)
    W = torch.randn((N, Nin), device="cuda", generator=g)
    G = torch.randn((B, N, T), device="cuda", generator=g)
    words = torch.zeros((B, Nin, (T + 31) // 32), dtype=torch.int32, device="cuda")
    gS = alif.syn_project_backward(words, G, W=W, want_gW=False, want_gS=True, want_gb=False)[1]
    assert alif.device_status() == 0
    want = torch.einsum("ij,bit->bjt", W.double(), G.double())
    size = torch.einsum("ij,bit->bjt", W.double().abs(), G.double().abs())
    assert ((gS.double() - want).abs() <= size * (3 * 2.0 ** -16 + (3 * N + 2) * 2.0 ** -24)).all()
