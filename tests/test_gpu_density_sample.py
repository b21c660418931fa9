"""The sample that chooses between lists and the dense kernels looks at all of a raster's time: rasters whose
density varies in time, at sizes whose words are a multiple of the sample's 4096.  Word 1 of a workspace holds
the verdict (1: too dense)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


def _raster(B, Nin, T, what):
    g = torch.Generator(device="cuda").manual_seed(T)
    S = (torch.rand((B, Nin, T), device="cuda", generator=g) < (0.002 if what == "onset" else 0.3)).float()
    S[:, :, :32] = 1.0 if what == "onset" else 0.0  # all of it in the first word, or none of it
    return S


def _zeros(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


@cuda
@pytest.mark.parametrize("what", ["onset", "late"])
@pytest.mark.parametrize("B, Nin, N, T", [(128, 256, 256, 1000), (64, 512, 64, 4096), (610, 33, 64, 1024)])
def test_weight_gradients(B, Nin, N, T, what):
    from paper_2311_11390_gb300 import alif
    L, p = alif.lib(), lambda t: t.data_ptr()
    S = _raster(B, Nin, T, what)
    G = torch.randn((B, N, T), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    words = alif.pack_spikes(S)
    gW, gb = torch.empty((N, Nin), device="cuda"), torch.empty(N, device="cuda")
    need, size = L.syn_project_backward_workspace_size(B, N, Nin), L.syn_project_backward_lists_size(B, Nin, N, T)
    assert size > 0
    ws, lists = _zeros(need), _zeros(size)
    assert L.syn_project_backward_ws(B, Nin, N, T, None, p(words), p(G), p(gW), None, p(gb), p(ws), need, p(lists), size,
                                     torch.cuda.current_stream().cuda_stream) == 0
    assert int(lists[4:8].view(torch.int32)) == (what == "late" and Nin > 33)  # 33 inputs fit at any density
    want, mag = (sum(f(G[b].double()) @ S[b].double().T for b in range(B)) for f in (lambda x: x, torch.abs))
    m = S.double().sum((0, 2)) + B * ((T + 511) // 512) + 64
    assert ((gW.double() - want).abs() <= m * 2.0 ** -24 * mag + 1e-30).all()


@cuda
@pytest.mark.parametrize("what", ["onset", "late"])
@pytest.mark.parametrize("B, Nin, N, T", [(32, 1024, 128, 16384), (64, 512, 512, 4096)])
def test_projection(B, Nin, N, T, what):
    from paper_2311_11390_gb300 import alif
    L, p = alif.lib(), lambda t: t.data_ptr()
    words = alif.pack_spikes(_raster(B, Nin, T, what))
    hi, lo = alif.split_bf16(torch.randn((N, Nin), device="cuda", generator=torch.Generator(device="cuda").manual_seed(2)))
    I = torch.empty((B, N, T), device="cuda")
    size = L.syn_project_workspace_size(B, Nin, N, T)
    assert size > 0
    ws = _zeros(size)
    assert L.syn_project_ws(B, Nin, N, T, p(hi), p(lo), hi.shape[1], p(words), None, p(I), p(ws), size,
                            torch.cuda.current_stream().cuda_stream) == 0
    assert int(ws[4:8].view(torch.int32)) == (what == "late")
