"""The density sample counts active inputs per step of the recording: rows whose last word holds few steps.  Word 1 of
the workspace holds the verdict (1: too dense); the lists of 1000 inputs hold 14 active ones per step."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("T, n, dense", [(20, 18, True), (32, 18, True), (33, 18, True), (20, 4, False), (40, 4, False)])
def test_steps_of_the_last_word(T, n, dense):
    from paper_2311_11390_gb300 import alif
    L, p = alif.lib(), lambda t: t.data_ptr()
    B, Nin, N = 1000, 1000, 1024
    S = torch.rand((B, Nin, T), device="cuda", generator=torch.Generator(device="cuda").manual_seed(T)) < n / Nin
    words, Wt, I = alif.pack_spikes(S.float()), torch.ones((Nin, N), device="cuda"), torch.empty((B, N, T), device="cuda")
    size = int(L.syn_project_events_workspace_size(B, Nin, N, T))
    assert size > 0
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    assert L.syn_project_events_ws(B, Nin, N, T, p(Wt), p(words), None, p(I), p(ws), size, torch.cuda.current_stream().cuda_stream) == 0
    assert int(ws[4:8].view(torch.int32)) == dense
    assert torch.equal(I, S.sum(1, dtype=torch.int32).float()[:, None].expand(B, N, T))  # whole numbers: exact


@cuda
@pytest.mark.parametrize("Nin, n, dense", [(1000, 8, False), (1000, 12, True), (512, 22, False), (512, 27, True)])
def test_rasters_that_overfill_the_lists(Nin, n, dense):
    """Counts spread about their mean: the lists hold 14 (30 at 512 inputs) with the padding, not on average."""
    from paper_2311_11390_gb300 import alif
    L, p = alif.lib(), lambda t: t.data_ptr()
    B, N, T = 32, 64, 4000
    words = alif.pack_spikes((torch.rand((B, Nin, T), device="cuda", generator=torch.Generator(device="cuda").manual_seed(n)) < n / Nin).float())
    Wt, I = torch.ones((Nin, N), device="cuda"), torch.empty((B, N, T), device="cuda")
    size = int(L.syn_project_events_workspace_size(B, Nin, N, T))
    assert size > 0
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    assert L.syn_project_events_ws(B, Nin, N, T, p(Wt), p(words), None, p(I), p(ws), size, torch.cuda.current_stream().cuda_stream) == 0
    assert int(ws[4:8].view(torch.int32)) == dense
    assert dense or int(ws[:4].view(torch.int32)) < B * ((T + 255) // 256) // 4  # most tiles by lists
