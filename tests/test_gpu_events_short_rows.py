"""The event projection of short rows whose tiles are too dense for the lists: their chunks are spread over all CTAs
(as a time: no more than twice that of the entry without lists, it was seven times), against float64."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


def _time(f):
    f()
    best = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            f()
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b))
    return min(best)


@cuda
def test_dense_tiles_of_short_rows():
    from paper_2311_11390_gb300 import alif
    L, p = alif.lib(), lambda t: t.data_ptr()
    B, Nin, N, T = 1000, 1000, 1024, 32
    g = torch.Generator(device="cuda").manual_seed(1)
    S = torch.zeros((B, Nin, T), device="cuda")
    busy = torch.randperm(B, device="cuda", generator=g)[:400]
    S[busy, 500:518] = 1.0  # 18 active inputs a step there, more than a list holds, and 7 on average
    words, Wt = alif.pack_spikes(S), torch.randn((Nin, N), device="cuda", generator=g)
    size = int(L.syn_project_events_workspace_size(B, Nin, N, T))
    assert size > 0
    I, ws, st = torch.empty((B, N, T), device="cuda"), torch.empty(size, dtype=torch.uint8, device="cuda"), torch.cuda.current_stream().cuda_stream
    with_lists = _time(lambda: L.syn_project_events_ws(B, Nin, N, T, p(Wt), p(words), None, p(I), p(ws), size, st))
    assert int(ws[4:8].view(torch.int32)) == 0 and int(ws[:4].view(torch.int32)) == 400  # tiles over capacity
    want = torch.einsum("jn,bjt->bnt", Wt.double(), S.double())
    mag = torch.einsum("jn,bjt->bnt", Wt.double().abs(), S.double())
    assert ((I.double() - want).abs() <= 20 * 2.0 ** -24 * mag).all()
    without = _time(lambda: L.syn_project_events(B, Nin, N, T, p(Wt), p(words), None, p(I), st))
    assert with_lists <= 2 * without, (with_lists, without)
