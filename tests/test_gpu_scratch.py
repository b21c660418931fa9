"""Calls whose event lists no longer fit on the device run without them, as the entries without a workspace do:
the same bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
def test_calls_without_room_for_lists(monkeypatch):
    from paper_2311_11390_gb300 import alif
    B, Nin, N, T = 16, 512, 1024, 8000
    L, stream = alif.lib(), torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device="cuda").manual_seed(3)
    S = alif.pack_spikes((torch.rand((B, Nin, T), device="cuda", generator=g) < 0.003).float())
    W = torch.randn((N, Nin), device="cuda", generator=g)
    bias, G = torch.randn(N, device="cuda", generator=g), torch.randn((B, N, T), device="cuda", generator=g)
    hi, lo = alif.split_bf16(W)
    Wt = alif.transpose_weights(W)
    sizes = (L.syn_project_workspace_size(B, Nin, N, T), L.syn_project_events_workspace_size(B, Nin, N, T),
             L.syn_project_backward_lists_size(B, Nin, N, T))
    assert all(n > 0 for n in sizes)
    p = lambda t: t.data_ptr()  # noqa: E731
    I, J = torch.empty((B, N, T), device="cuda"), torch.empty((B, N, T), device="cuda")
    gW, gb = torch.empty((N, Nin), device="cuda"), torch.empty(N, device="cuda")
    need = int(L.syn_project_backward_workspace_size(B, N, Nin))
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    assert L.syn_project(B, Nin, N, T, p(hi), p(lo), hi.shape[1], p(S), p(bias), p(I), stream) == 0
    assert L.syn_project_events(B, Nin, N, T, p(Wt), p(S), p(bias), p(J), stream) == 0
    assert L.syn_project_backward(B, Nin, N, T, None, p(S), p(G), p(gW), None, p(gb), p(ws), need, stream) == 0
    empty = torch.empty

    def full(*args, **kw):  # a device without room for the lists
        if args and args[0] in sizes and kw.get("dtype") == torch.uint8:
            raise torch.cuda.OutOfMemoryError("out of memory")
        return empty(*args, **kw)

    monkeypatch.setattr(torch, "empty", full)
    assert torch.equal(alif.syn_project(S, hi, lo, bias, Nin=Nin, T=T), I)
    assert torch.equal(alif.syn_project_events(S, Wt, bias, Nin=Nin, T=T), J)
    gW2, _, gb2 = alif.syn_project_backward(S, G, Nin=Nin)
    assert torch.equal(gW2, gW) and torch.equal(gb2, gb)
    assert alif.device_status() == 0
