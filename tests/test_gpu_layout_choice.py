"""The layout alif_forward chooses by itself on both sides of its lines: its states are, bit for bit, those of the
named layout (the layouts' states differ in rounding)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("per_sm, T, lanes", [(31, 100, False), (33, 100, True), (33, 36, True), (33, 180, False), (54, 180, True),
                                              (54, 184, False), (79, 400, False), (81, 400, True)])
def test_layout_by_rows_and_steps(per_sm, T, lanes):
    from paper_2311_11390_gb300 import alif
    N = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator().manual_seed(T)
    r = lambda lo, hi: (lo + (hi - lo) * torch.rand(N, generator=g)).numpy()  # noqa: E731
    table = alif.neuron_table(r(10, 30), r(100, 500), r(1, 1), r(0, 0.2), dt_ms=0.1, arp_ms=2.0)
    I = (1.5 + torch.randn((1, N, T), generator=g)).cuda()
    states = {}
    for layout in (0, 1, 2):
        before = alif.forward_layout(layout)
        states[layout] = alif.forward(I, table)["final"]
        alif.forward_layout(before)
    assert alif.device_status() == 0
    assert torch.equal(states[0], states[2 if lanes else 1]) and not torch.equal(states[1], states[2])
