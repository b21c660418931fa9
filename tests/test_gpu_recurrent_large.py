"""The recurrent layer of more than 256 neurons a CTA with more spikes in a Block than weight slots: units of 4, 2 and 1
steps, weight rows that do and do not keep 16 bytes, a last partial Block: the total current against float64, the spikes
against the block forward on it."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("B, N, T, arp", [(1, 2100, 300, 2.0), (2, 2101, 302, 1.0), (1, 4097, 133, 2.0), (1, 6000, 90, 1.0),
                                          (1, 8192, 61, 0.5), (1, 3000, 300, 6.0)])
def test_recurrent_many_neurons(B, N, T, arp):
    """A total current is I_ff plus at most N weights summed in double-single and rounded once."""
    from paper_2311_11390_gb300 import alif
    g = torch.Generator(device="cuda").manual_seed(T)
    u = lambda lo, hi: (lo + (hi - lo) * torch.rand(N, generator=g, device="cuda")).cpu().numpy()  # noqa: E731
    table = alif.neuron_table(u(10, 30), u(100, 500), u(1, 1), u(0, 0.02), dt_ms=0.1, arp_ms=arp)
    I = 8.0 + torch.randn((B, N, T), generator=g, device="cuda")
    W = torch.randn((N, N), generator=g, device="cuda") / N ** 0.5
    out = alif.forward_recurrent(I, alif.transpose_weights(W), table, 0.1, arp)
    assert alif.device_status() == 0
    TR = alif.tr(0.1, arp)
    S = alif.spikes_to_float(out["spikes"], T).double()
    blocks = S[:, :, :T // TR * TR].reshape(B, N, -1, TR).sum((1, 3))
    assert blocks.max() > 128
    late = torch.nn.functional.pad(S, (TR, 0))[:, :, :T]
    ref = I.double() + torch.einsum("ij,bjt->bit", W.double(), late)
    mag = I.double().abs() + torch.einsum("ij,bjt->bit", W.double().abs(), late)
    assert ((out["I_total"].double() - ref).abs() <= 2.0 ** -24 * ref.abs() + (N + 2) * 2.0 ** -46 * mag).all()
    again = alif.forward(out["I_total"], table)
    assert torch.equal(again["spikes"], out["spikes"])
