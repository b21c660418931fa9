"""Weight and bias gradients over event lists (products large enough to take that path): partial
neuron tiles, chunks and words, rows that do and do not keep 16 bytes, the most inputs, an input
active in every step, units at and over a list's capacity, empty and dense rasters -- against the
float64 sums."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
EPS = 2.0 ** -24


def _check(alif, S, gI):
    """A weight's terms pass at most the spikes of a 512-step unit, the units and the 64 ranges in
    sequence; a bias's the units, 4 steps of a load, 8 lanes, 16 warps and the ranges."""
    B, Nin, T = S.shape
    N = gI.shape[1]
    assert alif.lib().syn_project_backward_lists_size(B, Nin, N, T) > 0
    gW, _, gb = alif.syn_project_backward(alif.pack_spikes(S), gI, Nin=Nin)
    gW2, _, none = alif.syn_project_backward(alif.pack_spikes(S), gI, Nin=Nin, want_gb=False)
    assert none is None and torch.equal(gW, gW2)
    ref, mag = torch.zeros((N, Nin), dtype=torch.float64, device="cuda"), torch.zeros((N, Nin), dtype=torch.float64, device="cuda")
    for b in range(B):
        Sb, g = S[b].double(), gI[b].double()
        ref += g @ Sb.T
        mag += g.abs() @ Sb.T
    units = B * -(-T // 512)
    pad = torch.nn.functional.pad(S, (0, -T % 512)).reshape(B, Nin, -1, 512).sum(-1)
    chain = pad.amax((0, 2))  # spikes of an input in its busiest unit
    # the kernel without lists: a chain of all spikes of an input in a batch element, then the batch
    chain = torch.maximum(S.sum(-1).amax(0) + B, chain + units + 64)
    assert ((gW.double() - ref).abs() <= chain.double() * EPS * mag + 1e-30).all()
    g64 = gI.double()
    assert ((gb.double() - g64.sum((0, 2))).abs() <= (T + B + 100) * EPS * g64.abs().sum((0, 2)) + 1e-30).all()


def _make(seed, B, Nin, N, T, p):
    g = torch.Generator(device="cuda").manual_seed(seed)
    S = (torch.rand((B, Nin, T), generator=g, device="cuda") < p).float()
    return S, torch.randn((B, N, T), generator=g, device="cuda")


@cuda
@pytest.mark.parametrize("B, Nin, N, T, p", [(44, 1000, 256, 2048, 0.003), (31, 1024, 500, 1537, 0.003), (31, 33, 1000, 8002, 0.03),
                                             (1000, 256, 33, 1000, 0.008), (64, 700, 17, 25001, 0.004), (720, 1000, 64, 512, 0.002)])
def test_grad_weights_sizes(B, Nin, N, T, p):
    from paper_2311_11390_gb300 import alif
    _check(alif, *_make(T, B, Nin, N, T, p))


@cuda
@pytest.mark.parametrize("what", ["empty", "always", "full list", "over", "dense"])
def test_grad_weights_densities(what):
    from paper_2311_11390_gb300 import alif
    S, gI = _make(7, 44, 1000, 256, 2048, 0.05 if what == "dense" else -1.0 if what == "empty" else 0.001)
    if what == "always":
        S[1, 17], S[:, 999], S[2, 0] = 1.0, 1.0, 1.0
    if what in ("full list", "over"):  # rows that fit a unit's record at 1000 inputs
        rows = ((227 * 1024 - 64 - 67712 - 1001 * 128) // 2 - 512) // 16
        S[1, :, 512:1024] = 0.0
        S[1, 100:116, 512:1024] = 1.0  # 16 inputs in every step: 4 groups of 257 rows
        S[1, 500, 512:512 + 2 * (rows - 4 * 257 - 1) + (what == "over")] = 1.0
    _check(alif, S, gI)
