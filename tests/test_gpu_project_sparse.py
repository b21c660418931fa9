"""The projections over event lists (products large enough to take that path): output rows that
keep 32, 16 and 4 bytes, partial weight tiles and chunks, the most inputs a weight tile holds,
steps around the lists' capacity, tiles that fall back to the dense kernels, empty rasters,
weights that are not finite -- against the float64 product."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
EPS = 2.0 ** -24


def _raster(g, B, Nin, T, p, full):
    S = (torch.rand((B, Nin, T), generator=g, device="cuda") < p).float()
    for b, t, n in full:  # exactly n active inputs at 32 steps from t
        S[b, :, t:t + 32] = 0.0
        S[b, Nin - n:, t:t + 32] = 1.0
    return S


def _check(alif, g, B, Nin, N, T, p=0.003, full=(), W=None):
    S = _raster(g, B, Nin, T, p, full)
    W = torch.randn((N, Nin), generator=g, device="cuda") * (2.0 / Nin) ** 0.5 if W is None else W
    bias = 0.8 + 0.8 * torch.rand(N, generator=g, device="cuda")
    words = alif.pack_spikes(S)
    assert alif.lib().syn_project_workspace_size(B, Nin, N, T) > 0
    hi, lo = alif.split_bf16(W)
    got = alif.syn_project(words, hi, lo, bias, Nin=Nin, T=T)
    ev = alif.syn_project_events(words, alif.transpose_weights(W), bias, Nin=Nin, T=T)
    assert alif.device_status() == 0
    for b in range(B):
        Sb, Wd, bd = S[b].double(), W.double(), bias.double()[:, None]
        ref, mag, k = Wd @ Sb + bd, Wd.abs() @ Sb, Sb.sum(0)
        run = (k + 1) * EPS * (mag + bd)  # the running sum and the bias, each rounded once per step
        assert ((ev[b].double() - ref).abs() <= run + 1e-30).all()
        # split weights: 2^-16 of each; the tensor cores' accumulation of dense tiles over all inputs
        lim = run + 2.0 ** -16 * mag + (Nin + 2) * EPS * mag + 2.0 ** -23 * ref.abs()
        assert ((got[b].double() - ref).abs() <= lim + 1e-30).all()
        if p > 0.005 and Nin > 64:
            continue  # which tiles are sparse is the kernel's choice
        sparse = torch.ones(T, dtype=torch.bool, device="cuda")
        for fb, t, n in full:
            if fb == b and n > 12:
                sparse[t // 256 * 256:t // 256 * 256 + 256] = False
        lim = run + 2.0 ** -16 * mag  # no accumulation over the inputs that are silent
        assert ((got[b].double() - ref).abs() <= lim + 1e-30)[:, sparse].all()


@cuda
@pytest.mark.parametrize("B, Nin, N, T", [(30, 1000, 1024, 2048), (45, 1000, 1030, 1308), (30, 1024, 1024, 2053),
                                          (15, 33, 8200, 16000), (460, 512, 257, 1001)])
def test_sparse_projection_sizes(B, Nin, N, T):
    from paper_2311_11390_gb300 import alif
    g = torch.Generator(device="cuda").manual_seed(T)
    _check(alif, g, B, Nin, N, T, p=0.1 if Nin < 64 else 0.003)


@cuda
@pytest.mark.parametrize("n", [11, 12, 13, 14, 31, 1000])
def test_lists_at_capacity_and_dense_tiles(n):
    """32 steps of n inputs: 384 to 448 events with the padding, of which a record of 1000 inputs holds
    432 (448 less a pair of zero rows per group), and more; the first and the last, partial, tile."""
    from paper_2311_11390_gb300 import alif
    g = torch.Generator(device="cuda").manual_seed(n)
    _check(alif, g, 30, 1000, 1024, 2053, full=[(0, 256 + 32, n), (1, 2016, n)])


@cuda
def test_empty_and_full_rasters_and_weights_not_finite():
    from paper_2311_11390_gb300 import alif
    g = torch.Generator(device="cuda").manual_seed(5)
    _check(alif, g, 30, 1000, 1024, 2048, p=-1.0)
    _check(alif, g, 30, 1000, 1024, 2048, p=0.011)  # tiles around the records' capacity
    _check(alif, g, 30, 1000, 1024, 2048, p=0.02)   # dense as a whole
    W = torch.randn((1024, 1000), generator=g, device="cuda")
    W[5, 17], W[6, 18] = float("inf"), float("nan")
    S = _raster(g, 30, 1000, 2048, 0.003, ())
    words, (hi, lo) = alif.pack_spikes(S), alif.split_bf16(W)
    got = alif.syn_project(words, hi, lo, None, Nin=1000, T=2048)
    dense = torch.empty_like(got)
    L = alif.lib()
    assert L.syn_project(30, 1000, 1024, 2048, alif._ptr(hi), alif._ptr(lo), hi.shape[1], alif._ptr(words), None,
                         alif._ptr(dense), alif._stream()) == 0
    assert torch.equal(torch.isnan(got), torch.isnan(dense)) and torch.isnan(got[:, 5:7]).all()
    assert int(torch.isnan(got).any(0).any(1).sum()) == 2
