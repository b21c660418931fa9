"""Rows whose windows start at any 4-byte boundary (T not a multiple of 16, arrays off a 16-byte
boundary): against the same rows padded with zero currents and gradients to a multiple of 16, which
take the tiled staging.  Padding changes no step below T and the two run the same operations on the
same numbers, so everything is compared bit for bit (multi-Gaussian surrogate: the fast sigmoid's tiled kernel
sums the tau_mem gradient in another order, which the oracle's tests bound)."""
import numpy as np
import pytest
import torch

from paper_2311_11390_gb300 import synth

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


def off(x, k):
    """x as a contiguous tensor that starts k floats past a 16-byte boundary."""
    y = torch.empty(x.numel() + k, device=x.device)[k:].view(x.shape)
    assert y.data_ptr() % 16 == 4 * k
    return y.copy_(x)


@cuda
@pytest.mark.parametrize("T", [1, 2, 3, 5, 31, 250, 255, 257, 259, 508, 511, 513, 515, 1000, 1025])
@pytest.mark.parametrize("shift", [(0, 0), (1, 3), (2, 1), (3, 2)])
def test_any_start_is_the_padded_row(T, shift):
    from paper_2311_11390_gb300 import alif
    B, N, P = 2, 3, (T + 15) // 16 * 16
    w = synth.population(seed=T, B=B, N=N, T=P)
    p = w.params
    table = alif.neuron_table(p.tau_mem, p.tau_adapt, p.theta0, p.d, p.R, w.dt, w.arp)
    I = torch.from_numpy(np.ascontiguousarray(w.I)).cuda() * 1.5
    I[..., T:] = 0.0
    g = torch.Generator(device="cuda").manual_seed(T)
    gS, gV, ga = (torch.randn(I.shape, device="cuda", generator=g) for _ in range(3))
    for x in (gS, gV, ga):
        x[..., T:] = 0.0
    cut = lambda x, k: off(x[..., :T].contiguous(), k)
    before = alif.forward_window(256), alif.backward_window(256), alif.forward_layout(1)
    try:
        for traces in (False, True):
            kw = dict(want_v=traces, want_a=traces)
            full = alif.forward(I, table, **kw)
            o = alif.forward(cut(I, shift[0]), table, **kw)
            bits = alif.unpack_spikes(full["spikes"], P)[..., :T]
            assert torch.equal(alif.unpack_spikes(o["spikes"], T), bits)
            assert torch.equal(o["ckpt"], full["ckpt"])
            for k in ("v", "a"):
                if traces:
                    assert torch.equal(o[k], full[k][..., :T])
            kw = dict(surrogate="multi_gaussian")
            if traces:
                kw.update(grad_v=gV, grad_a=ga)
            ref = alif.backward(I, table, full["spikes"], gS, ckpt=full["ckpt"], **kw)
            if traces:
                kw.update(grad_v=cut(gV, shift[1]), grad_a=cut(ga, shift[0]))
            got = alif.backward(cut(I, shift[0]), table, o["spikes"], cut(gS, shift[1]), ckpt=o["ckpt"], **kw)
            assert torch.equal(got[0], ref[0][..., :T])
            assert torch.equal(got[2], ref[2])
    finally:
        alif.forward_window(before[0]), alif.backward_window(before[1]), alif.forward_layout(before[2])
