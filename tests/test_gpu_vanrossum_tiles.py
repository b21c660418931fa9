"""van Rossum kernels at the edges of their tiles: a word of 32 steps per thread, 512 words per
tile, rows of several tiles, gradient rows that do and do not keep 16 or 32 bytes, a carry from
the steps after the call."""
import numpy as np
import pytest
import torch

from paper_2311_11390_gb300 import synth

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
EPS = 2.0 ** -24


def _filter(d, dec, start):
    """y[t] = dec y[t-1] + d[t] in float64, y[-1] = start [rows]."""
    y, acc = np.empty(d.shape), np.asarray(start, np.float64).copy()
    for t in range(d.shape[1]):
        acc = dec * acc + d[:, t]
        y[:, t] = acc
    return y


@cuda
@pytest.mark.parametrize("T", [1, 31, 32, 33, 1023, 1024, 1056, 16383, 16384, 16385, 16416, 40003])
@pytest.mark.parametrize("dt", [0.05, 1.0])
def test_vanrossum_tiles(T, dt):
    """Bounds: a filtered value passes at most 8 + 3 steps' and chains' roundings in its word, 5 + 4
    scan levels of two roundings, the tile's carry (3) and a rounded decay (8 factors): under 48 u
    of the filter of |d|; the reverse filter meets as many again on top."""
    from paper_2311_11390_gb300 import alif
    rng = np.random.default_rng(T)
    rows, tau = 3, 5.0
    x, y = rng.random((rows, T)) < 0.03, rng.random((rows, T)) < 0.03
    x[1] = y[1]  # a row without any difference
    dev = lambda a: torch.from_numpy(synth.pack_bits(a).view(np.int32)).cuda()  # noqa: E731
    xw, yw = dev(x), dev(y)
    dec, d = np.exp(-dt / tau), x.astype(float) - y.astype(float)
    f, F = _filter(d, dec, np.zeros(rows)), _filter(np.abs(d), dec, np.zeros(rows))
    nck = -(-T // 256)
    fck, loss = torch.full((rows, nck), 9.0, device="cuda"), torch.empty(rows, device="cuda")
    alif.vanrossum_forward(xw, yw, T, dt, tau, 256, fck, loss)
    entering = np.concatenate([np.zeros((rows, 1)), f], 1)[:, :-1][:, ::256]
    bound = np.concatenate([np.zeros((rows, 1)), F], 1)[:, :-1][:, ::256]
    assert (np.abs(fck.cpu().numpy() - entering) <= 48 * EPS * bound + 1e-30).all()
    ref = dt / tau * (f ** 2).sum(1)
    assert (np.abs(loss.cpu().numpy() - ref) <= (2 * 48 + 40) * EPS * dt / tau * (F ** 2).sum(1)).all()
    gc0 = rng.standard_normal(rows).astype(np.float32)
    rev = lambda v, s: _filter(v[:, ::-1], dec, s)[:, ::-1]  # noqa: E731
    g, G = rev(f, gc0), rev(F, np.abs(gc0))
    for t0 in {0, (T - 1) // 256 // 2 * 256, (T - 1) // 256 * 256}:
        gc, out = torch.from_numpy(gc0).cuda(), torch.full((rows, T - t0), 9.0, device="cuda")
        alif.vanrossum_backward(xw, yw, T, dt, tau, t0, T, fck[:, t0 // 256].contiguous(), gc, out)
        scale = 2.0 * dt / tau
        assert (np.abs(out.cpu().numpy() / scale - g[:, t0:]) <= (2 * 48 + 2) * EPS * G[:, t0:] + 1e-30).all()
        assert (np.abs(gc.cpu().numpy() - g[:, t0]) <= 2 * 48 * EPS * G[:, t0] + 1e-30).all()
