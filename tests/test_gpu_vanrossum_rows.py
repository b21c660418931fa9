"""van Rossum kernels with a warp per row: more rows than warps on the chip, rows of a few steps, of one tile of
32 words and of several, the longest taken so and one beyond it, gradient rows on and off the 16-byte grid, a
chunk's gradient.  Bounds as at the edges of the tiles: 48 roundings of a filtered value, as many for the reverse."""
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
@pytest.mark.parametrize("rows, T", [(9, 5), (20003, 40), (10001, 257), (5000, 1001), (1023, 1500), (1024, 1056), (1025, 4003),
                                     (1024, 32768), (1024, 32772)])
def test_rows_by_warps(rows, T):
    from paper_2311_11390_gb300 import alif
    rng = np.random.default_rng(T)
    dt, tau = 0.1, 5.0
    x, y = rng.random((rows, T), dtype=np.float32) < 0.03, rng.random((rows, T), dtype=np.float32) < 0.03
    x[1] = y[1]
    xw, yw = (torch.from_numpy(synth.pack_bits(a).view(np.int32)).cuda() for a in (x, y))
    dec, d = np.exp(-dt / tau), x.astype(float) - y.astype(float)
    f, F = _filter(d, dec, np.zeros(rows)), _filter(np.abs(d), dec, np.zeros(rows))
    fck, loss = torch.full((rows, -(-T // 256)), 9.0, device="cuda"), torch.empty(rows, device="cuda")
    alif.vanrossum_forward(xw, yw, T, dt, tau, 256, fck, loss)
    entering = np.concatenate([np.zeros((rows, 1)), f], 1)[:, :-1][:, ::256]
    bound = np.concatenate([np.zeros((rows, 1)), F], 1)[:, :-1][:, ::256]
    assert (np.abs(fck.cpu().numpy() - entering) <= 48 * EPS * bound + 1e-30).all()
    assert (np.abs(loss.cpu().numpy() - dt / tau * (f ** 2).sum(1)) <= (2 * 48 + 40) * EPS * dt / tau * (F ** 2).sum(1)).all()
    gc0 = rng.standard_normal(rows).astype(np.float32)
    rev = lambda v, s: _filter(v[:, ::-1], dec, s)[:, ::-1]  # noqa: E731
    g, G = rev(f, gc0), rev(F, np.abs(gc0))
    for t0 in {0, (T - 1) // 256 // 2 * 256}:
        gc, out = torch.from_numpy(gc0).cuda(), torch.full((rows, T - t0), 9.0, device="cuda")
        alif.vanrossum_backward(xw, yw, T, dt, tau, t0, T, fck[:, t0 // 256].contiguous(), gc, out)
        scale = 2.0 * dt / tau
        assert (np.abs(out.cpu().numpy() / scale - g[:, t0:]) <= (2 * 48 + 2) * EPS * G[:, t0:] + 1e-30).all()
        assert (np.abs(gc.cpu().numpy() - g[:, t0]) <= 2 * 48 * EPS * G[:, t0] + 1e-30).all()
