"""Rows with T_eff = 2 and 3 under the lane-per-row layout, which walks them step by step: against the
warp-per-row kernel (spikes equal; v and a within FP32 rounding, 2^-22 of the states' magnitude) and
against FP64 where every margin is too close for FP32."""
import numpy as np
import pytest
import torch

from paper_2311_11390_gb300 import synth

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


def _forward(alif, layout, I, table, init=None):
    before = alif.forward_layout(layout)
    out = alif.forward(I, table, init=init)
    alif.forward_layout(before)
    assert alif.device_status() == 0
    return out


def _close(a, b):
    a, b = a.cpu().numpy(), b.cpu().numpy()
    assert np.array_equal(a[..., 2], b[..., 2])
    x, y = np.ascontiguousarray(a).view(np.float32)[..., :2], np.ascontiguousarray(b).view(np.float32)[..., :2]
    assert (np.abs(x - y) <= 2.0 ** -22 * np.maximum(np.abs(y), 4.0)).all()


@cuda
@pytest.mark.parametrize("T", [4, 28, 32, 36, 60, 64, 68, 256, 260, 1000])
@pytest.mark.parametrize("arp", [2.0, 3.0])
def test_steps_against_the_warp_layout(T, arp):
    from paper_2311_11390_gb300 import alif
    B, N = 3, 45  # 135 rows: the last warp's lanes are partly idle
    w = synth.population(seed=T, B=B, N=N, T=T, dt=1.0, arp=arp, bias=(1.0, 4.0), tau_mem=(2.0, 40.0),
                         tau_adapt=(20.0, 400.0), d=(0.0, 0.8))
    p = w.params
    table = alif.neuron_table(p.tau_mem, p.tau_adapt, p.theta0, p.d, p.R, w.dt, w.arp)
    I = torch.from_numpy(np.ascontiguousarray(w.I)).cuda()
    g = torch.Generator().manual_seed(T)
    rem = torch.randint(0, 4, (B, N), generator=g, dtype=torch.int32)
    v = torch.where(rem > 0, 0.0, torch.rand(B, N, generator=g))
    init = alif.state_tensor(B, N, v=v, a=torch.rand(B, N, generator=g) * 3, rem=rem)
    one, ref = _forward(alif, 2, I, table, init), _forward(alif, 1, I, table, init)
    assert torch.equal(one["spikes"], ref["spikes"])
    _close(one["ckpt"], ref["ckpt"])
    _close(one["final"], ref["final"])


@cuda
def test_steps_where_every_margin_is_close():
    """A constant current that drives V to theta from below (theta - V = theta beta^(t+1), 2e-9 theta at
    the last step) and, scaled by 1 + 1e-8, across it: the spikes of FP64."""
    from paper_2311_11390_gb300 import alif
    N, T = 64, 40
    tau = np.full(N, 2.0, np.float32)
    one = np.ones(N, np.float32)
    table = alif.neuron_table(tau, 50 * tau, one, 0 * one, one, 1.0, 2.0)
    scale = np.where(np.arange(N) % 2 == 0, np.float32(1.0), np.float32(1.0 + 2.0 ** -23))
    I = np.broadcast_to(scale[None, :, None], (1, N, T)).astype(np.float32).copy()
    out = _forward(alif, 2, torch.from_numpy(I).cuda(), table)
    beta, V, S = np.exp(-0.5), np.zeros(N), np.zeros((N, T), bool)
    mask = np.zeros(N, int)
    for t in range(T):
        V = beta * V + (mask <= 0) * (1 - beta) * I[0, :, t].astype(np.float64)
        S[:, t] = (mask <= 0) & (V > 1.0)
        V[S[:, t]] = 0.0
        mask = np.where(S[:, t], 2, mask) - 1
    got = alif.unpack_spikes(out["spikes"], T)[0].cpu().numpy() != 0
    assert S.any() and not S[::2].any()
    assert np.array_equal(got, S)
