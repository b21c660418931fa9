"""Rows whose length is not a multiple of 4 under the lane-per-row layout: T_eff = 2 (step by step), 4, 8
and 20 (Blocks of 4, 8 and 16), row counts that are not a multiple of 4 or of 32, a refractory initial
state; against the warp-per-row kernel (spikes and refractory counts equal, v and a within FP32 rounding,
the tolerance the layouts are compared with elsewhere)."""
import numpy as np
import pytest
import torch

from paper_2311_11390_gb300 import synth

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("T", [65, 66, 67, 95, 97, 127, 129, 255, 257, 514, 1001])
@pytest.mark.parametrize("arp, B, N", [(2.0, 3, 45), (4.0, 2, 17), (8.0, 1, 7), (20.0, 5, 33), (20.0, 4, 24)])
def test_ragged_rows_against_the_warp_layout(T, arp, B, N):
    from paper_2311_11390_gb300 import alif
    w = synth.population(seed=T, B=B, N=N, T=T, dt=1.0, arp=arp, bias=(1.0, 4.0), tau_mem=(2.0, 40.0),
                         tau_adapt=(20.0, 400.0), d=(0.0, 0.8))
    p = w.params
    table = alif.neuron_table(p.tau_mem, p.tau_adapt, p.theta0, p.d, p.R, w.dt, w.arp)
    I = torch.from_numpy(np.ascontiguousarray(w.I)).cuda()
    g = torch.Generator().manual_seed(T)
    rem = torch.randint(0, 4, (B, N), generator=g, dtype=torch.int32)
    v = torch.where(rem > 0, 0.0, torch.rand(B, N, generator=g))
    init = alif.state_tensor(B, N, v=v, a=torch.rand(B, N, generator=g) * 3, rem=rem)
    out = []
    for layout in (2, 1):
        before = alif.forward_layout(layout)
        alif.forward_stats()
        out.append(alif.forward(I, table, init=init))
        alif.forward_layout(before)
        assert alif.device_status() == 0 and alif.forward_stats()["rows"] == B * N
    one, ref = out
    assert torch.equal(one["spikes"], ref["spikes"])
    for k in ("ckpt", "final"):
        a, b = one[k].cpu().numpy(), ref[k].cpu().numpy()
        assert np.array_equal(a[..., 2], b[..., 2])
        x, y = np.ascontiguousarray(a).view(np.float32)[..., :2], np.ascontiguousarray(b).view(np.float32)[..., :2]
        assert np.allclose(x, y, rtol=1e-5, atol=1e-6)
