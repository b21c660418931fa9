"""The squared distance sums at most 8 squares in FP32 before the double-single sum.  With a decay of 1/2 the
filter is (nearly) exact in FP32, and for these pairs of 32-step trains the exact distance is further from a
rounding boundary than the sum's error, while FP32 additions of the four partial sums of a word round to the
neighbouring number: the loss has to be the exact distance, rounded once."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
PAIRS = [(0x09000003, 0x10124040), (0x00200000, 0x880c1000), (0x42080406, 0x00004000), (0x00005022, 0x10010036),
         (0x00012040, 0x08004004), (0x81408050, 0x00000924), (0x40412800, 0x00009000), (0x00020040, 0x11284020),
         (0x00288060, 0x00004000), (0x0440020a, 0x00010000)]


def _exact(x, y):
    f = total = Fraction(0)
    for t in range(32):
        f = f / 2 + ((x >> t) & 1) - ((y >> t) & 1)
        total += f * f
    return np.float32(float(Fraction(math.log(2.0)) * total))


@cuda
def test_partial_sums_join_without_rounding():
    from paper_2311_11390_gb300 import alif
    assert math.exp(-math.log(2.0)) == 0.5
    x, y = (torch.from_numpy(np.array([p[k] for p in PAIRS], dtype=np.uint32).view(np.int32)[:, None]).cuda() for k in (0, 1))
    loss = torch.empty(len(PAIRS), device="cuda")
    alif.vanrossum_forward(x, y, 32, math.log(2.0), 1.0, 256, loss=loss)
    want = np.array([_exact(*p) for p in PAIRS], dtype=np.float32)
    assert (loss.cpu().numpy() == want).all()
