"""Which event projections take the lists, at sizes timed both ways: short rows with one 32-step chunk are left to the
kernel without lists, two chunks and more are not."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")


@cuda
@pytest.mark.parametrize("size, lists", [((2048, 64, 64, 32), False), ((5000, 100, 64, 32), False), ((512, 700, 256, 32), False),
                                         ((2048, 64, 64, 33), True), ((512, 700, 256, 40), True),
                                         ((5000, 100, 64, 64), True), ((1000, 100, 500, 100), True)])
def test_choice(size, lists):
    from paper_2311_11390_gb300 import alif
    assert (alif.lib().syn_project_events_workspace_size(*size) > 0) == lists
