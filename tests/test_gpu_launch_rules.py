"""Both sides of the lines at which the stored-C kernels change their launch."""
import pytest

import test_gpu_shortlist_stored as shortlists
from test_gpu_parity import rl  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gate", ["none", "all", "every third"])
@pytest.mark.parametrize("cols", [0, 1])
def test_learned_blocks_singly_and_in_pairs(rl, cols, gate):  # noqa: F811
    """Up to twelve blocks per SM a warp takes one shortlisted block and the
    CTAs single entries; beyond, two at a time from runs of eight."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shortlists.test_edges_of_the_work_list(rl, 4 * 38, 4 * (12 * sms // 38 + cols), gate)
