"""Both sides of the lines at which the stored-C kernels change their launch."""
import pytest

import test_gpu_shortlist_stored as shortlists
import test_gpu_stored_routes as routes
from paper_2205_02646_gb300 import synth
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


@pytest.mark.parametrize("beyond", [0, 1])
@pytest.mark.parametrize("per_sm", [8, 12, 16, 24])
def test_no_more_rounds_than_twelve_warps_need(rl, per_sm, beyond):  # noqa: F811
    """The mirrored loop's eight warps an SM may not cost an image another
    round, and where it does run its columns are exact."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    h, w = 4 * 38, 4 * (per_sm * sms // 38 + beyond)
    blocks = h * w // 16
    info = rl.Plan(synth.recurrent_mask(h // 2, w // 2, 4, 8200), rl.default_params(c_supply=1)).info()
    rounds = -(-(-(-blocks // sms)) // 12)
    assert rounds * info["grid"] * info["warps_per_cta"] >= blocks
    routes.test_mirrored_columns_are_exact(rl, h, w, 12)
