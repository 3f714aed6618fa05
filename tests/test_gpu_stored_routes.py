"""The stored-C loop's kernels against each other.  The mirrored loop reads
column -uv as the conjugate of column uv, which is exact when the frequency
weight is symmetric; a weight that differs in the last bit at one candidate no
block selects takes the plain loop, and every other candidate's arithmetic is
the same, so outputs and traces agree bit for bit.  Sizes sit at the edges of
the launch rules: one block row, fewer blocks than SMs, one CTA's warps partly
filled, and both sides of the mirrored loop's limit (27 blocks per SM)."""
import numpy as np
import pytest

from paper_2205_02646_gb300 import synth
from test_gpu_parity import rl  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def default_q():
    k = np.arange(32.0)
    k = np.where(k <= 16, k, k - 32)
    return (1 - np.hypot(*np.meshgrid(k, k, indexing="ij")) / (32 / np.sqrt(2))) ** 2 + 1e-3


@pytest.mark.parametrize("h,w,nu", [(8, 8, 30), (8, 300, 2), (64, 64, 60), (124, 84, 25), (252, 256, 20), (272, 260, 20)])
def test_mirrored_columns_are_exact(rl, h, w, nu):  # noqa: F811
    import torch
    f = synth.image(h, w, 32, 4, 8100 + h)
    mask = synth.recurrent_mask(h // 2, w // 2, 4, 8200)
    lr = torch.from_numpy(synth.measure(f, mask).astype(np.float32)).cuda()
    nb, odd = (h // 4) * (w // 4), 16 * 32 + 15            # (16, 15): its mirror (16, 17) keeps its weight
    out = []
    for trace in (True, False):
        for bump in (False, True):
            q = default_q()
            if bump:
                q[16, 15] = np.nextafter(q[16, 15], 2.0)
            plan = rl.Plan(mask, rl.default_params(nu_max=nu, q_table=q, c_supply=1))
            hr = torch.full((h, w), float("nan"), device="cuda")
            if trace:
                sel = torch.zeros(nb * nu, dtype=torch.int16, device="cuda")
                dc = torch.zeros(nb * nu * 2, device="cuda")
                plan.reconstruct_trace(lr, hr, sel, dc)
                s = sel.cpu().numpy()
                out.append((hr.cpu().numpy(), s, dc.cpu().numpy()))
                assert not np.isin(s, (odd, odd + 2)).any()
            else:
                plan.reconstruct(lr, hr)
                out.append((hr.cpu().numpy(),))
            plan.check()
    (h0, s0, d0), (h1, s1, d1), (h2,), (h3,) = out
    assert np.isfinite(h0).all()
    assert np.array_equal(s0, s1) and np.array_equal(d0, d1)
    assert np.array_equal(h0, h1) and np.array_equal(h0, h2) and np.array_equal(h0, h3)
