"""The FP64 loop with stored FP64 Gram matrices against the factored FP64 loop
(params.c_supply = 2): the same selections and, to FP64 rounding before the
float output, the same image.  The stored loop screens its scores in FP32 and
gives only the leading candidates their FP64 score, so the inputs include
scales at which the screen's floats under- or overflow and an image of zeros
(every candidate ties), other layouts, whose unobservable candidates score 0,
and a frequency weight with zeros."""
import numpy as np
import pytest

from paper_2205_02646_gb300 import synth
from test_gpu_parity import rl  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def both(rl, mask, y, nu, **kw):  # noqa: F811
    import torch
    lr = torch.from_numpy(y).cuda()
    nb = (mask.shape[0] // 2) * (mask.shape[1] // 2)
    out = []
    for supply in (0, 2):
        plan = rl.Plan(mask, rl.default_params(nu_max=nu, precision=1, c_supply=supply, **kw))
        assert (plan.info()["n_stored_c_tables"] > 0) == (supply == 0)
        hr = torch.full((2 * mask.shape[0], 2 * mask.shape[1]), float("nan"), device="cuda")
        sel = torch.zeros(nb * nu, dtype=torch.int16, device="cuda")
        dc = torch.zeros(nb * nu * 2, device="cuda")
        plan.reconstruct_trace(lr, hr, sel, dc)
        plan.check()
        out.append((hr.cpu().numpy(), sel.cpu().numpy(), dc.cpu().numpy()))
    return out


@pytest.mark.parametrize("scale", [1.0, 0.0, 1e-15, 1e-22, 1e-32, 1e15, 1e22])
def test_screen_at_every_scale(rl, scale):  # noqa: F811
    f = synth.image(60, 68, 32, 4, 8300)
    mask = synth.recurrent_mask(30, 34, 4, 8301)
    y = (synth.measure(f, mask) * scale).astype(np.float32)
    (h0, s0, d0), (h1, s1, d1) = both(rl, mask, y, 100)
    assert np.isfinite(h0).all()
    # scores that round to the same binary32 value tie; a sum in another order may fall on either side of
    # that rounding (about 1e-8 of the comparisons): no block of this image does
    assert np.array_equal(s0, s1)
    assert np.allclose(h0, h1, rtol=0, atol=2e-7 * 3 * scale)
    assert np.allclose(d0, d1, rtol=0, atol=2e-7 * 3 * scale)


@pytest.mark.parametrize("layout,size,nu", [("quarter", (64, 64), 100), ("mixed", (68, 72), 100),
                                            ("three_quarter", (16, 240), 60)])
def test_other_layouts_and_zero_weights(rl, layout, size, nu):  # noqa: F811
    h, w = size
    f = synth.image(h, w, 32, 4, 8400)
    mask = synth.aperture_mask(h // 2, w // 2, 4, 8401, synth.APERTURE_SETS[layout])
    y = synth.measure(f, mask, 1).astype(np.float32)
    q = np.linspace(1.0, 2.0, 1024)
    q[5::7] = 0.0
    (h0, s0, _), (h1, s1, _) = both(rl, mask, y, nu, layout=1, q_table=q)
    assert np.array_equal(s0, s1) and np.allclose(h0, h1, rtol=0, atol=1e-6)


def test_small_runs_keep_the_factored_loop(rl):  # noqa: F811
    """A plan whose single pass would not earn back the matrices' build stores none."""
    f, mask, y = synth.workload("rljsde_64x64")
    assert rl.Plan(mask, rl.default_params(nu_max=10, precision=1)).info()["n_stored_c_tables"] == 0
    assert rl.Plan(mask, rl.default_params(nu_max=100, precision=1)).info()["n_stored_c_tables"] > 0
