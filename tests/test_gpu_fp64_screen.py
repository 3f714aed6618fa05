"""The FP64 loop with stored Gram matrices screens its scores in FP32.  Here
the scores' factors lie far apart: a small frequency weight's denominator D
makes q / D large where |R|^2 underflows a float, q / D itself leaves the
floats' range, or nothing is measured at all.  The selections must be those of
the factored loop (params.c_supply = 2), which scores every candidate in FP64.
(On these inputs the oracle's direct and recurrent forms, whose rounding
differs throughout, select alike in every block, so no near-tie decides.)"""
import numpy as np
import pytest

import oracle
from paper_2205_02646_gb300 import synth
from test_gpu_parity import rl  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def holes(lr, keep, seed):
    """An aperture mask that measures only where keep(p, q) holds in a 16x16 tile."""
    rng = np.random.default_rng(seed)
    tile = np.zeros((16, 16), np.uint8)
    m = keep(*np.meshgrid(np.arange(16), np.arange(16), indexing="ij"))
    tile[m] = rng.choice(np.array([1, 3, 7, 8], np.uint8), int(m.sum()))
    return np.ascontiguousarray(np.tile(tile, (-(-lr // 16),) * 2)[:lr, :lr])


def both(rl, mask, layout, ys, nu, **kw):  # noqa: F811
    import torch
    lr_n = mask.shape[0]
    y = (synth.measure(synth.image(2 * lr_n, 2 * lr_n, 32, 4, 8700), mask, layout) * ys).astype(np.float32)
    lr = torch.from_numpy(y).cuda()
    nb = (lr_n // 2) ** 2
    out = []
    for supply in (0, 2):
        plan = rl.Plan(mask, rl.default_params(nu_max=nu, precision=1, c_supply=supply, layout=layout, **kw))
        assert (plan.info()["n_stored_c_tables"] == plan.info()["n_tables"]) == (supply == 0)
        hr = torch.full((2 * lr_n, 2 * lr_n), float("nan"), device="cuda")
        sel = torch.zeros(nb * nu, dtype=torch.int16, device="cuda")
        dc = torch.zeros(nb * nu * 2, device="cuda")
        plan.reconstruct_trace(lr, hr, sel, dc)
        plan.check()
        out.append((hr.cpu().numpy(), sel.cpu().numpy().reshape(nb, nu)))
    (h0, s0), (h1, s1) = out
    differ = (s0 != s1).any(axis=1)
    assert not differ.any(), "%d of %d blocks differ" % (differ.sum(), nb)
    # FP64 sums of 256 values before the float output: only its own rounding is left
    assert np.allclose(h0, h1, rtol=0, atol=2.0 ** -22 * np.abs(h1).max())


@pytest.mark.parametrize("ys", [1.0, 1e-2, 1e-4])
@pytest.mark.parametrize("name,rho", [("clusters", 0.1), ("lines", 0.05)])
def test_few_measurements_at_the_windows_edge(rl, name, rho, ys):  # noqa: F811
    keep = {"clusters": lambda p, q: (p < 2) & (q < 2), "lines": lambda p, q: (p == 0) | (q == 0)}[name]
    both(rl, holes(128, keep, 1 + len(name)), 1, ys, 24, rho_decay=rho)


@pytest.mark.parametrize("rho,ys,qs,nu", [(0.1, 1e-2, 1.0, 40), (1e-12, 1.0, 1.0, 30), (0.7, 1e-23, 1e30, 40),
                                          (0.7, 1e20, 1e-30, 40), (0.7, 1.0, 1e200, 30), (0.7, 0.0, 1e30, 30)])
def test_weights_and_measurements_of_opposite_scale(rl, rho, ys, qs, nu):  # noqa: F811
    mask = synth.recurrent_mask(64, 64, 4, 8301)
    both(rl, mask, 0, ys, nu, rho_decay=rho, q_table=oracle.frequency_weight(oracle.Params()).ravel() * qs)


def test_weights_that_no_float_holds(rl):  # noqa: F811
    """q / D beyond 2^600, infinite for some candidates, and zero for others."""
    mask = synth.recurrent_mask(64, 64, 4, 8302)
    q = oracle.frequency_weight(oracle.Params()).ravel()
    q[3::11] *= 1e-290
    q[5::7] = 0.0
    both(rl, mask, 0, 1.0, 30, rho_decay=0.7, q_table=q)
    q[100::37] = 1e308
    both(rl, mask, 0, 1.0, 30, rho_decay=1e-12, q_table=q)
