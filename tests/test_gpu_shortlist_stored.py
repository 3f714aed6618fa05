"""The shortlist kernel on stored Gram matrices at the edges of its work list:
an odd number of blocks (a warp takes two), both blocks of a warp gated
differently, table sets that change inside a pair, and the gate sending none
or all of the blocks to the full loop.  With a shortlist that holds every
candidate a block's plain loop selects, the restricted loop makes the same
choices with the same stored columns, so its trace equals the plain one's; a
gated block's output equals the plain loop's bit for bit."""
import numpy as np
import pytest

from paper_2205_02646_gb300 import synth
from test_gpu_parity import rl  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w", [(8, 8), (12, 20), (36, 100), (100, 260)])
@pytest.mark.parametrize("gate", ["none", "all", "every third"])
def test_edges_of_the_work_list(rl, h, w, gate):  # noqa: F811
    import torch
    nu = 30                                     # at most 30 distinct candidates: they fit a shortlist of 64
    f = synth.image(h, w, 32, 4, 8500 + w)
    mask = synth.recurrent_mask(h // 2, w // 2, 4, 8501)
    lr = torch.from_numpy(synth.measure(f, mask).astype(np.float32)).cuda()
    nb = (h // 4) * (w // 4)
    plan = rl.Plan(mask, rl.default_params(nu_max=nu, c_supply=1))
    hr0, hr1 = (torch.full((h, w), float("nan"), device="cuda") for _ in range(2))
    sel0, sel1 = (torch.zeros(nb * nu, dtype=torch.int16, device="cuda") for _ in range(2))
    dc0, dc1 = (torch.zeros(nb * nu * 2, device="cuda") for _ in range(2))
    plan.reconstruct_trace(lr, hr0, sel0, dc0)
    s0 = sel0.cpu().numpy().reshape(nb, nu).astype(np.int64)
    idx = np.empty((nb, 64), np.int64)
    for b in range(nb):
        have = np.unique(s0[b])
        rest = np.setdiff1d(np.arange(1024), have)
        idx[b] = np.sort(np.concatenate([have, rest[:: max(1, len(rest) // 64)][:64 - len(have)]]))
    back = {"none": np.zeros(nb, bool), "all": np.ones(nb, bool), "every third": np.arange(nb) % 3 == 1}[gate]
    sl = torch.from_numpy(rl.shortlist_from_indices(idx, missing=back.astype(np.float32))).cuda()
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    plan.reconstruct_learned(lr, hr1, sl, max_missing=0.5, sel=sel1, dc=dc1, counter=count)
    plan.check()
    assert int(count) == int((~back).sum())
    s1 = sel1.cpu().numpy().reshape(nb, nu)
    # the restricted loop's initial projection sums in another order: a block may part at a near-tie
    same = np.all(s0 == s1, axis=1)
    assert same[back].all() and same.mean() > 0.98
    d0, d1 = (d.cpu().numpy().reshape(nb, nu, 2) for d in (dc0, dc1))
    blocks = lambda t: t.cpu().numpy().reshape(h // 4, 4, w // 4, 4).transpose(0, 2, 1, 3).reshape(nb, 16)  # noqa: E731
    p0, p1 = blocks(hr0), blocks(hr1)
    assert np.isfinite(p1).all()
    assert np.array_equal(p0[back], p1[back]) and np.array_equal(d0[back], d1[back])
    # binary32 sums over 256 window values: 2^-24 x 256 of values up to about 3
    assert np.abs(p0 - p1)[same].max(initial=0) < 5e-5


def test_gated_blocks_with_an_asymmetric_weight(rl):  # noqa: F811
    """A frequency weight that differs between k and -k: no column may be read
    as its mirror, in the gated full loop either."""
    import torch
    f = synth.image(64, 96, 32, 4, 8600)
    mask = synth.recurrent_mask(32, 48, 4, 8601)
    lr = torch.from_numpy(synth.measure(f, mask).astype(np.float32)).cuda()
    q = np.linspace(2.0, 1.0, 1024)
    nb, nu = 16 * 24, 40
    plan = rl.Plan(mask, rl.default_params(nu_max=nu, c_supply=1, q_table=q))
    hr0, hr1 = (torch.full((64, 96), float("nan"), device="cuda") for _ in range(2))
    plan.reconstruct(lr, hr0)
    idx = np.tile(np.arange(64), (nb, 1))
    sl = torch.from_numpy(rl.shortlist_from_indices(idx, missing=np.ones(nb, np.float32))).cuda()
    plan.reconstruct_learned(lr, hr1, sl, max_missing=0.5)
    plan.check()
    factored = rl.Plan(mask, rl.default_params(nu_max=nu, c_supply=2, q_table=q))
    hr2 = torch.full((64, 96), float("nan"), device="cuda")
    factored.reconstruct(lr, hr2)
    h0, h1, h2 = (h.cpu().numpy() for h in (hr0, hr1, hr2))
    assert np.array_equal(h0, h1)
    # the factored loop agrees but for rounding, except where a near-tie parts a block
    far = np.abs(h0 - h2).reshape(16, 4, 24, 4).max(axis=(1, 3)) > 1e-4
    assert far.mean() < 0.02
