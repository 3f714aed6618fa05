"""Loss, gradient and logits of the proposal network against a 64-bit
reference at ragged batch sizes on both sides of every launch rule: one
sample, head tiles of 64 and 128 rows (128 from 2049 samples on 152 SMs), one
to twelve parts of the head's weight gradient with a ragged last one, more
than one sample per warp (from 6, 8 and 12 times the SMs) or per CTA (from
twice the SMs), many partial sums to add, and a small batch in buffers that a
larger one left behind."""
import numpy as np
import pytest

from oracle import cnn_ref
from paper_2205_02646_gb300 import synth
from test_gpu_proposal import rl  # noqa: F401  (fixture)

SHAPE = (40, 56)                                            # 20 x 28 blocks, a third of them near a border


def batch(n, seed):
    rng = np.random.default_rng(seed)
    y = synth.measure(synth.image(2 * SHAPE[0], 2 * SHAPE[1], 24, 3, 9300), synth.recurrent_mask(*SHAPE, 4, 31))
    blocks = np.stack([rng.integers(0, SHAPE[0] // 2, n), rng.integers(0, SHAPE[1] // 2, n)], 1).astype(np.int32)
    targets = (rng.random((n, 1024)) < 0.06).astype(np.uint8)
    mass = (rng.random((n, 1024)) * (rng.random((n, 1024)) < 0.1)).astype(np.float32)
    return y.astype(np.float32), blocks, targets, rng.random(n).astype(np.float32), mass


def params_of(seed):
    rng = np.random.default_rng(seed)
    p = {name: rng.normal(0, 0.3 if name.startswith("conv1") else 0.08, shape) for name, shape in cnn_ref.SHAPES}
    return cnn_ref.flatten(p).astype(np.float32)


def reference(params, x, blocks, targets, nu_t, mass):
    """cnn_ref.loss_and_grads on a whole batch, in 64-bit torch on x's device."""
    import torch
    dev = x.device
    flat = [torch.from_numpy(cnn_ref.bf16_round(v) if name.endswith(".w") else np.asarray(v, np.float64)).to(dev)
            for name, v in cnn_ref.unflatten(params).items()]
    flat = [t.requires_grad_() for t in flat]
    w1, b1, w2, b2, w3, b3, wh, bh = flat
    n, loss_sum, z_all, grads = x.shape[0], 0.0, [], [torch.zeros_like(t) for t in flat]

    def conv(a, w, b, stride, inside):
        cols = torch.nn.functional.unfold(a, 3, padding=1, stride=stride)
        side = a.shape[2] // stride
        return torch.relu((w.reshape(32, -1) @ cols + b[None, :, None]).view(a.shape[0], 32, side, side)) * inside

    for i in range(0, n, 512):
        at = slice(i, min(n, i + 512))
        blk = torch.from_numpy(blocks[at]).to(dev).long()

        def inside(scale):
            size = 16 // scale
            r = [((2 * blk[:, j:j + 1] - 8) // scale + torch.arange(size, device=dev)) for j in (0, 1)]
            ok = [(c >= 0) & (c < SHAPE[j] // scale) for j, c in enumerate(r)]
            return (ok[0][:, None, :, None] & ok[1][:, None, None, :]).double()
        a = conv(x[at].double(), w1, b1, 1, inside(1))
        a = conv(conv(a, w2, b2, 2, inside(2)), w3, b3, 1, inside(2))
        z = a[:, :, 3:6, 3:6].flatten(1) @ wh.T + bh
        c, t = z[:, :1024], torch.from_numpy(targets[at]).to(dev).double()
        m = torch.from_numpy(mass[at]).to(dev).double()
        with torch.no_grad():
            out = (c < c.topk(64).values[:, -1:]).double()
            share = (m * out).sum(1) / m.sum(1)
        loss = (((1 + 7 * t) * (torch.nn.functional.softplus(c) - t * c)).mean(1)
                + 0.1 * (z[:, 1024] - torch.from_numpy(nu_t[at]).to(dev).double()) ** 2
                + (torch.sigmoid(z[:, 1025]) - share) ** 2).sum() / n
        for g, d in zip(grads, torch.autograd.grad(loss, flat)):
            g += d
        loss_sum += loss.item()
        z_all.append(z.detach())
    return loss_sum, [g.cpu().numpy() for g in grads], torch.cat(z_all).cpu().numpy()


def test_reference_is_the_one_of_the_other_tests():
    import torch
    y, blocks, targets, nu_t, mass = batch(5, 0)
    params = params_of(1)
    mask = synth.recurrent_mask(*SHAPE, 4, 31)
    xs, origins = zip(*[cnn_ref.patch(y, mask, int(a), int(b)) for a, b in blocks])
    want = cnn_ref.loss_and_grads(cnn_ref.unflatten(params), list(xs), list(origins), SHAPE, list(targets), list(nu_t),
                                  list(mass))
    loss, grads, z = reference(params, torch.from_numpy(np.array(xs)), blocks, targets, nu_t, mass)
    assert abs(loss - want[0]) < 1e-12 * abs(loss)
    for (name, _), g in zip(cnn_ref.SHAPES, grads):
        assert np.abs(g - want[1][name]).max() < 1e-12 * np.abs(g).max(), name


@pytest.mark.gpu
@pytest.mark.parametrize("sizes", [(1,), (129,), (305, 7), (1000,), (2047,), (2049, 2), (4097, 130)])
def test_gradient_loss_and_logits(rl, sizes):  # noqa: F811
    import torch
    net, params = rl.Net(seed=2), params_of(3)
    net.set_params(params)
    mask = torch.from_numpy(synth.recurrent_mask(*SHAPE, 4, 31)).cuda()
    for n in sizes:
        y, blocks, targets, nu_t, mass = batch(n, n)
        bd = torch.from_numpy(blocks).cuda()
        x = rl.Net.patches(torch.from_numpy(y).cuda(), mask, bd)
        args = [torch.from_numpy(v).cuda() for v in (targets, nu_t, mass)]
        loss, grads, z = reference(params, x, blocks, targets, nu_t, mass)
        got, got_loss = net.gradient(x, bd, SHAPE, *args)
        got_z = net.logits(x, bd, SHAPE).cpu().numpy()
        # binary32 sums: 288 products behind a logit; at most about 700 terms in a row behind a gradient
        # (one part of the head's sum over samples), each rounding 2^-24 of the running sum
        assert np.abs(got_z - z).max() <= 288 * 2.0 ** -24 * np.abs(z).max(), n
        assert abs(got_loss - loss) <= 1e-5 * abs(loss), n
        for (name, _), g in zip(cnn_ref.SHAPES, grads):
            a = cnn_ref.unflatten(got.cpu().numpy())[name]
            assert np.abs(a - g).max() <= 700 * 2.0 ** -24 * np.abs(g).max(), (n, name, np.abs(a - g).max() / np.abs(g).max())
