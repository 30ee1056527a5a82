"""The fused network kernels at the edges of their shapes against the FP64 reference MLP.

Fused: widths that are multiples of 64 up to 256, n_in <= 64, n_out <= 256; a batch tile has 16 rows (32 above
2432 rows), a weight-gradient split 256.  The last two shapes run layer by layer.  The reference takes
the same bfloat16-rounded weights and inputs, so what differs is the bfloat16 rounding (relative 2^-9)
of each hidden activation and each backward signal: 1e-2 of max|y| on outputs, as derived in
tests/test_gpu_mlp.py for four hidden layers.  A gradient is a sum over the batch of products
d(b, o) h(b, i) whose factors each carry such relative errors, a few 2^-9 after several layers, so its error is
bounded by 3e-2 = 15 * 2^-9 of the sum of the products' magnitudes (the sum itself cancels: with
random labels its size falls like batch^-1/2 while the rounding of the factors is common to the rows).
"""
import numpy as np
import pytest

import paper_1705_03141_gb300 as pkg
from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu

# n_in, width, depth, n_pos, n_cls, batch
SHAPES = [(5, 256, 4, 64, 4, 1), (5, 256, 4, 64, 4, 17), (5, 256, 4, 64, 4, 64), (5, 256, 4, 64, 4, 2433),
          (1, 64, 1, 1, 0, 16), (64, 128, 2, 0, 3, 33), (7, 192, 3, 63, 2, 257), (3, 256, 1, 252, 4, 31),
          (5, 64, 8, 9, 4, 48), (5, 96, 2, 8, 4, 40), (65, 128, 2, 8, 4, 40)]


def bf16(a):
    u = np.asarray(a, dtype=np.float32).view(np.uint32).astype(np.uint64)
    return (((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32)).view(np.float32).astype(np.float64)


@pytest.mark.parametrize("n_in,width,depth,n_pos,n_cls,batch", SHAPES)
def test_forward_gradient_and_step(cuda, n_in, width, depth, n_pos, n_cls, batch):
    import torch

    sizes = [n_in] + [width] * depth + [n_pos + n_cls]
    flat = M.flatten(M.init_params(sizes, seed=3)).astype(np.float32)
    net = pkg.Mlp(n_in=n_in, width=width, depth=depth, n_pos=n_pos, n_cls=n_cls, max_batch=batch)
    net.set_params(flat)
    ref = [(bf16(W), b.astype(np.float32).astype(np.float64)) for W, b in M.unflatten(flat.astype(np.float64), sizes)]
    rng = np.random.default_rng(4)
    x = rng.uniform(-1, 1, size=(batch, n_in)).astype(np.float32)
    t = (0.3 * rng.normal(size=(batch, n_pos))).astype(np.float32)
    lab = rng.integers(0, max(n_cls, 1), size=batch).astype(np.int32)
    y = net.forward(x)
    yr, cache = M.forward(ref, bf16(x))
    assert np.max(np.abs(y - yr)) < 1e-2 * np.max(np.abs(yr))
    xd = torch.from_numpy(x).cuda()
    np.testing.assert_array_equal(net.forward(xd).cpu().numpy(), y)  # the caller's device buffers, no staging
    # loss and gradient: positions and classes may be absent
    dy = np.zeros_like(yr)
    want = 0.0
    if n_pos:
        d = yr[:, :n_pos] - t
        want += np.mean(d * d)
        dy[:, :n_pos] = 2.0 * d / d.size
    if n_cls:
        z = yr[:, n_pos:] - yr[:, n_pos:].max(axis=1, keepdims=True)
        p = np.exp(z) / np.exp(z).sum(axis=1, keepdims=True)
        want += 0.5 * -np.mean(np.log(p[np.arange(batch), lab]))
        dy[:, n_pos:] = 0.5 * (p - np.eye(n_cls)[lab]) / batch
    gr = M.flatten(M.backward(ref, cache, dy))
    mags, d = [], dy  # per layer the sums of |d| |h| behind its weight and bias gradients
    for l in range(len(ref) - 1, -1, -1):
        h, z = cache[l]
        if l < len(ref) - 1:
            d = d * M.silu_grad(z)
        mags.insert(0, (np.abs(d).T @ np.abs(h), np.abs(d).sum(0)))
        d = d @ ref[l][0]
    mag = M.flatten(mags)
    loss, g = net.loss_grad(x, t, lab, w_pos=1.0, w_cls=0.5)
    assert loss == pytest.approx(want, rel=1e-2, abs=1e-6)
    o = 0
    for a, b in zip(sizes[:-1], sizes[1:]):
        for n in (a * b, b):
            assert np.max(np.abs(g[o:o + n] - gr[o:o + n])) < 3e-2 * np.max(mag[o:o + n]) + 1e-9, (a, b, n)
            o += n
    loss2, g2 = net.loss_grad(x, t, lab, w_pos=1.0, w_cls=0.5)
    assert loss2 == loss
    np.testing.assert_array_equal(g2, g)
    # the first Adam step from this gradient moves every parameter by lr g / (|g| + 1e-8)
    assert net.train_step(x, t, lab, lr=1e-2, w_pos=1.0, w_cls=0.5) == loss
    step = net.get_params() - flat
    np.testing.assert_allclose(step, -1e-2 * g / (np.abs(g) + 1e-8), rtol=0, atol=1e-2 * 2e-4 + 2.0 ** -23)
    # the bfloat16 copies follow the parameters, the transposed one among them
    fresh = pkg.Mlp(n_in=n_in, width=width, depth=depth, n_pos=n_pos, n_cls=n_cls, max_batch=batch)
    fresh.set_params(net.get_params())
    la, ga = net.loss_grad(x, t, lab)
    lb, gb = fresh.loss_grad(x, t, lab)
    assert la == lb
    np.testing.assert_array_equal(ga, gb)
    if n_cls:  # a label out of range is reported, and the next call is clean
        with pytest.raises(pkg.LbmError):
            net.loss_grad(x, t, np.full(batch, n_cls, np.int32))
        assert net.loss_grad(x, t, lab)[0] == la
    net.close()
    fresh.close()


# n_in, n_out and batch of more than one block, y ahead of, at and behind the start of x
@pytest.mark.parametrize("offset", [-340, -5, 0, 5, 340])
@pytest.mark.parametrize("n_in,n_out,batch", [(5, 68, 4096), (40, 4, 3000), (8, 8, 333)])
def test_output_overlapping_the_input(cuda, n_in, n_out, batch, offset):
    import torch

    net = pkg.Mlp(n_in=n_in, width=128, depth=2, n_pos=n_out, n_cls=0, max_batch=batch, seed=3)
    x = torch.rand(batch, n_in, generator=torch.Generator().manual_seed(1)).cuda()
    want = net.forward(x)
    buf = torch.zeros(512 + batch * max(n_in, n_out) + 512, device="cuda")
    xv = buf[512:512 + batch * n_in].view(batch, n_in)
    xv.copy_(x)
    yv = buf[512 + offset:512 + offset + batch * n_out].view(batch, n_out)
    got = net.forward(xv, out=yv)
    assert got.data_ptr() == yv.data_ptr() and torch.equal(got, want)
    net.close()


@pytest.mark.parametrize("width", [64, 96])  # fused, layer by layer
def test_silu_over_the_whole_range(cuda, width):
    """One hidden layer with the pre-activations as biases and one output per unit: y = bf16(z sigmoid(z)), with z
    where sigmoid is normal, subnormal and zero in FP32.  bfloat16 holds 8 bits, so it rounds a value in [1, 2) to
    half of 2^-7, at most 2^-8 of it (2^-134 where it is subnormal itself); expf errs by 2 units of 2^-24, and
    a subnormal sigmoid by a unit of 2^-149."""
    z = np.concatenate([np.linspace(-103.0, -80.0, 24), np.linspace(-8.0, 8.0, 33), [-120.0, -30.0, 0.0, 40.0, 120.0]])
    z = np.resize(z, width).astype(np.float32)
    net = pkg.Mlp(n_in=1, width=width, depth=1, n_pos=width, n_cls=0, max_batch=1)
    net.set_params(np.concatenate([np.zeros(width), z, np.eye(width).ravel(), np.zeros(width)]).astype(np.float32))
    y = net.forward(np.zeros((1, 1), np.float32))[0].astype(np.float64)
    net.close()
    zd = z.astype(np.float64)
    e = np.exp(-zd)
    want = np.where(e > np.finfo(np.float32).max, 0.0, zd / (1.0 + e))
    tiny = np.abs(zd) * 2.0 ** -148
    bad = np.abs(y - want) > (2.0 ** -8 + 2.0 ** -22) * np.abs(want) + tiny + 2.0 ** -134
    assert not bad.any(), (z[bad], y[bad], want[bad])
