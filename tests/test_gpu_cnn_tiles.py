"""The post-filter network's kernels at the sizes where a tile ends: pixel
tiles of 128 columns, K-steps of 16 pixels, row strips and segments, images
of one row, one column and one pixel.  Weights, inputs and targets are
dyadic, wired so that every activation is exact in bf16 (asserted here) and
every gradient the exact sum of two products, so that the only roundings are
the network's own: the gradient's scale and the gradients between the layers
to bf16, which the reference applies to the fp64 oracle's operations."""
import numpy as np
import pytest

from oracle import cnn as OC

torch = pytest.importorskip("torch")

SHAPES = [(1, 1, 1), (2, 1, 5), (1, 5, 1), (1, 3, 17), (3, 4, 16), (1, 9, 120), (2, 6, 121), (1, 7, 127), (2, 4, 128),
          (1, 16, 129), (1, 33, 130), (2, 21, 145), (1, 40, 241), (1, 70, 260)]


def bf16(a):
    u = np.asarray(a, np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def dyadic_net(seed):
    """Every hidden channel reads two channels of the layer below, and is read
    by two of the layer above, with weights of one half."""
    rng = np.random.default_rng(seed)
    layers = []
    for co, ci in OC.SHAPES:
        w = np.zeros((co, ci, 3, 3))
        if co == 1:
            for c in range(ci):
                w[0, c, rng.integers(3), rng.integers(3)] = rng.choice([-0.125, 0.125])
        else:
            for o, (a, b) in enumerate(zip(rng.permutation(max(ci, 32)) % ci, rng.permutation(max(ci, 32)) % ci)):
                w[o, a, rng.integers(3), rng.integers(3)] += 0.5
                w[o, b, rng.integers(3), rng.integers(3)] += rng.choice([-0.5, 0.5])
        layers.append((w, rng.integers(0, 2, co) / 8.0))
    return layers


def workload(shape):
    rng = np.random.default_rng(sum(shape))
    layers = dyadic_net(shape[2])
    x = rng.integers(0, 4, shape) / 4.0
    y, acts = OC.forward(layers, x)
    t = y + rng.choice([-1.0, 1.0], shape)
    return layers, x, y, acts, t


@pytest.mark.parametrize("shape", SHAPES)
def test_workload_is_exact(shape):
    """The premise: activations and outputs are exact in the network's types."""
    layers, x, y, acts, t = workload(shape)
    for a in acts[1:-1]:
        assert np.array_equal(bf16(a), a)
    assert np.array_equal(y.astype(np.float32), y) and np.array_equal(t.astype(np.float32), t)


def gradients(layers, x, y, acts, t):
    """The oracle's backward pass with the gradients between the layers held
    as bf16, as the network holds them: per layer and tensor the gradient and
    the largest sum of its terms' magnitudes (what fp32 summation errors are
    relative to; the terms have both signs)."""
    def layer(a, g):
        s = np.abs(g)
        return [(OC.conv3x3_grad_weight(a, g), OC.conv3x3_grad_weight(np.abs(a), s).max()),
                (g.sum(axis=(0, 2, 3)), s.sum(axis=(0, 2, 3)).max())]

    dz = (np.float32(2.0) / np.float32(x.size)) * (y - t).astype(np.float32)
    g = dz.astype(np.float64)[:, None]
    out = [layer(acts[4], g)]
    g = bf16(dz)[:, None]
    for k in range(4, 0, -1):
        g = bf16(OC.conv3x3_grad_input(g, layers[k][0]) * (acts[k] > 0))
        out.insert(0, layer(acts[k - 1], g))
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
def test_exact_workload(shape):
    from paper_2208_10859_gb300 import wv
    layers, x, y, acts, t = workload(shape)
    flat = np.concatenate([np.concatenate([w.ravel(), b]) for w, b in layers]).astype(np.float32)
    net = wv.CNN(flat)
    xd, td = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (x, t))
    assert np.array_equal(net.forward(xd).cpu().numpy(), y)
    loss, g = net.gradients(xd, td)
    assert loss == pytest.approx(float(np.mean((y - t) ** 2)), rel=1e-6)
    o = 0
    for k, tensors in enumerate(gradients(layers, x, y, acts, t)):
        for v, terms in tensors:
            got = g[o:o + v.size].astype(np.float64)
            o += v.size
            assert np.abs(got - v.ravel()).max() <= 1e-6 * terms, k
    assert net.sync_status() == 0
