"""The tensor-core convolutions and weight gradients where their rings of stages wrap (a CTA takes more
than 12 tiles of a convolution, more than 4 of a weight gradient) and at the edges of their tiles.

The networks here have non-negative weights, biases and inputs and a target below every prediction, so
every sum the kernels form has non-negative terms: no cancellation, and a relative bound holds for every
element of the gradient, tap by tap."""
import numpy as np
import pytest

import paper_2507_04147_gb300 as a3fr
from paper_2507_04147_gb300 import periphery

pytestmark = pytest.mark.gpu

ARCHS = [periphery.RESIDUAL, periphery.COMPACT]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def positive_net(seed, arch, bias):
    """(weights, biases): mean output of a layer about its mean input."""
    rng = np.random.default_rng(seed)
    ws, bs = periphery.unpack(periphery.init_params(seed, arch).copy(), arch)
    ws = [rng.uniform(0.2, 1.8, w.shape).astype(np.float32) / np.prod(w.shape[1:]) for w in ws]
    ws[0][:, 4:] = 0.0
    bs = [rng.uniform(0.0, bias, b.shape).astype(np.float32) for b in bs]
    return ws, bs


def cuda(*arrays):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda() for a in arrays]


@pytest.mark.parametrize("arch", ARCHS)
def test_a_batch_equals_its_crops(arch):
    """16 crops of 180 x 170 blocks are 4,224 tiles, 28 a CTA of 152: the convolutions' ring of 12 wraps
    twice, the weight gradients' ring of 4 six times; a crop alone is 264 tiles, at most two a CTA.  The
    residuals agree bit for bit.  The batch's mean gradient is the crops' average: a factor of 16 is
    exact in every BF16 and fp32 value, so only the order of the fp32 sums differs.  The longest chain
    is 28 tiles x 8 MMAs of 17 terms, then 152 CTAs' partial sums; a crop's is 2 x 8 x 17 and 152; an
    addition is off by at most 2^-23 of the (non-negative) sum, however it rounds: 5.3e-4."""
    import torch
    b, h, w = 16, 359, 339
    rng = np.random.default_rng(7 + arch)
    ws, bs = positive_net(3, arch, 0.05)
    img, depth = cuda(rng.uniform(0, 1, (b, h, w, 3)), rng.uniform(0, 6, (b, h, w)))
    target = torch.full_like(img, -0.25)
    net = periphery.Periphery(periphery.pack(ws, bs), arch=arch)
    res = net.forward(img, depth)
    g, loss = net.grads(img, depth, target)
    total = np.zeros(g.shape, np.float64)
    losses = []
    for k in range(b):
        one = [t[k:k + 1].contiguous() for t in (img, depth, target)]
        assert torch.equal(net.forward(*one[:2])[0], res[k]), k
        gk, lk = net.grads(*one)
        total += gk
        losses.append(lk)
    net.close()
    assert loss == pytest.approx(np.mean(losses), rel=1e-3)
    ref = total / b
    ws, bs = [np.ones_like(v) for v in ws], [np.ones_like(v) for v in bs]
    ws[0][:, 4:] = 0.0                        # padding channels of the input
    ws[-1][12:] = bs[-1][12:] = 0.0           # and of the residuals
    used = periphery.pack(ws, bs) > 0.0
    assert np.array_equal(used, ref > 0.0) and np.array_equal(used, g > 0.0)
    rel = np.abs(g[used] - ref[used]) / ref[used]
    assert rel.max() <= 5.3e-4, rel.max()


@pytest.mark.parametrize("arch", ARCHS)
@pytest.mark.parametrize("y,x", [(0, 0), (34, 22), (15, 7), (16, 8), (31, 16), (0, 22)])
def test_gradients_of_one_bright_block(arch, y, x):
    """One lit block of a 35 x 23 image (ragged tiles of 16 x 8 blocks) and no biases: activations are
    zero away from it, so a product lost at a corner, an edge or a seam of tiles is a large part of some
    element.  Against the oracle, which keeps gradients in float64: up to ten tensors of them rounded to
    BF16 here (2^-9 each, 2 %), and a rounding of an activation to the other neighbour (2^-8): 3 %."""
    from oracle import cnn as ocnn
    h, w = 70, 45
    ws, bs = positive_net(11, arch, 0.0)
    img, depth = np.zeros((1, h, w, 3), np.float32), np.zeros((1, h, w), np.float32)
    img[0, 2 * y, 2 * x] = (1.0, 0.75, 0.5)
    depth[0, 2 * y, 2 * x] = 6.0
    target = np.full_like(img, -1.0)
    net = periphery.Periphery(periphery.pack(ws, bs), arch=arch)
    g, loss = net.grads(*cuda(img, depth, target))
    net.close()
    x0, tl = ocnn.make_input(img, depth)
    ref_loss, gw, gb, _ = ocnn.loss_and_grads(x0, tl, target, ws, bs,
                                              net=ocnn.forward_compact if arch else ocnn.forward)
    assert loss == pytest.approx(ref_loss, rel=2e-3)
    gws, gbs = periphery.unpack(g, arch)
    for li, (got_w, got_b, ref_w, ref_b) in enumerate(zip(gws, gbs, gw, gb)):
        for kind, got, ref in (("w", got_w, ref_w.reshape(got_w.shape)), ("b", got_b, ref_b)):
            assert np.array_equal(got > 0, ref > 0), (li, kind)
            rel = np.abs(got - ref)[ref > 0] / ref[ref > 0]
            assert rel.size == 0 or rel.max() <= 3e-2, (li, kind, rel.max())


@pytest.mark.parametrize("arch", ARCHS)
def test_fused_fill_where_the_ring_wraps(arch):
    """The fill of a stereo frame of 521 x 502 blocks an eye: 4,158 tiles, 28 a CTA, against the training
    forward's residuals composed by the test of the small sizes."""
    import test_gpu_cnn
    test_gpu_cnn.test_fused_fill_equals_forward_plus_compose(32, 1003, 1041, 2, arch)
