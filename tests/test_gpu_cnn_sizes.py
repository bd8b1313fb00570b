"""Learned periphery at the edges of its tiles: gradients of images smaller than a tile, one row or
column past it, and with more tiles than one CTA takes, against the CPU oracle (the tolerances of
the ordinary sizes: BF16 storage is emulated, so what is left is fp32 summation and rare roundings
of a sum to the other BF16 neighbour, ~4e-4 measured there)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arch", [0, 1])
@pytest.mark.parametrize("b,h,w", [(1, 2, 2), (1, 33, 17), (3, 31, 34), (1, 64, 16), (2, 258, 270)])
def test_gradients_at_tile_edges(arch, b, h, w):
    import torch
    from oracle import cnn as ocnn
    from paper_2507_04147_gb300 import periphery
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(100 * h + w)
    ws, bs = periphery.unpack(periphery.init_params(h, arch), arch)
    ws = [v + rng.normal(0, 0.02, v.shape).astype(np.float32) for v in ws]
    ws[0][:, 4:] = 0.0
    bs = [rng.normal(0, 0.05, v.shape).astype(np.float32) for v in bs]
    img = rng.uniform(0, 1, (b, h, w, 3)).astype(np.float32)
    depth = rng.uniform(0, 6, (b, h, w)).astype(np.float32)
    target = np.clip(img + rng.normal(0, 0.1, img.shape), 0, 1).astype(np.float32)
    net = periphery.Periphery(periphery.pack(ws, bs), arch=arch)
    g, loss = net.grads(*(torch.from_numpy(a).cuda() for a in (img, depth, target)))
    net.close()
    x0, tl = ocnn.make_input(img, depth)
    ref_loss, gw, gb, _ = ocnn.loss_and_grads(x0, tl, target, ws, bs,
                                              net=ocnn.forward_compact if arch else ocnn.forward)
    assert loss == pytest.approx(ref_loss, rel=2e-3)
    gws, gbs = periphery.unpack(g, arch)
    for li, (got_w, got_b, ref_w, ref_b) in enumerate(zip(gws, gbs, gw, gb)):
        for got, ref in ((got_w, ref_w), (got_b, ref_b)):
            rel = np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-12)
            assert rel <= 5e-2, (li, rel)
