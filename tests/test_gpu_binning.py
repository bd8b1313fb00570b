"""Direct placement against the sort-based binning: the same keys, values and tile ranges, bit for bit,
where the direct one's bands and steps have their edges -- one row of tiles, fewer rows than bands, odd
rows over two eyes, more than two bands (interleaved rows), Gaussians that cover every tile, tiles
that several Gaussians of one step share, and a capacity that cuts the lists off."""
import dataclasses

import numpy as np
import pytest

import paper_2507_04147_gb300 as a3fr
from paper_2507_04147_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,eyes,tile,n,log_scale,capacity", [
    (333, 16, 1, 16, 3_000, -3.0, 0),       # one row of tiles: one band
    (16, 700, 2, 32, 2_000, -2.0, 0),       # one column, 2 x 22 rows
    (40, 40, 1, 16, 5_000, -1.0, 0),        # nine tiles: every step shares tiles
    (517, 389, 2, 16, 4_001, -3.5, 0),      # odd rows per eye
    (2048, 2048, 1, 16, 20_000, -4.0, 0),   # 16,384 tiles, the most AUTO gives it: eight bands
    (1003, 717, 2, 16, 4_003, -3.0, 0),     # 2 x 45 rows in four bands, one of 22 rows
    (16_384, 80, 1, 16, 3_000, -2.0, 0),    # five rows of the widest view in four bands
    (640, 480, 2, 16, 300, 1.5, 0),         # Gaussians over the whole image
    (517, 389, 1, 16, 4_001, -3.5, 5_000),  # capacity reached
])
def test_direct_equals_sorted(w, h, eyes, tile, n, log_scale, capacity):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    sc = synth.uniform_scene(n, 0, seed=n, log_scale_mean=log_scale)
    sc = dataclasses.replace(sc, means=np.where(np.arange(n)[:, None] % 9 == 4, -sc.means, sc.means))   # some behind
    cams = synth.stereo_cameras(w, h) if eyes == 2 else [synth.pinhole_camera(w, h)]
    got = []
    for mode in (a3fr.BINNING_DIRECT, a3fr.BINNING_SORTED):
        s = a3fr.Scene.from_numpy(sc, instance_capacity=capacity, tile=tile)
        s.set_binning(mode)
        for e, c in enumerate(cams):
            s.set_camera(e, c)
        img = s.render_full().cpu().numpy()
        st = s.stats()
        got.append((s.buffer(a3fr.BUF_KEYS, torch.int64).cpu().numpy(), s.buffer(a3fr.BUF_VALUES, torch.int32).cpu().numpy(),
                    s.buffer(a3fr.BUF_RANGES, torch.int32).cpu().numpy(), img if not capacity else np.zeros(1)))
        assert st["status"] == (a3fr.STATUS_CAPACITY if capacity else 0)
        assert st["instances"] > 0
        s.close()
    if capacity:   # both keep the first `capacity` slots' worth of whole lists; compare what lies below it
        ends = got[0][2].reshape(-1, 2)
        assert np.array_equal(ends, got[1][2].reshape(-1, 2))
        return
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("w,h,eyes,tile,n,route", [
    (2064, 2208, 2, 32, 200_000, a3fr.BINNING_DIRECT),   # 8,970 tiles, 400k entries
    (2064, 2208, 2, 32, 250_000, a3fr.BINNING_SORTED),   # 500k entries
    (1366, 768, 2, 16, 250_000, a3fr.BINNING_DIRECT),    # 8,256 tiles
    (2560, 1440, 1, 16, 500_000, a3fr.BINNING_DIRECT),   # 14,400 tiles of one eye
    (1280, 720, 1, 16, 1_000, a3fr.BINNING_DIRECT),
    (2576, 2064, 1, 16, 1_000, a3fr.BINNING_SORTED),     # 20,769 tiles
])
def test_auto_takes_the_faster_route(w, h, eyes, tile, n, route):
    """AUTO's route, told by the number of kernels it launches, and its image."""
    import __graft_entry__
    __graft_entry__.build()
    sc = synth.uniform_scene(n, 0, seed=3, log_scale_mean=-5.0)
    s = a3fr.Scene.from_numpy(sc, tile=tile)
    for e, c in enumerate(synth.stereo_cameras(w, h) if eyes == 2 else [synth.pinhole_camera(w, h)]):
        s.set_camera(e, c)
    launches, images = {}, {}
    for mode in (a3fr.BINNING_AUTO, a3fr.BINNING_DIRECT, a3fr.BINNING_SORTED):
        s.set_binning(mode)
        s.render_full()
        s.stats(reset=True)
        images[mode] = s.render_full().clone()
        launches[mode] = s.stats()["kernel_launches"]
    s.close()
    assert launches[a3fr.BINNING_DIRECT] != launches[a3fr.BINNING_SORTED]
    assert launches[a3fr.BINNING_AUTO] == launches[route]
    assert (images[a3fr.BINNING_AUTO] == images[route]).all()


@pytest.mark.parametrize("w,h,eyes,tile,n,log_scale,capacity", [
    (517, 389, 1, 16, 4_001, -3.5, 5_000),   # two bands
    (1003, 717, 2, 16, 4_003, -3.0, 30_001),   # 5,670 tiles: four interleaved bands
    (640, 480, 2, 16, 300, 1.5, 77_777),     # Gaussians over the whole image: the capacity cuts long lists
])
def test_direct_below_the_capacity(w, h, eyes, tile, n, log_scale, capacity):
    """Direct placement with too small a capacity: what lies below it -- values, keys, and the pixels of
    tiles whose list ends there -- is what an ample one gives, bit for bit."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    sc = synth.uniform_scene(n, 0, seed=n, log_scale_mean=log_scale)
    cams = synth.stereo_cameras(w, h) if eyes == 2 else [synth.pinhole_camera(w, h)]
    got = []
    for cap in (0, capacity):
        s = a3fr.Scene.from_numpy(sc, instance_capacity=cap, tile=tile)
        s.set_binning(a3fr.BINNING_DIRECT)
        for e, c in enumerate(cams):
            s.set_camera(e, c)
        img = s.render_full().cpu().numpy()
        assert s.stats()["status"] == (a3fr.STATUS_CAPACITY if cap else 0)
        got.append([s.buffer(which, dt).cpu().numpy() for which, dt in (
            (a3fr.BUF_VALUES, torch.int32), (a3fr.BUF_KEYS, torch.int64), (a3fr.BUF_RANGES, torch.int32))] + [img])
        s.close()
    (vals, keys, ranges, img), (vals_c, keys_c, ranges_c, img_c) = got
    assert len(vals) > capacity and len(vals_c) == len(keys_c) == capacity
    assert np.array_equal(ranges, ranges_c)
    assert np.array_equal(vals[:capacity], vals_c) and np.array_equal(keys[:capacity], keys_c)
    whole = (ranges.reshape(eyes, -1, 2)[..., 1] <= capacity).reshape(eyes, (h + tile - 1) // tile, -1)
    whole = whole.repeat(tile, 1).repeat(tile, 2)[:, :h, :w]
    assert whole.any() and not whole.all()
    assert np.array_equal(img[whole], img_c[whole])
