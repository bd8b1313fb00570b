"""Non-finite values in the backward stay where they are blended: an image gradient that is NaN or
infinite at one pixel, and a Gaussian of infinite colour, reach the gradients of the Gaussians blended
at the same pixels and no others -- not those that the kernel only evaluates because they share a patch
of pixels.  Both shapes of the kernel (half quadrants for the small image, quadrants above 16 per SM)."""
import dataclasses

import numpy as np
import pytest

import paper_2507_04147_gb300 as a3fr
from paper_2507_04147_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [(96, 64, 16, 600, -2.8), (96, 64, 32, 600, -2.8), (1024, 640, 16, 20_000, -3.6)]


def grads_and_records(sc, cam, tile, dls):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    s = a3fr.Scene.from_numpy(sc, tile=tile)
    s.set_camera(0, cam)
    s.keep_aux(True)
    s.render_full()
    rec = s.buffer(a3fr.BUF_RECORDS, torch.float32).cpu().numpy().reshape(-1, 12)
    out = [{k: v.cpu().numpy() for k, v in s.backward(torch.from_numpy(d).cuda()).items()} for d in dls]
    s.close()
    return out, rec


def may_touch(rec, xy, slack=0.99):
    """[n]: whether a Gaussian may be blended at one of the pixels xy [p, 2] (its alpha >= 1/255 there,
    with a margin for rounding; slack > 1: whether it surely reaches that)."""
    with np.errstate(all="ignore"):
        r = rec.astype(np.float64)[:, None, :]
        dx, dy = r[..., 0] - xy[None, :, 0], r[..., 1] - xy[None, :, 1]
        power = -0.5 * (r[..., 2] * dx * dx + r[..., 4] * dy * dy) - r[..., 3] * dx * dy
        return ((r[..., 11] != 0) & (r[..., 5] * np.exp(np.minimum(power, 0.0)) >= slack / 255.0)).any(1)


def check(got, ref, free):
    assert free.sum() > 0.5 * len(free)
    for k in got:
        a, b = got[k][free], ref[k][free]
        assert np.isfinite(a).all(), (k, int((~np.isfinite(a)).sum()))
        # the same terms in another order of fp32 additions
        assert np.abs(a - b).max() <= 1e-3 * np.abs(b).max(), k


@pytest.mark.parametrize("w,h,tile,n,log_scale", SIZES)
def test_image_gradient_of_one_pixel(w, h, tile, n, log_scale):
    cam = synth.pinhole_camera(w, h)
    sc = synth.uniform_scene(n, 1, seed=n, log_scale_mean=log_scale)
    x, y = w // 2 + 3, h // 2 - 5
    dl = np.random.default_rng(n).normal(size=(1, h, w, 3)).astype(np.float32)
    dl[0, y, x] = 0.0
    bad = dl.copy()
    bad[0, y, x] = (np.nan, 1.0, np.inf)
    (ref, got), rec = grads_and_records(sc, cam, tile, (dl, bad))
    pixel = np.array([[x, y]], np.float64)
    check(got, ref, ~may_touch(rec, pixel))
    touched = may_touch(rec, pixel, 1.01)
    assert touched.any() and not np.isfinite(got["sh"][touched]).all()   # and it does reach those


@pytest.mark.parametrize("w,h,tile,n,log_scale", SIZES)
def test_infinite_colour_of_one_gaussian(w, h, tile, n, log_scale):
    cam = synth.pinhole_camera(w, h)
    sc = synth.uniform_scene(n, 1, seed=n + 1, log_scale_mean=log_scale)
    dl = np.random.default_rng(n).normal(size=(1, h, w, 3)).astype(np.float32)
    (ref,), rec = grads_and_records(sc, cam, tile, (dl,))
    # an opaque one in the middle of the image
    mid = (rec[:, 11] != 0) & (np.abs(rec[:, 0] - w / 2) < w / 4) & (np.abs(rec[:, 1] - h / 2) < h / 4)
    i = int(np.argmax(np.where(mid, rec[:, 5], -1.0)))
    sh = sc.sh.copy()
    sh[i] = 0.0
    sh[i, 0] = np.inf
    (got,), rec2 = grads_and_records(dataclasses.replace(sc, sh=sh), cam, tile, (dl,))
    assert np.isinf(rec2[i, 6:9]).all()
    xs, ys = np.meshgrid(np.arange(w), np.arange(h))
    xy = np.stack([xs.ravel(), ys.ravel()], 1).astype(np.float64)
    r = float(rec[i, 10]) + 32.0   # its pixels lie within its radius
    xy = xy[(np.abs(xy[:, 0] - rec[i, 0]) <= r) & (np.abs(xy[:, 1] - rec[i, 1]) <= r)]
    own = np.array([may_touch(rec[i:i + 1], p[None])[0] for p in xy])
    assert own.any()
    check(got, ref, ~may_touch(rec, xy[own]))
