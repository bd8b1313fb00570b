"""The two shapes of the 16-pixel-tile composite (a tile per work item, and half tiles for renders of
few tiles) give the same pixels bit for bit: images of the same camera one row of tiles apart, on
either side of the line between them, agree on the rows they share."""
import numpy as np
import pytest

import paper_2507_04147_gb300 as a3fr
from paper_2507_04147_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 2])
@pytest.mark.parametrize("aux", [False, True])
@pytest.mark.parametrize("levels", [(4,), (3,), (1,), (4, 3, 2, 1)])
def test_shapes_agree_across_the_line(levels, aux, batch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cols = 64
    rows = 16 * sms // cols                      # the most rows of tiles rendered in halves
    width = 16 * cols - 5                        # ragged columns
    scene_np = synth.uniform_scene(30_000, 1, seed=5, log_scale_mean=-3.5)
    base = synth.pinhole_camera(width, 16 * rows, 90.0)
    out = []
    for h in (16 * rows, 16 * (rows + 1)):
        s = a3fr.Scene.from_numpy(scene_np)
        s.set_batch(batch)
        s.keep_aux(aux)
        s.set_camera(0, synth.Camera(width, h, base.fx, base.fy, base.cx, base.cy, base.znear, base.world_to_cam))
        s.set_gaze([[0.4 * width, 6.0 * rows]])
        img = s.render_foveated(a3fr.Fovea((4.0, 9.0, 16.0)[:len(levels) - 1], 0.0, levels))
        got = [img[0, :16 * rows].cpu().numpy()]
        if aux:
            for which, dt in ((a3fr.BUF_T_FINAL, torch.float32), (a3fr.BUF_N_CONTRIB, torch.int32),
                              (a3fr.BUF_DEPTH, torch.float32)):
                got.append(s.buffer(which, dt).cpu().numpy().reshape(h, width)[:16 * rows])
        assert s.stats()["status"] == 0
        s.close()
        out.append(got)
    assert out[0][0].max() > 0.1
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("levels", [None, (4, 3, 2, 1)])
def test_backward_shapes_agree_across_the_line(levels):
    """The same for the backward (quadrants and half quadrants): with no gradient in the taller
    image's last row of tiles the gradients agree up to the order of fp32 sums (of a few thousand terms: ~1e-6 of a
    group's norm; 1e-4 allowed)."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cols = 64
    rows = 16 * sms // cols
    width = 16 * cols - 5
    scene_np = synth.uniform_scene(30_000, 1, seed=6, log_scale_mean=-3.5)
    base = synth.pinhole_camera(width, 16 * rows, 90.0)
    dl = torch.randn(1, 16 * rows, width, 3, generator=torch.Generator().manual_seed(3))
    grads = []
    for h in (16 * rows, 16 * (rows + 1)):
        s = a3fr.Scene.from_numpy(scene_np)
        s.keep_aux(True)
        s.set_camera(0, synth.Camera(width, h, base.fx, base.fy, base.cx, base.cy, base.znear, base.world_to_cam))
        s.set_gaze([[0.4 * width, 6.0 * rows]])
        if levels is None:
            s.render_full()
        else:
            s.render_foveated(a3fr.Fovea((4.0, 9.0, 16.0), 0.0, levels))
        d = torch.zeros(1, h, width, 3)
        d[:, :16 * rows] = dl
        grads.append({k: v.cpu().double() for k, v in s.backward(d.cuda()).items()})
        s.close()
    for k in grads[0]:
        a, b = grads[0][k], grads[1][k]
        assert float(a.norm()) > 0
        assert float((a - b).norm()) <= 1e-4 * float(a.norm()), k
