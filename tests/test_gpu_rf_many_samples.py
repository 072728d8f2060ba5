"""Root finding where one group of pixels has far more samples than the others:
a thin plate over a whole window and a rod seen from its end, whose rays take
140 times the samples of the plate's.  At 3840 x 2160 with 2.0e9 samples there
are more (group, chunk of four samples) combinations than an int holds; small
windows take chunks of every length.  The frames equal their windows around the
rod and at the plate's edge, rendered alone.  Beyond INT_MAX samples the call is
refused, from every start."""
import dataclasses

import numpy as np
import pytest

from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

T = 0.05


def plate_and_rod(width, height, samples):
    kn = np.array([0, 0, 0, 0, 1, 1, 1, 1], dtype=np.float64)
    g = np.linspace(0, 1, 4)
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    unit = np.stack([x, y, z], -1)
    rng = np.random.default_rng(9)
    box = [((-1.0, -0.6, 0.0), (1.0, 0.6, T)), ((0.3, 0.2, 0.1), (0.315, 0.215, 0.1 + 140 * T))]
    blocks = [scenes.Block((3, 3, 3), [kn.copy() for _ in range(3)], np.array(a) + unit * (np.array(b) - np.array(a)),
                           rng.uniform(0, 1, (4, 4, 4))) for a, b in box]
    base = scenes.degenerate_cube(width=width, height=height)
    cam = scenes.Camera(True, (0.0, 0.0, -3.0), (0.0, 0.0, 1.0), (0.0, 1.0, 0.0), ortho_height=1.1)
    tf = dataclasses.replace(base.tf, sigma=0.5)
    prm = dataclasses.replace(base.params, method=1, use_mlp_guess=2, rf_tol=1e-3, ds=T / samples)
    return dataclasses.replace(base, name="plate_and_rod", blocks=blocks, tf=tf, camera=cam, params=prm)


def _same(a, b):
    assert a[..., 3].max() > 0.0
    assert np.abs(a - b).max() <= 1e-6


# samples on a ray of the plate; 240.5 of them on 3840 x 2160 pixels: 2.0e9
@pytest.mark.parametrize("w,h,samples", [(160, 90, 0.7), (160, 90, 3.5), (640, 360, 30.5), (3840, 2160, 240.5)])
def test_one_long_group(w, h, samples):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    sc = plate_and_rod(w, h, samples)
    vol = ivv.volume_for(sc)
    img = vol.render(sc.camera, sc.params, w, h).cpu().numpy()
    cnt = vol.render_pairs(sc.camera, sc.params, w, h, max_pairs=2)[0].cpu().numpy().reshape(h, w)
    assert cnt.min() == 1
    py, px = np.argwhere(cnt == 2)[0]
    for x0, y0 in ((int(px) - 16, int(py) - 16), (0, 0)):
        part = vol.render(sc.camera, sc.params, 33, 35, window=(x0, y0, w, h)).cpu().numpy()
        _same(part, img[y0:y0 + 35, x0:x0 + 33])
    assert vol.stats()["rf_unconverged"] == 0


@pytest.mark.parametrize("cut_planes", [(), ((1.0, 0.0, 0.0, -0.9),)])      # counted in stage 2, and after it
@pytest.mark.parametrize("guess", [0, 1, 2])
def test_beyond_int_max(guess, cut_planes):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    w, h = 3840, 2160
    sc = plate_and_rod(w, h, 300.5)
    vol = ivv.volume_for(sc)
    if guess == 1:
        vol.train_guess(samples_per_block=1 << 10, epochs=1, batch=1024)
    with pytest.raises(ivv.IvvError, match="UNSUPPORTED"):
        vol.render(sc.camera, dataclasses.replace(sc.params, use_mlp_guess=guess, cut_planes=cut_planes), w, h)
