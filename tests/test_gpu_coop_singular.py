"""Small FP64 frames (a group of lanes per ray, k_coop64.cuh) where the
Jacobian is singular on a face: right-hand sides are infinite there, and so is
the error of a step that touches it, which has to be retried shorter.  A half
cylinder by radius, angle and height, whose axis is a collapsed face, seen by
rays that pass it at 1e-5 to 8e-4, and the cube with a degenerate face from
above and below, against the one-lane kernel, which a frame with statistics
takes, and the cube against the FP64 oracle (next to the cylinder's axis, where
the scalar depends on the angle, the oracle itself is 4e-3 off the closed form
of that map).  No ray may reach the step cap, set far above the some 160 steps
that these rays take."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def half_cylinder(width, height):
    kn = np.array([0, 0, 0, 0, 1, 1, 1, 1], dtype=np.float64)
    arc = np.array([(1, 0), (1, 4 / 3), (-1, 4 / 3), (-1, 0)])
    cp = np.zeros((4, 4, 4, 3))
    for k in range(4):
        for j in range(4):
            for i in range(4):
                cp[k, j, i] = (*(arc[j] * i / 3), k / 3)
    scal = np.random.default_rng(5).uniform(0, 1, (4, 4, 4))
    blk = scenes.Block((3, 3, 3), [kn.copy(), kn.copy(), kn.copy()], cp, scal)
    base = scenes.degenerate_cube(width=width, height=height)
    d = np.array([0.3, -1.0, 0.1])
    target = np.array([0.0, 0.0, 0.5])
    cam = scenes.Camera(True, tuple(target - 4 * d), tuple(target), (0.0, 0.0, 1.0), ortho_height=1.6e-3)
    prm = dataclasses.replace(base.params, ds=np.sqrt(4 + 16 / 9 + 1) / 128)
    return dataclasses.replace(base, name="half_cylinder", blocks=[blk], camera=cam, params=prm)


def _scene(name):
    if name == "half_cylinder":
        return half_cylinder(48, 48)
    return scenes.degenerate_cube(width=64, height=64,
                                  direction=(0.35, 0.25, 0.9) if name == "cube_above" else (0.35, 0.25, -0.9))


@pytest.mark.parametrize("tol", [1e-4, 1e-5, 1e-6])
@pytest.mark.parametrize("name", ["half_cylinder", "cube_above", "cube_below"])
def test_steps_touching_a_singular_face(name, tol):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    sc = _scene(name)
    sc.params = dataclasses.replace(sc.params, precision=2, rk_tol=tol)
    vol = ivv.volume_for(sc)
    vol.set_limits(max_rk_steps=4000)
    img, caps = [], []
    for flags in (0, ivv.FLAG_STATS):
        vol.reset_stats()
        img.append(vol.render(sc.camera, sc.params, sc.width, sc.height, flags=flags).cpu().numpy())
        caps.append(vol.stats()["step_cap"])
    assert np.isfinite(img[0]).all() and img[0][..., 3].max() > 0.1
    assert caps == [0, 0]
    # same steps; images are FP32
    assert np.abs(img[0] - img[1]).max() <= 1e-6
    if name != "half_cylinder" and tol <= 1e-5:
        assert np.abs(img[0] - oracle.render(sc)).max() <= 1e-3
