"""The bound on the pixels that can see a volume (screen_bound.h), which sizes
sample buffers: compiled for the host and compared with projections of random
points of the box, and with the pixels where the oracle finds entry and exit
pairs."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1404_3363_gb300 import scenes

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1404_3363_gb300", "csrc")


@pytest.fixture(scope="module")
def pixels_met(tmp_path_factory):
    d = tmp_path_factory.mktemp("screen_bound")
    src = d / "b.cpp"
    src.write_text('#include "screen_bound.h"\n'
                   "struct Frame { double eye[3], f[3], r[3], u[3], sx, sy; int ortho, W, H, x0, y0, w, h; };\n"
                   'extern "C" double b(const Frame* f, const double* lo, const double* hi) '
                   "{ return ivv::pixels_met(*f, lo, hi); }\n")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(d / "b.so")],
                   check=True)
    b = ctypes.CDLL(str(d / "b.so")).b
    b.restype = ctypes.c_double

    class Frame(ctypes.Structure):
        _fields_ = [(n, ctypes.c_double * 3) for n in ("eye", "f", "r", "u")] + \
                   [(n, ctypes.c_double) for n in ("sx", "sy")] + \
                   [(n, ctypes.c_int) for n in ("ortho", "W", "H", "x0", "y0", "w", "h")]

    def call(cam, lo, hi, full, window):
        eye, f = np.array(cam.eye, float), np.subtract(cam.target, cam.eye)
        f = f / np.linalg.norm(f)
        r = np.cross(f, cam.up)
        r /= np.linalg.norm(r)
        u = np.cross(r, f)
        sy = 0.5 * cam.ortho_height if cam.ortho else np.tan(0.5 * np.radians(cam.fovy_deg))
        v3 = ctypes.c_double * 3
        fr = Frame(v3(*eye), v3(*f), v3(*r), v3(*u), sy * full[0] / full[1], sy, int(cam.ortho), *full, *window)
        return b(ctypes.byref(fr), v3(*lo), v3(*hi)), (eye, f, r, u, sy * full[0] / full[1], sy)

    return call


@pytest.mark.parametrize("ortho", [True, False])
def test_points_of_the_box_lie_within(pixels_met, ortho):
    """Every pixel that a point of the box before the eye projects to counts:
    the bound is at least the extent of the projections in the window, and at
    most the window."""
    rng = np.random.default_rng(11)
    for _ in range(300):
        lo = rng.normal(size=3)
        hi = lo + 10.0 ** rng.uniform(-2, 1, 3)
        centre, diag = 0.5 * (lo + hi), np.linalg.norm(hi - lo)
        eye = centre + rng.normal(size=3) * diag * 10.0 ** rng.uniform(-1, 1)
        target = centre + rng.normal(size=3) * diag
        cam = scenes.Camera(ortho, tuple(eye), tuple(target), tuple(rng.normal(size=3)),
                            fovy_deg=rng.uniform(5, 120), ortho_height=diag * 10.0 ** rng.uniform(-1, 1))
        W, H = (int(x) for x in rng.integers(16, 400, 2))
        w, h = int(rng.integers(1, W + 1)), int(rng.integers(1, H + 1))
        x0, y0 = int(rng.integers(0, W - w + 1)), int(rng.integers(0, H - h + 1))
        got, (e, f, r, u, sx, sy) = pixels_met(cam, lo, hi, (W, H), (x0, y0, w, h))
        assert 0 <= got <= w * h
        p = lo + rng.uniform(size=(4000, 3)) * (hi - lo) - e
        z = p @ f
        q = np.ones_like(z) if ortho else z
        ok = z > 0
        x = ((p @ r)[ok] / q[ok] / sx + 1) / 2 * W - x0
        y = (1 - (p @ u)[ok] / q[ok] / sy) / 2 * H - y0
        inside = (x > 0) & (x < w) & (y > 0) & (y < h)
        if inside.any():
            nx = int(np.floor(x[inside].max())) - int(np.floor(x[inside].min())) + 1
            ny = int(np.floor(y[inside].max())) - int(np.floor(y[inside].min())) + 1
            assert got >= nx * ny


@pytest.mark.parametrize("scene", [scenes.twisted_cube, scenes.twisted_bar, scenes.bent_beam, scenes.backstep])
def test_pixels_with_pairs_are_within(pixels_met, scene):
    sc = scene(width=120, height=90)
    lo, hi = sc.cp_bbox()
    got, _ = pixels_met(sc.camera, lo, hi, (120, 90), (0, 0, 120, 90))
    cnt = oracle.OracleVolume(sc.blocks, sc.scalar_mode).window_pairs(sc.camera, 120, 90, cap=4)[0].reshape(90, 120)
    ys, xs = np.nonzero(cnt)
    assert got >= (np.ptp(xs) + 1) * (np.ptp(ys) + 1) >= cnt.astype(bool).sum()
    assert got <= 0.6 * 120 * 90
