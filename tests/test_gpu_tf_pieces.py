"""The transfer function by pieces: two to 256 knots, steep ramps, doubled knots
at the ends, scalars beyond both ends of the range, several sub-sample counts;
single frames, every kernel that composites, against the oracle.

FP64: the colours are FP32 (1e-6), and a ramp of width 1/512 turns the FP32
rounding of the normalised scalar (6e-8) into 3e-5 per sub-sample: 1e-4.  FP32
kernels on maps without steep ramps: the suite's image bound, 1e-3."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _tf(kind, lo, hi):
    rng = np.random.default_rng(11)
    if kind == "two":
        r = np.array([0, 1])
    elif kind == "many":
        r = np.linspace(0, 1, 256)
    elif kind == "ramps":
        r = np.array([0, 0.25, 0.25 + 1 / 512, 0.5, 0.5 + 1 / 512, 0.75, 1])
    else:                                            # doubled knots at both ends
        r = np.array([0, 0, 0.4, 0.7, 1, 1])
    rgba = rng.uniform(0, 1, (len(r), 4))
    if kind == "many":                               # smooth: no slope beyond a few per unit
        t = r[:, None] * np.array([[1.0, 2.0, 3.0, 1.5]])
        rgba = 0.5 + 0.45 * np.sin(2 * t + rgba[:1])
    w = hi - lo
    return scenes.TransferFunction(r.astype(np.float32), rgba.astype(np.float32), 4.0, lo + 0.2 * w, hi - 0.2 * w)


@pytest.mark.parametrize("kind", ["two", "many", "ramps", "ends"])
@pytest.mark.parametrize("K", [1, 4, 5])
def test_tf_pieces(kind, K):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    sc = scenes.twisted_cube(width=40, height=30)
    s = sc.blocks[0].scalar_cp
    tf = _tf(kind, float(s.min()), float(s.max()))
    prm = dataclasses.replace(sc.params, precision=2, rk_tol=1e-8, supersample_k=K)
    sc = dataclasses.replace(sc, tf=tf, params=prm)
    vol = ivv.volume_for(sc)
    ref = oracle.render(sc)
    img = vol.render(sc.camera, prm, 40, 30).cpu().numpy()
    assert np.abs(img - ref).max() <= 1e-4
    if kind in ("two", "many"):
        for over in ({}, {"rk_method": 4}, {"method": 1, "rf_tol": 1e-3, "use_mlp_guess": 2}):
            p = dataclasses.replace(prm, precision=0, rk_tol=1e-5, **over)
            for flags in (0, ivv.FLAG_STATS):
                img = vol.render(sc.camera, p, 40, 30, flags=flags).cpu().numpy()
                assert np.abs(img - ref).max() <= 1e-3, (over, flags)
