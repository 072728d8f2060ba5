"""Root finding on frames whose active pixels do not fill their groups of 32:
one pixel, a few, odd widths, pixels with several pairs, samples counted by the
stage-2 kernel and (cutting planes) after the fix-up solves, every start, few
and many blocks.  Images against the FP64 oracle (1e-3, rf_tol 1e-3 of the
pixel half width), and every start gives the same image: each solve ends within
rf_tol of the pixel, 1e-3 of half a pixel, so twice that times the scalar's and
the transfer function's slopes, below 1e-3 as well."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,kw,size,params", [
    ("twisted_cube", {"precision": 0}, (1, 1), {}),
    ("twisted_cube", {"precision": 0}, (7, 5), {"supersample_k": 3}),
    ("twisted_bar", {}, (61, 35), {}),
    ("bent_beam", {"precision": 1}, (83, 47), {"cut_planes": ((0.2, 0.1, 0.9, -3.0),)}),
    ("backstep", {"precision": 0}, (75, 43), {}),
])
def test_rf_small_frames(name, kw, size, params):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    sc = getattr(scenes, name)(width=size[0], height=size[1], **kw)
    r = np.linspace(0, 1, len(sc.tf.r), dtype=np.float32)
    prm = dataclasses.replace(sc.params, method=1, rf_tol=1e-3, **params)
    sc = dataclasses.replace(sc, tf=dataclasses.replace(sc.tf, r=r), params=prm)
    vol = ivv.volume_for(sc)
    vol.train_guess(samples_per_block=1 << 14, epochs=8, batch=2048, seed=2)
    ref = oracle.render(sc)
    for guess in (0, 1, 2):
        p = dataclasses.replace(prm, use_mlp_guess=guess)
        for flags in (0, ivv.FLAG_STATS):
            img = vol.render(sc.camera, p, size[0], size[1], flags=flags).cpu().numpy()
            assert np.abs(img - ref).max() <= 1e-3, (guess, flags)
