"""The learned guess's inference in pieces of the frame's places (a frame near
INT_MAX samples takes more than one): a library built with pieces of 4096 places
renders the same images as the ordinary one, with the starts sorted by block
(the beam, 16 blocks) and not (the bar).  A point's inference does not depend on
its neighbours, so the images are equal."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RENDER = """
import dataclasses, sys
import numpy as np
from paper_1404_3363_gb300 import ivv, scenes
ivv.load(sys.argv[1])
frames = {}
for name in ("bent_beam", "twisted_bar"):
    sc = getattr(scenes, name)(width=321, height=203)
    vol = ivv.volume_for(sc)
    vol.train_guess(samples_per_block=1 << 14, epochs=4, batch=2048, seed=2)
    prm = dataclasses.replace(sc.params, method=1, use_mlp_guess=1, rf_tol=1e-3)
    frames[name] = vol.render(sc.camera, prm, 321, 203, flags=ivv.FLAG_STATS).cpu().numpy()
    frames[name + "_newton"] = vol.stats()["rf_newton_iters"]
np.savez(sys.argv[2], **frames)
"""


def test_pieces_render_the_same(tmp_path):
    from paper_1404_3363_gb300 import build
    lib = build.build()
    pieces = str(tmp_path / "libpieces.so")
    objs = {s: os.path.join(build.OUT_DIR, s + ".o") for s in build.CU_SOURCES + build.CXX_SOURCES}
    objs["ivv_api.cu"] = str(tmp_path / "ivv_api.o")
    subprocess.run([build.NVCC] + build.ARCH + build.CU_FLAGS + ["-DIVV_INFER_PLACES=4096", "-c",
                    os.path.join(build.SRC_DIR, "ivv_api.cu"), "-o", objs["ivv_api.cu"]], check=True)
    subprocess.run([build.NVCC] + build.ARCH + ["-shared", "-o", pieces] + list(objs.values()), check=True)
    out = []
    for k, path in enumerate((lib, pieces)):
        f = str(tmp_path / ("%d.npz" % k))
        subprocess.run([sys.executable, "-c", RENDER, path, f], check=True,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
        out.append(np.load(f))
    assert out[0]["bent_beam"].max() > 0
    for key in out[0].files:
        assert np.array_equal(out[0][key], out[1][key]), key
