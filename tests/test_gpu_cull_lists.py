"""The cull's item list where one 8 x 4 tile meets many patches (more than the
32 that a warp gathers before it appends them) and where few: tiny images of
volumes with hundreds of face patches, ragged sizes, against the FP64 oracle
(max |dRGBA| <= 1e-3, the suite's bound for small FP32 images)."""
import numpy as np
import pytest

import oracle
from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(1, 1), (9, 5), (16, 9)])
@pytest.mark.parametrize("name", ["twisted_bar", "bent_beam"])
def test_tiny_images_match_the_oracle(name, size):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    w, h = size
    sc = getattr(scenes, name)(width=w, height=h, precision=0)
    vol = ivv.volume_for(sc)
    vol.reset_stats()
    img = vol.render(sc.camera, sc.params, w, h, flags=ivv.FLAG_STATS).cpu().numpy().astype(np.float64)
    assert vol.stats()["abuf_overflow"] == 0
    ref = oracle.render(sc, oracle.OracleVolume(sc.blocks, sc.scalar_mode))
    assert np.abs(img - ref).max() <= 1e-3
    assert name == "bent_beam" or (ref[..., 3] > 0.05).any()
