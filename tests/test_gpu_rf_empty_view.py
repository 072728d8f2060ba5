"""Root finding on windows that no ray of the volume meets: a frame in view,
then one looking away (and back), with every start, with the starts sorted by
block (eight blocks and more) and not.  The empty frames are zero everywhere,
the frames in view equal each other."""
import dataclasses

import numpy as np
import pytest

from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("name", ["bent_beam", "twisted_bar"])       # 16 blocks, one
def test_frame_without_samples(name, prec):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    w, h = 160, 90
    sc = getattr(scenes, name)(width=w, height=h, precision=prec)
    eye, target = np.array(sc.camera.eye), np.array(sc.camera.target)
    away = dataclasses.replace(sc.camera, target=tuple(2 * eye - target))
    vol = ivv.volume_for(sc)
    vol.train_guess(samples_per_block=1 << 12, epochs=1, batch=1024, seed=3)
    for guess in (1, 2, 0):
        prm = dataclasses.replace(sc.params, method=1, use_mlp_guess=guess, rf_tol=1e-3)
        first = vol.render(sc.camera, prm, w, h).cpu().numpy()
        assert first[..., 3].max() > 0
        for flags in (0, ivv.FLAG_STATS):
            assert not vol.render(away, prm, w, h, flags=flags).cpu().numpy().any()
        assert np.array_equal(vol.render(sc.camera, prm, w, h).cpu().numpy(), first)
    # a new volume, whose sample buffer holds nothing yet
    fresh = ivv.volume_for(sc)
    fresh.train_guess(samples_per_block=1 << 12, epochs=1, batch=1024, seed=3)
    prm = dataclasses.replace(sc.params, method=1, use_mlp_guess=1, rf_tol=1e-3)
    assert not fresh.render(away, prm, w, h).cpu().numpy().any()
