"""ivv_render_to_host leaves the caller's image as it was when the call is
refused, also where it writes pinned memory directly (4 MiB and more): bad
camera, bad parameters, a window outside the image, a missing guess network, no
memory for the sample buffer."""
import dataclasses

import numpy as np
import pytest

from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

W, H = 640, 411


@pytest.mark.parametrize("size", [(W, H), (96, 61)])
def test_refused_call_leaves_the_image(size):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    w, h = size
    sc = scenes.twisted_bar(width=w, height=h)
    vol = ivv.volume_for(sc)
    out = torch.full((h, w, 4), 7.0).pin_memory()
    bad = [(dataclasses.replace(sc.camera, target=sc.camera.eye), {}, None),
           (dataclasses.replace(sc.camera, eye=(float("nan"), 0.0, 0.0)), {}, None),
           (sc.camera, {"rk_tol": -1.0}, None),
           (sc.camera, {"supersample_k": 0}, None),
           (sc.camera, {}, (8, 0, w, h)),
           (sc.camera, {"method": 1, "use_mlp_guess": 1}, None),
           (sc.camera, {"precision": 2, "rk_method": 2}, None)]
    for cam, over, window in bad:
        with pytest.raises(ivv.IvvError):
            vol.render_to_host(cam, dataclasses.replace(sc.params, **over), w, h, out, window=window)
        torch.cuda.synchronize()
        assert (out.numpy() == 7.0).all(), (over, window)
    vol.render_to_host(sc.camera, sc.params, w, h, out)
    assert torch.equal(out, vol.render(sc.camera, sc.params, w, h).cpu())


@pytest.mark.parametrize("over", [{}, {"method": 1, "use_mlp_guess": 2}])
def test_no_memory_for_the_samples(over):
    """A frame of 170 M samples (2.7 GB; 0.7 GB of scalars) with 96 MB left, on
    a volume that has a workspace from the midpoint rule and no samples yet."""
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    w, h = 1920, 1080
    sc = scenes.twisted_bar(width=w, height=h)
    vol = ivv.volume_for(sc)
    out = torch.full((h, w, 4), 7.0).pin_memory()
    vol.render_to_host(sc.camera, dataclasses.replace(sc.params, rk_method=2), w, h, out)
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - (96 << 20), dtype=torch.uint8, device="cuda")
    try:
        out.fill_(7.0)
        with pytest.raises(ivv.IvvError, match="OOM"):
            vol.render_to_host(sc.camera, dataclasses.replace(sc.params, ds=sc.params.ds / 80, **over), w, h, out)
        torch.cuda.synchronize()
        assert (out.numpy() == 7.0).all()
    finally:
        del rest
        torch.cuda.empty_cache()
    vol.render_to_host(sc.camera, sc.params, w, h, out)
    assert np.isfinite(out.numpy()).all() and (out.numpy() != 7.0).all()
