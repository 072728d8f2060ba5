"""ivv_render_to_host: images written into pinned memory directly (4 MiB and
more) and by copy (smaller, pageable, not 16-byte aligned) equal the device
image, frame after frame into the same memory, for every integrator; nothing
outside the image is written, also when the call fails."""
import dataclasses

import numpy as np
import pytest

from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BIG, SMALL = (640, 411), (96, 61)          # 4.2 MB and 94 KB


def _memory(kind, w, h):
    n = w * h * 4
    if kind == "pageable":
        buf = np.full(n + 64, 7.0, np.float32)
        return buf, buf[32:32 + n].reshape(h, w, 4)
    buf = torch.full((n + 64,), 7.0).pin_memory()
    at = 33 if kind == "misaligned" else 32
    return buf, buf[at:at + n].view(h, w, 4)


@pytest.mark.parametrize("kind", ["pinned", "misaligned", "pageable"])
@pytest.mark.parametrize("size", [BIG, SMALL])
@pytest.mark.parametrize("over", [{}, {"rk_method": 2}, {"rk_method": 7, "c": 100.0},
                                  {"method": 1, "use_mlp_guess": 2, "rf_tol": 1e-3}, {"precision": 2, "ds": 0.5}])
def test_host_image_equals_device_image(kind, size, over):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    w, h = size
    sc = scenes.twisted_bar(width=w, height=h)
    prm = dataclasses.replace(sc.params, **over)
    vol = ivv.volume_for(sc)
    buf, out = _memory(kind, w, h)
    eye = np.array(sc.camera.eye)
    for f in (1.0, 1.6):                    # the second frame leaves other pixels empty
        cam = dataclasses.replace(sc.camera, eye=tuple(np.array(sc.camera.target) + f * (eye - sc.camera.target)))
        vol.render_to_host(cam, prm, w, h, out)
        dev = vol.render(cam, prm, w, h).cpu().numpy()
        assert np.array_equal(np.asarray(out), dev)
    edge = np.asarray(buf)
    n = w * h * 4
    assert (edge[:32] == 7.0).all() and (edge[33 + n:] == 7.0).all()
    with pytest.raises(ivv.IvvError):
        vol.render_to_host(cam, dataclasses.replace(prm, method=1, use_mlp_guess=1, precision=0, rk_method=0), w, h,
                           out)
