"""Batch tiles without candidates (finished by the cull, skipped by the pairing)
against fresh batches of the same cameras: images whose 16 x 16 tiles are
partly outside the image or hold one pixel, for every warp tile shape, with a
poisoned output before each render and cameras that move the object into and
out of the tiles.  The same kernels on the same requests: equal bits."""
import dataclasses

import pytest

from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 4), (4, 8), (16, 2)])
def test_empty_tiles_follow_the_cameras(shape):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    vols, reqs = scenes.batch_requests()
    gpu = [ivv.volume_for(v) for v in vols]
    sizes = [(1, 1), (15, 17), (16, 16), (65, 31), (130, 70)]
    q = [reqs[i] for i in range(len(sizes))]

    def shifted(c, f):
        # the target off by f times the eye distance: f = 0.2 a part of the
        # object in other tiles, f = 3 nothing in view
        return dataclasses.replace(c, target=tuple(t + f * (e - t0) for t, e, t0 in
                                                   zip(c.target, c.eye[1:] + c.eye[:1], c.target[1:] + c.target[:1])))

    def batch(f):
        b = ivv.Batch([(gpu[r.volume], shifted(r.camera, f), w, h, r.tf) for r, (w, h) in zip(q, sizes)])
        b.tuning = dict(b.tuning, tile_w=shape[0], tile_h=shape[1])
        return b

    moved = batch(0.0)
    lit = []
    for f in (0.0, 0.2, 3.0, 0.0):
        for i, r in enumerate(q):
            moved.set_camera(i, shifted(r.camera, f))
        for o in moved.outputs:
            o.fill_(7.0)
        got = [o.clone() for o in moved.render()]
        want = batch(f).render()
        torch.cuda.synchronize()
        for x, y in zip(got, want):
            assert torch.equal(x, y), (shape, f)
        lit.append(int((got[-1][..., 3] > 0).sum()))
    assert lit[0] > 100 and lit[3] == lit[0]
    assert lit[2] == 0
