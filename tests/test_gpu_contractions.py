"""FP32 evaluation on the device (geometry-only control points, scalar apart)
against the library's FP64 host evaluation, at the places where its element
lookup and its packed layouts can go wrong: knots, corners, faces and the
middle of elements, for cubic and quadratic volumes."""
import numpy as np
import pytest

from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


@pytest.mark.parametrize("name", ["twisted_cube", "twisted_bar", "bent_beam", "backstep"])
def test_eval_at_element_edges(name):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    sc = getattr(scenes, name)(width=8, height=8)
    vol = ivv.volume_for(sc)
    blk = len(sc.blocks) - 1
    b = sc.blocks[blk]
    axes = []
    for d in range(3):
        brk = np.unique(b.knots[d])
        axes.append(np.unique(np.concatenate([brk, 0.5 * (brk[1:] + brk[:-1])]).astype(np.float32))[:9])
    P = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)
    P = np.concatenate([P, np.random.default_rng(3).uniform(0, 1, (257, 3)).astype(np.float32)])
    phi, J, rho = (x.cpu().numpy().astype(np.float64) for x in vol.eval_points(blk, torch.from_numpy(P).cuda()))
    f, Jr, r = ivv.host_eval(sc.blocks, sc.scalar_mode, blk, P.astype(np.float64))
    # a point: three nested convex sums of up to four terms (12 roundings, and
    # those of the basis) over control points relative to the element, its
    # origin added; a partial: the same over differences of control points
    # times the degree and the element count, whose parameter is rounded too
    nseg = max(len(np.unique(k)) - 1 for k in b.knots)
    ext = max(np.ptp(b.geom_cp.reshape(-1, 3), axis=0))
    assert np.abs(phi - f).max() <= 32 * EPS * (np.abs(f).max() + ext)
    assert np.abs(J - Jr).max() <= 64 * EPS * nseg * 3 * ext
    # det / |J|_F has the relative error of J; control-point scalars the
    # rounding of their sum and of the parameter (slope: degree x elements x range)
    scale = np.abs(r).max()
    if sc.scalar_mode == scenes.SCALAR_CP:
        bound = 64 * EPS * (scale + 3 * nseg * np.ptp(b.scalar_cp))
    else:
        bound = 64 * EPS * 3 * nseg * 3 * scale * ext
    assert np.abs(rho - r).max() <= bound
