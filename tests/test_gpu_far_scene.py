"""Scenes far from the coordinate origin: the rounding of box tests grows with
the coordinates, not with the scene, and no box may lose a hit that the
triangle test accepts. The binary layout (beams) against the 8-wide one (ray by
ray), and rays down to the ground, which cannot miss it."""
import numpy as np
import pytest

from paper_2303_11103_gb300 import rt
from paper_2303_11103_gb300 import scenes as S

from gpu_helpers import FC

pytestmark = pytest.mark.gpu

SIZE, RAYS = 150.0, 60000


def _city(offset):
    sc = S.city_scene(n_side=6, size=SIZE, seed=4)
    v = sc.verts.reshape(-1, 3) + np.array([offset, -offset, 0.0], np.float32)
    return S.Scene(v.reshape(-1, 9).astype(np.float32), sc.mat_id, sc.materials)


def _both(offset, calls):
    out = []
    for width in (2, 8):
        tr = rt.Tracer(0, FC)
        try:
            tr.set_bvh_width(width)
            tr.load_scene(_city(offset))
            pos = np.array([[offset + 1.0, -offset + 2.0, 70.0], [offset - 30.0, -offset + 20.0, 65.0]], np.float32)
            tr.set_tx(pos, np.zeros((2, 3), np.float32), S.V_ISO)
            tr.set_rx(np.array([[offset, -offset, 1.5]], np.float32), np.zeros((1, 3), np.float32), S.V_ISO)
            out.append(calls(tr, pos))
        finally:
            tr.close()
    return out


@pytest.mark.parametrize("offset", [0.0, 5e3, 5e4, 4e5])
def test_the_same_hits(offset):
    def calls(tr, pos):
        assert RAYS >= 40 * (12 * 36 + 2)   # beams
        tr.compute_paths(2, RAYS, record_rays=True)
        return tr.ray_hits().cpu().numpy(), tr.ray_directions(RAYS).cpu().numpy().astype(np.float64), pos

    (a, d, pos), (b, _, _) = _both(offset, calls)
    assert np.array_equal(a, b)
    for k in range(2):
        o = pos[k].astype(np.float64) - [offset, -offset, 0.0]
        with np.errstate(divide="ignore"):
            g = o[:2] + d[:, :2] * (-o[2] / d[:, 2])[:, None]
        down = (d[:, 2] < -0.1) & (np.abs(g) < 0.45 * SIZE).all(1)
        assert down.sum() > 1000
        assert (a[k, down, 0] >= 0).all() and (b[k, down, 0] >= 0).all()


@pytest.mark.parametrize("offset", [0.0, 5e3, 5e4])
def test_the_same_diffracted_map(offset):
    grid = dict(x0=offset - 75.0, y0=-offset - 75.0, cell=1.5, nx=100, ny=100, h=1.5)
    a, b = _both(offset, lambda tr, pos: tr.coverage_map_diffraction(grid).cpu().numpy())
    assert (a > 0).any()
    assert np.array_equal(a != 0, b != 0)
    assert np.allclose(a, b, rtol=1e-4, atol=1e-6 * b.max())
