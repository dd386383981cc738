"""Traversal of a warp's rays as beams against the per-ray traversal: the same
hits, map counts and diffracted paths. The 8-wide layout always traverses ray
by ray; the binary layout takes beams from 40 rays per triangle on, so the same
scene on both gives both sides."""
import numpy as np
import pytest
import torch

from paper_2303_11103_gb300 import rt
from paper_2303_11103_gb300 import scenes as S

from gpu_helpers import FC

pytestmark = pytest.mark.gpu


def _soup(n, n_big, seed):
    """n triangles of every orientation (some on a plane, some degenerate) and n_big that span the scene."""
    rng = np.random.default_rng(seed)
    c = rng.uniform(-60.0, 60.0, (n, 1, 3)) * np.array([1.0, 1.0, 0.3])
    v = c + rng.normal(0.0, 1.0, (n, 3, 3)) * rng.uniform(0.2, 6.0, (n, 1, 1))
    v[::5, :, 2] = c[::5, :, 2]            # horizontal: boxes without height
    v[1::7, :, 0] = c[1::7, :, 0]          # vertical, on x = const
    v[3::11, 2] = v[3::11, 1]              # no area
    b = rng.uniform(-60.0, 60.0, (n_big, 3, 3)) * np.array([1.0, 1.0, 0.05])
    b[:, 0, 0], b[:, 1, 0] = -70.0, 70.0
    b[:, :, 2] -= 25.0
    v = np.concatenate([v, b]).reshape(n + n_big, 9).astype(np.float32)
    return S.Scene(v, np.zeros(n + n_big, np.int32), np.array([S.CONCRETE], np.float32))


def _city(n_side):
    return S.city_scene(n_side=n_side, size=25.0 * n_side, seed=4)


@pytest.mark.parametrize("scene,rays,n_tx", [
    (lambda: _soup(1, 0, 0), 100, 1),            # one leaf, warps of few rays
    (lambda: _soup(0, 3, 1), 5000, 2),           # large triangles alone
    (lambda: _soup(31, 1, 2), 4000, 1),          # less than one group
    (lambda: _soup(33, 40, 3), 20000, 3),        # one leaf in the second group, two rounds of large ones
    (lambda: _soup(1025, 2, 4), 60000, 1),       # one leaf in the second set
    (lambda: _soup(3000, 0, 5), 121000, 2),
    (lambda: _city(6), 40000, 2)])
@pytest.mark.parametrize("builder", [rt.BVH_PLOC, rt.BVH_KARRAS])
def test_beams_find_the_rays_hits(scene, rays, n_tx, builder):
    sc = scene()
    assert rays >= 40 * sc.n_tris
    pos = np.array([[1.0, 2.0, 30.0], [-30.0, 15.0, 12.0], [40.0, -20.0, 45.0]], np.float32)[:n_tx]
    ypr = np.array([[0.3, 0.1, 0.0]] * n_tx, np.float32)
    grid = dict(x0=-60.0, y0=-60.0, cell=3.0, nx=40, ny=40, h=1.5)
    out = []
    for width in (2, 8):
        tr = rt.Tracer(0, FC)
        try:
            tr.set_bvh_builder(builder)
            tr.set_bvh_width(width)
            tr.load_scene(sc)
            tr.set_tx(pos, ypr, S.TR38901_V)
            tr.set_rx(np.array([[10.0, 5.0, 1.5]], np.float32), np.zeros((1, 3), np.float32), S.V_ISO)
            tr.compute_paths(3, rays, record_rays=True)
            hits = tr.ray_hits().cpu().numpy()
            gain, count = (t.cpu().numpy() for t in tr.coverage_map(grid, 3, rays))
            up = np.ones_like(gain)
            out.append((hits, gain, count, tr.coverage_map_backward(grid, 3, rays, up).cpu().numpy()))
        finally:
            tr.close()
    a, b = out
    assert np.array_equal(a[0], b[0])
    assert np.array_equal(a[2], b[2])
    # sums of the same terms in another order
    assert np.allclose(a[1], b[1], rtol=1e-4, atol=1e-6 * max(b[1].max(), 1e-30))
    assert np.allclose(a[3], b[3], rtol=1e-3, atol=1e-4 * max(np.abs(b[3]).max(), 1e-30))


@pytest.mark.parametrize("nx,ny", [(1, 1), (8, 4), (9, 33), (61, 50)])
def test_segment_beams_find_the_same_paths(nx, ny):
    """The diffracted map and paths of a city, binary (beams) against 8-wide
    (segment by segment): maps at the edges of the tiles, receivers in no order."""
    sc = _city(5)
    rng = np.random.default_rng(nx)
    rx = np.concatenate([rng.uniform(-60.0, 60.0, (70, 2)), np.full((70, 1), 1.5)], 1).astype(np.float32)
    grid = dict(x0=-62.5, y0=-62.5, cell=125.0 / max(nx, ny), nx=nx, ny=ny, h=1.5)
    out = []
    for width in (2, 8):
        tr = rt.Tracer(0, FC)
        try:
            tr.set_bvh_width(width)
            tr.load_scene(sc)
            tr.set_tx(np.array([[3.0, -4.0, 40.0], [-20.0, 30.0, 8.0]], np.float32), np.zeros((2, 3), np.float32), S.V_ISO)
            tr.set_rx(rx, np.zeros((70, 3), np.float32), S.V_ISO)
            tr.compute_diffraction()
            out.append((tr.diffraction(), tr.coverage_map_diffraction(grid).cpu().numpy()))
        finally:
            tr.close()
    (pa, ga), (pb, gb) = out
    for k in ("offsets", "wedge"):
        assert np.array_equal(pa[k].cpu().numpy(), pb[k].cpu().numpy()), k
    assert len(pa["wedge"]) > 0
    assert np.array_equal(ga != 0, gb != 0)
    assert np.allclose(ga, gb, rtol=1e-4, atol=1e-6 * max(gb.max(), 1e-30))


@pytest.mark.parametrize("n_rx,sets", [(2000, False), (1999, True)])
def test_handed_out_validation_units(n_rx, sets):
    """Enough candidates and receivers that the validation hands its units out in
    runs (the binary layout), against units dealt one by one (8-wide): the same
    paths, also with uneven receiver sets (one empty, ragged last units)."""
    sc = _city(8)
    rng = np.random.default_rng(n_rx)
    n_tx = 8
    pos = np.concatenate([rng.uniform(-80.0, 80.0, (n_tx, 2)), rng.uniform(30.0, 60.0, (n_tx, 1))], 1).astype(np.float32)
    cut = np.array([0, 3000, 3000, 5001, 9000, 9001, 12000, 14000, 15990]) if sets else None
    n = int(cut[-1]) if sets else n_rx
    rx = np.concatenate([rng.uniform(-95.0, 95.0, (n, 2)), np.full((n, 1), 1.5)], 1).astype(np.float32)
    out = []
    for width in (2, 8):
        tr = rt.Tracer(0, FC)
        try:
            tr.set_bvh_width(width)
            tr.load_scene(sc)
            tr.set_tx(pos, np.zeros((n_tx, 3), np.float32), S.V_ISO)
            tr.set_rx(rx, np.zeros((n, 3), np.float32), S.V_ISO, None if cut is None else [int(v) for v in cut])
            tr.compute_paths(3, 200000)
            out.append({k: v.cpu().numpy() for k, v in tr.paths().items()})
            units = len(tr.candidates()[0]) * ((n if not sets else n // n_tx) + 31) // 32
        finally:
            tr.close()
    assert units >= 64 * 8 * 608   # what the rule asks for at 4 blocks on 152 SMs
    a, b = out
    assert len(a["depth"]) > 1000
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("n", [1, 2, 3000])
def test_width_changed_without_a_load(n):
    """A scene loaded for the 8-wide layout has no boxes for beams: set to the
    binary layout it is traversed ray by ray, with the same hits, map counts and
    diffracted paths (one triangle: no wide nodes either, so it has the boxes)."""
    sc = _soup(n, 1, 6) if n < 100 else _city(6)
    rays = 40 * sc.n_tris + 100
    grid = dict(x0=-60.0, y0=-60.0, cell=6.0, nx=20, ny=20, h=1.5)
    out = []
    for first in (2, 8):
        tr = rt.Tracer(0, FC)
        try:
            tr.set_bvh_width(first)
            tr.load_scene(sc)
            tr.set_bvh_width(2)
            tr.set_tx(np.array([[3.0, -4.0, 40.0]], np.float32), np.zeros((1, 3), np.float32), S.V_ISO)
            tr.set_rx(np.array([[10.0, 5.0, 1.5]] * 40, np.float32), np.zeros((40, 3), np.float32), S.V_ISO)
            tr.compute_paths(2, rays, record_rays=True)
            hits = tr.ray_hits().cpu().numpy()
            count = tr.coverage_map(grid, 2, rays)[1].cpu().numpy()
            tr.compute_diffraction()
            out.append((hits, count, tr.diffraction()["wedge"].cpu().numpy()))
        finally:
            tr.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("sets", [False, True])
def test_validation_units_on_one_layout(sets):
    """The binary layout against itself: the hash leaves the host the number of
    candidates, so that the validation hands out its units, the sort does not,
    so that they are dealt. The kernels that ran are read from a trace."""
    sc = _city(8)
    rng = np.random.default_rng(3)
    n_tx, n_rx = 8, 2000
    pos = np.concatenate([rng.uniform(-80.0, 80.0, (n_tx, 2)), rng.uniform(30.0, 60.0, (n_tx, 1))], 1).astype(np.float32)
    cut = [0, 3000, 3000, 5001, 9000, 9001, 12000, 14000, 15990] if sets else None
    n = cut[-1] if sets else n_rx
    rx = np.concatenate([rng.uniform(-95.0, 95.0, (n, 2)), np.full((n, 1), 1.5)], 1).astype(np.float32)
    out, ran = [], []

    def trace():
        return torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA])

    with trace():   # the process's first trace may come back empty
        torch.zeros(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    for mode in (rt.DEDUP_HASH, rt.DEDUP_SORT):
        tr = rt.Tracer(0, FC)
        try:
            tr.set_dedup(mode)
            tr.load_scene(sc)
            tr.set_tx(pos, np.zeros((n_tx, 3), np.float32), S.V_ISO)
            tr.set_rx(rx, np.zeros((n, 3), np.float32), S.V_ISO, cut)
            with trace() as prof:
                tr.compute_paths(3, 200000)
                torch.cuda.synchronize()
            ran.append({e.name for e in prof.events() if "k_validate" in e.name})
            out.append({k: v.cpu().numpy() for k, v in tr.paths().items()})
            per_candidate = ((n if sets else n_tx * n_rx) // n_tx + 31) // 32
            units = len(tr.candidates()[0]) * per_candidate
        finally:
            tr.close()
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert units >= 64 * 8 * 4 * sms   # the rule, at 4 blocks of 8 warps on an SM
    a, b = out
    assert len(a["depth"]) > 1000
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    if not any(ran):
        pytest.skip("the profiler recorded no kernels: the paths agree, which kernel gave them is not shown")
    handed = ["true>" in names.pop() for names in ran if len(names) == 1]   # k_validate's last parameter
    assert handed == [True, False], ran
