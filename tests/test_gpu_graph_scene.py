"""Replays of a captured coverage map after another scene was loaded into the
same buffers: refused unless the counts its kernels hold are the same."""
import numpy as np
import pytest
import torch

from paper_2303_11103_gb300 import rt
from paper_2303_11103_gb300 import scenes as S

from gpu_helpers import FC

pytestmark = pytest.mark.gpu

RAYS = 20000   # beams: 46 rays a triangle


def _load(tr, n_side, width=2, seed=4):
    tr.set_bvh_width(width)
    tr.load_scene(S.city_scene(n_side=n_side, size=150.0, seed=seed))


def test_a_replay_needs_the_scene_it_was_captured_with():
    tr = rt.Tracer(0, FC)
    try:
        _load(tr, 6, 8)   # the buffers of both layouts are there
        _load(tr, 6)
        tr.set_tx(np.array([[1.0, 2.0, 70.0]], np.float32), np.zeros((1, 3), np.float32), S.V_ISO)
        tr.set_rx(np.zeros((1, 3), np.float32), np.zeros((1, 3), np.float32), S.V_ISO)
        grid = rt.rt_grid(-75.0, -75.0, 3.0, 1.5, 50, 50)
        gain = torch.zeros((1, 50, 50), device="cuda")
        hits = torch.zeros((1, 50, 50), dtype=torch.int32, device="cuda")
        tr.sync_stream()
        rt.rt_coverage_map(tr.ctx, grid, 2, RAYS, 0, gain, hits)
        torch.cuda.synchronize()
        want = hits.clone()
        rt.rt_graph_begin(tr.ctx)
        rt.rt_coverage_map(tr.ctx, grid, 2, RAYS, 0, gain, hits)
        rt.rt_graph_end(tr.ctx)
        for n_side, width in ((3, 2), (6, 8)):   # fewer triangles; the same ones without boxes for beams
            _load(tr, n_side, width)
            tr.sync_stream()
            with pytest.raises(rt.RtError) as e:
                rt.rt_graph_launch(tr.ctx)
            assert e.value.code == -6 and "capture the graph again" in str(e.value)
        _load(tr, 6)
        tr.sync_stream()
        hits.zero_()
        rt.rt_graph_launch(tr.ctx)
        torch.cuda.synchronize()
        assert torch.equal(hits, want)
    finally:
        tr.close()
