"""Destinations that a kernel must not write directly: a buffer too small is
refused before anything is launched (as the copy or the memset of the same
range refuses it), and pinned host memory is filled."""
import numpy as np
import pytest
import torch

from paper_2303_11103_gb300 import rt
from paper_2303_11103_gb300 import scenes as S

from gpu_helpers import FC

pytestmark = pytest.mark.gpu

N_RX = 300_000   # offsets and H(f) of more bytes than a small tensor's segment (2 MB) has


@pytest.fixture(scope="module")
def los():
    tr = rt.Tracer(0, FC)
    tr.load_scene(S.tiny_scene())
    tr.set_tx(np.array([[-60.0, 0.0, 25.0]], np.float32), np.zeros((1, 3), np.float32), S.V_ISO)
    rx = np.random.default_rng(0).uniform(-95.0, 95.0, (N_RX, 3)).astype(np.float32)
    rx[:, 2] = 1.5
    tr.set_rx(rx, np.zeros_like(rx), S.V_ISO)
    tr.compute_paths(0, 0, reflection=False)
    yield tr
    tr.close()


def test_paths(los):
    want = los.paths()
    los.sync_stream()
    small = torch.empty(8, dtype=torch.int64, device="cuda")
    with pytest.raises(rt.RtError):
        rt.rt_get_paths(los.ctx, small)
    torch.cuda.synchronize()   # the context is as usable as before
    host = torch.full((N_RX + 1,), -1, dtype=torch.int64).pin_memory()
    assert rt.lib().rt_get_paths(los.ctx, host.data_ptr(), None, None, None, None) == rt.RT_OK
    torch.cuda.synchronize()
    assert torch.equal(host, want["offsets"].cpu())
    assert torch.equal(los.paths()["offsets"], want["offsets"])


def test_frequency_response(los):
    a, tau = los.cir_raw()
    off = los.paths()["offsets"]
    freqs = torch.arange(4, dtype=torch.float64, device="cuda") * 30e3
    want = torch.empty((N_RX, 1, 4, 2), device="cuda")
    los.sync_stream()
    rt.rt_freq_response_paths(los.ctx, off, 1, a, tau, freqs, want)
    small = torch.empty(8, device="cuda")
    with pytest.raises(rt.RtError):
        rt.rt_freq_response_paths(los.ctx, off, 1, a, tau, freqs, small)
    torch.cuda.synchronize()
    host = torch.full((N_RX, 1, 4, 2), -1.0).pin_memory()
    assert rt.lib().rt_freq_response_paths(los.ctx, off.data_ptr(), N_RX, 1, a.data_ptr(), tau.data_ptr(),
                                           freqs.data_ptr(), 4, host.data_ptr()) == rt.RT_OK
    torch.cuda.synchronize()
    assert torch.equal(host, want.cpu())
    # inside a graph capture the range is looked up too
    again = torch.zeros_like(want)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        los.sync_stream()
        rt.rt_freq_response_paths(los.ctx, off, 1, a, tau, freqs, again)
    g.replay()
    torch.cuda.synchronize()
    los.sync_stream()
    assert torch.equal(again, want)
