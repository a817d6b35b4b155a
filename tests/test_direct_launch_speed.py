"""Calls whose time depends on how kernels follow one another, or on the shape
of an image, against a neighbouring call of the same work on the same GPU."""

import pytest
import torch

import __graft_entry__
from paper_2012_07145_gb300 import hp, pipelines

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def us_per_realize(p, channels, w, h, out_channels, n=200):
    """Least mean over bursts of back-to-back realizes, device time."""
    x = hp.padded_copy(torch.rand((channels, h, w), device="cuda"))
    y = hp.padded_empty(out_channels, h, w, torch.float32)
    bi, bo = [hp.buffer_from_tensor(x, hp.HP_F32)], hp.buffer_from_tensor(y, hp.HP_F32)
    s = torch.cuda.current_stream().cuda_stream
    best = float("inf")
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(n):
            p.realize(bi, bo, s)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


@pytest.mark.parametrize("w,h", [(500, 375), (640, 480), (1000, 700)])
def test_bilateral_realizes_without_a_graph_overlap(w, h):
    """Three launches a realize: launched one after another they take no longer
    than the same realizes as graph replays."""
    us = []
    for graph in (False, True):
        p = pipelines.bilateral_grid(8, 0.1)
        pipelines.bilateral_grid_fused_schedule(p)
        p.use_cuda_graph(graph)
        us.append(us_per_realize(p, 1, w, h, 1))
    assert us[0] <= 1.05 * us[1]
