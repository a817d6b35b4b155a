"""The coarse end of a pyramid in one launch, on images far from square: the
values of the stage-per-kernel schedule, and no slower than a launch per level
would be."""

import pytest
import torch

import __graft_entry__
from gpu_util import bits, run, to_device
from paper_2012_07145_gb300 import hp, pipelines, synth
from test_direct_launch_speed import us_per_realize

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


NARROW = [(2048, 1), (1, 2048), (3000, 3), (3, 3000), (700, 5), (1024, 2), (2, 1025), (640, 9), (129, 31)]


@pytest.mark.parametrize("h,w", NARROW)
def test_interpolate_narrow(h, w):
    x = to_device(synth.rgba_sparse_f32(h, w, seed=h), hp.HP_F32)
    p, ids = pipelines.interpolate(10)
    plain = run(p, [x], [hp.HP_F32], (3, h, w), hp.HP_F32)
    pipelines.interpolate_fused_schedule(p, ids)
    assert torch.equal(bits(run(p, [x], [hp.HP_F32], (3, h, w), hp.HP_F32)), bits(plain))


@pytest.mark.parametrize("h,w", NARROW)
def test_local_laplacian_narrow(h, w):
    x = to_device(synth.rgb_u16_gradient_noise(h, w, seed=h + w), hp.HP_U16)
    p, ids = pipelines.local_laplacian(levels=8, k_levels=8, alpha=0.25, out_storage=hp.HP_F32)
    plain = run(p, [x], [hp.HP_U16], (3, h, w), hp.HP_F32)
    pipelines.local_laplacian_fused_schedule(p, ids)
    assert torch.equal(bits(run(p, [x], [hp.HP_U16], (3, h, w), hp.HP_F32)), bits(plain))


@pytest.mark.parametrize("w,h", [(16, 20000), (1, 30000), (64, 20000)])
def test_coarse_levels_cost_little_whatever_their_shape(w, h):
    """Five more levels, each of at most 1024 pixels, in one launch: less than
    the five finer ones take together (a launch per level and direction took
    0.41 to 0.54 of them; a warp per row took 1.5 to 4.2)."""
    us = []
    for levels in (5, 10):
        p, ids = pipelines.interpolate(levels)
        pipelines.interpolate_fused_schedule(p, ids)
        us.append(us_per_realize(p, 4, w, h, 3, n=50))
    assert us[1] <= 1.9 * us[0]
