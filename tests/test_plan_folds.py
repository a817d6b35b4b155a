"""Plan-level choices between a producer and its consumers (GPU): the blurred
grid handed to slices in pair layout, and the premultiply recomputed in its
consumers, each against a schedule that does neither, bit for bit."""

import pytest
import torch

import __graft_entry__
from gpu_util import bits, run, to_device
from paper_2012_07145_gb300 import hp, pipelines, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


@pytest.mark.parametrize("h,w", [(1, 1), (5, 33), (64, 96), (131, 257), (200, 31)])
@pytest.mark.parametrize("s,r", [(1, 0.5), (4, 0.2), (8, 0.1), (12, 0.1), (16, 0.05), (3, 0.04)])
def test_grid_pairs(h, w, s, r):
    """Cells of powers of two and others, even and odd level counts, images of
    less than a block; a plan per size of one pipeline."""
    img = synth.gray_f32_gradient_noise(h, w, seed=h + w)
    img[0, ::3, ::5] = 1.0    # the last range level
    x = to_device(img, hp.HP_F32)
    p = pipelines.bilateral_grid(s, r)
    plain = run(p, [x], [hp.HP_F32], (1, h, w), hp.HP_F32)
    pipelines.bilateral_grid_fused_schedule(p)
    for _ in range(2):
        assert torch.equal(bits(run(p, [x], [hp.HP_F32], (1, h, w), hp.HP_F32)), bits(plain))


def test_grid_read_by_more_than_slices_stays_planar():
    """The blurred grid is the output itself: written in planes."""
    F = hp.HP_F32
    h, w, s, r, gz = 70, 90, 8, 0.1, 11
    x = to_device(synth.gray_f32_gradient_noise(h, w, seed=2), F)
    outs = []
    for fused in (False, True):
        p = hp.Pipeline([F], [1])
        g = p.add_stage(hp.HP_GRID_SPLAT, [p.input(0)], 2 * gz, F, params=[s, r])
        bz = p.add_stage(hp.HP_POINTWISE, [g], 2 * gz, F, op=hp.HP_OP_ZBLUR, params=[gz])
        bx = p.add_stage(hp.HP_STENCIL, [bz], 2 * gz, F, rx=2, ry=0, wx=pipelines.BINOMIAL16, wy=[1.0])
        p.set_output(p.add_stage(hp.HP_STENCIL, [bx], 2 * gz, F, rx=0, ry=2, wx=[1.0], wy=pipelines.BINOMIAL16))
        if fused:
            p.schedule([0, 1, 1, 1])
        outs.append(run(p, [x], [F], (2 * gz, 10, 13), F))
    assert torch.equal(bits(outs[0]), bits(outs[1]))


def saved_by_tail(h, w, levels):
    """A tail takes the levels l >= 1 of at most 1024 pixels, if three or more: a
    downsample and a step each but its finest, as one launch."""
    n = 0
    for l in range(1, levels):
        h, w = (h + 1) // 2, (w + 1) // 2
        n += h * w <= 1024
    return 2 * (n - 1) - 1 if n >= 3 else 0


@pytest.mark.parametrize("h,w,levels", [(1, 1, 5), (3, 2, 2), (37, 53, 4), (130, 258, 5), (257, 131, 7), (64, 64, 4),
                                        (66, 64, 4), (128, 128, 4), (5, 700, 9), (263, 255, 10)])
def test_premultiply_fold_and_interpolate_tail(h, w, levels):
    """The premultiply folded into the first downsample and the finest level, and
    the coarse levels in one launch, at the tail's largest level (32x32) and just
    past it; neither where the levels run on the generic kernel."""
    x = to_device(synth.rgba_sparse_f32(h, w, seed=h), hp.HP_F32)
    p, ids = pipelines.interpolate(levels)
    plain = run(p, [x], [hp.HP_F32], (3, h, w), hp.HP_F32)
    pipelines.interpolate_fused_schedule(p, ids)
    groups = p.group_count()
    for _ in range(2):
        n0 = hp.launch_count()
        y = run(p, [x], [hp.HP_F32], (3, h, w), hp.HP_F32)
        assert hp.launch_count() - n0 == groups - 1 - saved_by_tail(h, w, levels)
        assert torch.equal(bits(y), bits(plain))
    pipelines.interpolate_fused_schedule(p, ids, impl=hp.HP_IMPL_GENERIC)
    n0 = hp.launch_count()
    y = run(p, [x], [hp.HP_F32], (3, h, w), hp.HP_F32)
    assert hp.launch_count() - n0 == p.group_count()
    assert torch.equal(bits(y), bits(plain))


@pytest.mark.parametrize("h,w,levels", [(1, 1, 4), (32, 64, 4), (66, 130, 5), (128, 128, 5), (131, 127, 6), (9, 640, 7)])
@pytest.mark.parametrize("alpha", [1.0, 0.25])
def test_local_laplacian_tail(h, w, levels, alpha):
    x = to_device(synth.rgb_u16_gradient_noise(h, w, seed=h + w), hp.HP_U16)
    p, ids = pipelines.local_laplacian(levels=levels, k_levels=8, alpha=alpha, out_storage=hp.HP_F32)
    plain = run(p, [x], [hp.HP_U16], (3, h, w), hp.HP_F32)
    pipelines.local_laplacian_fused_schedule(p, ids)
    n0 = hp.launch_count()
    y = run(p, [x], [hp.HP_U16], (3, h, w), hp.HP_F32)
    assert hp.launch_count() - n0 == p.group_count() - saved_by_tail(h, w, levels)
    assert torch.equal(bits(y), bits(plain))


def test_levels_read_outside_the_tail_stay_launches():
    """A coarse level that another stage reads is written as before."""
    F = hp.HP_F32
    p = hp.Pipeline([F], [4])
    d = [p.add_stage(hp.HP_POINTWISE, [p.input(0)], 4, F, op=hp.HP_OP_SCALE, params=[1.0, 0.0])]
    for _ in range(4):
        d.append(p.add_stage(hp.HP_DOWNSAMPLE2, [d[-1]], 4, F))
    r = d[-1]
    for k in range(3, -1, -1):
        u = p.add_stage(hp.HP_UPSAMPLE2, [r, d[k]], 4, F)
        r = p.add_stage(hp.HP_POINTWISE, [d[k], u], 4, F, op=hp.HP_OP_OVER)
    z = d[3]   # the level above the coarsest, upsampled to the finest size as well
    for k in (2, 1, 0):
        z = p.add_stage(hp.HP_UPSAMPLE2, [z, d[k]], 4, F)
    p.set_output(p.add_stage(hp.HP_POINTWISE, [r, z], 4, F, op=hp.HP_OP_ADD))
    h, w = 61, 90
    x = to_device(synth.rgba_sparse_f32(h, w, seed=5), F)
    plain = run(p, [x], [F], (4, h, w), F)
    n = len(p.stages)
    groups, g = [0] * n, 0
    for i in range(n):
        pair = p.stages[i]["kind"] == hp.HP_POINTWISE and p.stages[i]["op"] == hp.HP_OP_OVER
        g += 0 if i == 0 or pair else 1
        groups[i] = g
    p.schedule(groups)
    assert torch.equal(bits(run(p, [x], [F], (4, h, w), F)), bits(plain))
