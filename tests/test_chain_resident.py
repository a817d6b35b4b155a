"""The register-resident chain kernel (HP_IMPL_RESIDENT): its tiles cover every
pixel once (CPU), and its output is bit-identical to the generic interpreter run
stage by stage (GPU)."""

import pytest
import torch

import __graft_entry__
from paper_2012_07145_gb300 import hp, pipelines, synth

SIZES = [(1, 1), (3, 7), (17, 33), (65, 129), (77, 250), (130, 515), (300, 263), (431, 777)]
ST = {"f32": hp.HP_F32, "f16": hp.HP_F16, "bf16": hp.HP_BF16}


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def resident(n, depth, rows, threads, dtype="f32"):
    p = pipelines.stencil_chain(n, "alternate", storage=ST[dtype])
    pipelines.chain_schedule(p, depth=depth, tile_w=0, tile_h=0, threads=threads, serial_y=rows,
                             impl=hp.HP_IMPL_RESIDENT)
    return p


def is_resident(info):
    """The resident kernel's shared memory: two buffers of four 256-column f32 rows per warp."""
    return info.kernel == hp.HP_KERNEL_STENCIL_CHAIN and info.smem_bytes == info.threads // 32 * 8192


@pytest.mark.parametrize("h,w", SIZES + [(1536, 2560), (4097, 3001)])
@pytest.mark.parametrize("depth", [2, 3, 4, 8])
@pytest.mark.parametrize("rows,threads", [(20, 256), (11, 384), (5, 512), (9, 160)])
def test_tiles_cover_every_pixel_once(h, w, depth, rows, threads):
    """Along each axis the first tile stores from 0, an inner one its `step`
    pixels past the halo, the last one up to the image's end, and a tile holds
    2 depth pixels more on every side inside the image."""
    info = resident(depth, depth, rows, threads).group_info([(w, h)], 0)
    assert is_resident(info) and info.threads == threads
    full_y = rows * threads // 32
    hx, hy = (256 - info.tile_w) // 2, (full_y - info.tile_h) // 2
    if info.grid_x > 1 and info.grid_y > 1:
        assert hx == -(-2 * depth // 8) * 8 and hy == 2 * depth
    for n, grid, full, step, halo in ((w, info.grid_x, 256, info.tile_w, hx), (h, info.grid_y, full_y, info.tile_h, hy)):
        end = 0
        for t in range(grid):
            start = t * step
            lo = 0 if t == 0 else start + halo
            hi = n if t + 1 == grid else start + halo + step
            assert lo == end and lo < hi <= n
            assert start + full >= min(hi + halo, n)
            end = hi
        assert end == n


def test_shapes_out_of_range_are_refused_and_other_chains_keep_their_kernel():
    for rows, threads in ((7, 0), (20, 512), (5, 1024)):   # not a shape of the kernel
        with pytest.raises(hp.HPError):
            resident(8, 8, rows, threads).group_info([(640, 480)], 0)
    q = hp.Pipeline([hp.HP_F32], [1])   # stages of another type than the input's
    a = q.add_stage(hp.HP_STENCIL, [q.input(0)], 1, hp.HP_F16, rx=2, ry=2, wx=pipelines.BOX5, wy=pipelines.BOX5)
    q.set_output(q.add_stage(hp.HP_STENCIL, [a], 1, hp.HP_F16, rx=2, ry=2, wx=pipelines.BOX5, wy=pipelines.BOX5))
    q.schedule([0, 0], impl=[hp.HP_IMPL_RESIDENT])
    assert not is_resident(q.group_info([(64, 48)], 0))


def _base(n, h, w, dtype):
    from gpu_util import run, to_device
    img = synth.stencil_input(h, w, seed=h * 13 + w)
    p = pipelines.stencil_chain(n, "alternate", storage=ST[dtype])
    p.schedule(list(range(n)), impl=[hp.HP_IMPL_GENERIC] * n)
    x = to_device(img, ST[dtype])
    return x, run(p, [x], [ST[dtype]], img.shape, ST[dtype])


@pytest.mark.gpu
@pytest.mark.parametrize("h,w", SIZES)
@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
def test_bit_identical(h, w, dtype):
    """Every rows-per-thread instance, shapes given and chosen."""
    from gpu_util import bits, run
    n = 16
    x, base = _base(n, h, w, dtype)
    for depth, rows, threads in [(16, 0, 0), (8, 0, 0), (4, 5, 128), (6, 6, 256), (8, 8, 512), (4, 9, 192),
                                 (8, 11, 384), (2, 14, 64), (4, 17, 256), (8, 20, 256), (16, 20, 256), (4, 5, 160)]:
        p = resident(n, depth, rows, threads, dtype)
        assert is_resident(p.group_info([(w, h)], 0))
        n0 = hp.launch_count()
        y = run(p, [x], [ST[dtype]], (1, h, w), ST[dtype])
        assert hp.launch_count() - n0 == -(-n // depth)
        assert torch.equal(bits(y), bits(base)), (depth, rows, threads)


@pytest.mark.gpu
@pytest.mark.parametrize("h,w,planes", [(150, 400, 3), (1300, 1700, 3), (2000, 2100, 1)])
def test_planes_sixteen_stages_and_graph_replays(h, w, planes):
    """Planes of one image, 16 stages in one launch, several waves of tiles; as
    graph replays on a second stream."""
    from gpu_util import bits, run, to_device
    import numpy as np
    x = to_device(np.concatenate([synth.stencil_input(h, w, seed=k) for k in range(planes)]), hp.HP_F32)
    outs = []
    for impl in (hp.HP_IMPL_AUTO, hp.HP_IMPL_RESIDENT):
        p = hp.Pipeline([hp.HP_F32], [planes])
        prev = p.input(0)
        for k in range(16):
            t = pipelines.BOX5 if k % 2 else pipelines.BINOMIAL16
            prev = p.add_stage(hp.HP_STENCIL, [prev], planes, hp.HP_F32, rx=2, ry=2, wx=t, wy=t)
        p.set_output(prev)
        groups = list(range(16)) if impl == hp.HP_IMPL_AUTO else [0] * 16
        p.schedule(groups, impl=[impl] * (max(groups) + 1))
        outs.append(run(p, [x], [hp.HP_F32], (planes, h, w), hp.HP_F32))
    assert torch.equal(bits(outs[0]), bits(outs[1]))
    p.use_cuda_graph(True)
    y = hp.padded_empty(planes, h, w, torch.float32)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    for _ in range(3):
        y.zero_()
        torch.cuda.synchronize()
        p.realize([hp.buffer_from_tensor(x, hp.HP_F32)], hp.buffer_from_tensor(y, hp.HP_F32), s.cuda_stream)
        torch.cuda.synchronize()
        assert torch.equal(bits(y), bits(outs[0])) and p.device_error() == 0
