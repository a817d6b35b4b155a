"""Which realizes HP_OPT_CUDA_GRAPH replays and which it launches (GPU).  The
probe counts the kernels of a realize that launches them; a replay leaves it
at zero."""

import numpy as np
import pytest
import torch

import __graft_entry__
from gpu_util import bits, run, to_device
from paper_2012_07145_gb300 import hp, pipelines, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def one_kernel(name):
    """(pipeline of one kernel whose output has its input's shape and type, input for h, w)."""
    if name == "histeq":
        p = pipelines.histeq()
        return p, hp.HP_U8, lambda h, w: synth.gray_u8_lowcontrast(h, w, seed=h)
    p = pipelines.unsharp() if name == "unsharp" else pipelines.max_filter(3)
    return p, hp.HP_F32, lambda h, w: synth.rgb_f32(h, w, seed=w)


@pytest.mark.parametrize("name", ["unsharp", "maxfilter", "histeq"])
@pytest.mark.parametrize("h,w", [(16, 16), (96, 160), (480, 640), (1000, 1501)])
@pytest.mark.parametrize("overlap", [True, False])
def test_one_kernel(name, h, w, overlap):
    """Each option, realizes back to back on one stream where the output of one
    is the input of the next."""
    p, dt, gen = one_kernel(name)
    pipelines.fused_schedule(p, tile_w=0, tile_h=0)
    assert p.group_count() == 1
    info = p.group_info([(w, h)], 0)
    large = info.grid_x * info.grid_y * info.grid_z * info.threads >= 9728
    x = to_device(gen(h, w), dt)
    steps = [x]
    for _ in range(3):
        steps.append(run(p, [steps[-1]], [dt], x.shape, dt))
    p.overlap_launches(overlap)
    st = torch.cuda.current_stream().cuda_stream
    for option in (0, 1, 2):
        p.set_option(hp.HP_OPT_CUDA_GRAPH, option)
        ys = [x] + [hp.padded_empty(*x.shape, x.dtype).zero_() for _ in range(3)]
        bufs = [hp.buffer_from_tensor(y, dt) for y in ys]
        for rep in range(4):   # uncaptured, captured, replayed
            for y in ys[1:]:
                y.zero_()
            p.probe_kernel_attrs(True)
            for a, b in zip(bufs, bufs[1:]):
                p.realize([a], b, st)
            torch.cuda.synchronize()
            launched = p.kernel_attrs()[0] > 0
            p.probe_kernel_attrs(False)
            for got, want in zip(ys, steps):
                assert torch.equal(bits(got), bits(want)) and p.device_error() == 0
        assert launched == (option == 0 or (option == 1 and overlap and large)), option


def test_resident_chain_replayed():
    """Two launches of eight register-resident stages: captured, then replayed on a second stream."""
    h, w, n = 300, 515, 16
    x = to_device(synth.stencil_input(h, w, seed=3), hp.HP_F32)
    p = pipelines.stencil_chain(n, "alternate")
    want = run(p, [x], [hp.HP_F32], (1, h, w), hp.HP_F32)
    pipelines.chain_schedule(p, depth=8, tile_w=0, tile_h=0, threads=0, serial_y=0, impl=hp.HP_IMPL_RESIDENT)
    p.use_cuda_graph(True)
    y = hp.padded_empty(1, h, w, torch.float32)
    s = torch.cuda.Stream()
    launched = []
    for _ in range(4):
        y.zero_()
        torch.cuda.synchronize()
        p.probe_kernel_attrs(True)
        p.realize([hp.buffer_from_tensor(x, hp.HP_F32)], hp.buffer_from_tensor(y, hp.HP_F32), s.cuda_stream)
        torch.cuda.synchronize()
        launched.append(p.kernel_attrs()[0])
        p.probe_kernel_attrs(False)
        assert torch.equal(bits(y), bits(want)) and p.device_error() == 0
    assert launched[0] == 2 and launched[2:] == [0, 0]


@pytest.mark.parametrize("name", ["unsharp", "histeq"])
@pytest.mark.parametrize("h,w", [(48, 64), (480, 640)])
def test_server_slots_replay_prepared_shapes(name, h, w):
    """hp_server_prepare leaves the captured graph: every request of the shape is a replay."""
    p, dt, gen = one_kernel(name)
    pipelines.fused_schedule(p, tile_w=0, tile_h=0)
    arr = torch.from_numpy(np.ascontiguousarray(gen(h, w))).pin_memory()
    out = torch.zeros_like(arr).pin_memory()
    srv = hp.Server(hbm_budget_bytes=64 << 20, slots=1, max_batch=1)
    srv.prepare(p, [hp.buffer_from_tensor(arr, dt)])
    for _ in range(5):
        t = srv.submit(p, [hp.buffer_from_tensor(arr, dt)], hp.buffer_from_tensor(out, dt))
        assert srv.wait(t)[0] == hp.HP_OK
    stats = srv.stats()
    srv.close()
    assert stats.completed == 5 and stats.graph_replays == 5
