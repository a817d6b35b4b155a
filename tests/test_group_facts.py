"""hp_group_info_get against what a realize launches: groups folded into others
have no launch (grid_z = 0), a pyramid's coarse end is one CTA."""

import pytest

import __graft_entry__
from paper_2012_07145_gb300 import hp, pipelines, synth


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def facts(p, w, h):
    return [p.group_info([(w, h)], g) for g in range(p.group_count())]


def launched(infos):
    return [i for i in infos if i.grid_z > 0]


def tails(infos):
    return [i for i in launched(infos)
            if i.kernel in (hp.HP_KERNEL_INTERP_ROWS, hp.HP_KERNEL_LL_LEVEL_ROWS) and i.threads == 1024]


CASES = [("interpolate", 2560, 1536, 10, (40, 24)), ("interpolate", 64, 64, 5, (32, 32)),
         ("interpolate", 64, 64, 3, None), ("interpolate", 2559, 1535, 5, None),
         ("laplacian", 160, 96, 5, (40, 24)), ("laplacian", 2560, 1536, 8, None)]


def build(app, levels, impl=None):
    if app == "interpolate":
        p, ids = pipelines.interpolate(levels)
        pipelines.interpolate_fused_schedule(p, ids, impl=impl)
    else:
        p, ids = pipelines.local_laplacian(levels=levels, k_levels=8)
        pipelines.local_laplacian_fused_schedule(p, ids, impl=impl)
    return p


@pytest.mark.parametrize("app,w,h,levels,finest", CASES)
def test_facts_of_folded_groups(app, w, h, levels, finest):
    """Level sizes by hand: a tail takes levels 1 and up of at most 1024 pixels, if
    three or more."""
    sizes = [(w, h)]
    for _ in range(1, levels):
        sizes.append(((sizes[-1][0] + 1) // 2, (sizes[-1][1] + 1) // 2))
    inside = [s for s in sizes[1:] if s[0] * s[1] <= 1024]
    p = build(app, levels)
    infos = facts(p, w, h)
    assert all(i.grid_x > 0 and i.grid_y > 0 and i.grid_z >= 0 and i.threads >= 32 for i in infos)
    premul = 1 if app == "interpolate" else 0
    saved = 2 * (len(inside) - 1) - 1 if len(inside) >= 3 else 0
    assert len(launched(infos)) == p.group_count() - premul - saved
    t = tails(infos)
    if finest is None:
        assert not t
    else:
        assert len(t) == 1 and (t[0].tile_w, t[0].tile_h) == finest == inside[0]
        assert (t[0].grid_x, t[0].grid_y, t[0].grid_z) == (1, 1, 1)
        channels = 4 if app == "interpolate" else 9
        assert t[0].smem_bytes >= 4 * channels * sum(a * b for a, b in inside)
    generic = facts(build(app, levels, hp.HP_IMPL_GENERIC), w, h)
    assert len(launched(generic)) == len(generic)


@pytest.mark.gpu
@pytest.mark.parametrize("app,w,h,levels,finest", CASES)
def test_launches_are_the_groups_with_a_grid(app, w, h, levels, finest):
    from gpu_util import run, to_device
    p = build(app, levels)
    if app == "interpolate":
        x, dt, odt = synth.rgba_sparse_f32(h, w, seed=1), hp.HP_F32, hp.HP_F32
    else:
        x, dt, odt = synth.rgb_u16_gradient_noise(h, w, seed=1), hp.HP_U16, hp.HP_U16
    n0 = hp.launch_count()
    run(p, [to_device(x, dt)], [dt], (3, h, w), odt)
    assert hp.launch_count() - n0 == len(launched(facts(p, w, h)))
