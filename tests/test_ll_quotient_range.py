"""The u16 remap's quotient over all it is used for: exact rationals at the ends
of its range (CPU), and the fused levels against the stage-per-kernel schedule
for bands and gray scales inside and just outside the range (GPU)."""

import random

import numpy as np
import pytest

import __graft_entry__
from paper_2012_07145_gb300 import hp, pipelines, synth
from test_ll_quotient import div_by, q, rnd


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def test_quotient_over_the_admitted_range():
    """sigma in [2^-20, 2^20]; |g - g_k| in (2^-34, 65), as gray scales up to 2^-10 give;
    mantissas at the ends of a binade, where a reciprocal is hardest to round."""
    rng = random.Random(7)
    ends = [1.0, 1 + 2.0 ** -23, 2 - 2.0 ** -23, 2 - 2.0 ** -22, 1.5, 4 / 3]
    sigmas = [m * 2.0 ** e for m in ends for e in (-20, -7, -3, 0, 5, 19)] + [2.0 ** 20]
    sigmas += [2.0 ** rng.uniform(-20, 20) for _ in range(12)]
    for s in sigmas:
        b = np.float32(s)
        rb = rnd(1 / q(b))
        for _ in range(60):
            a = np.float32(rng.choice([2.0 ** rng.uniform(-34, 6), 64 * rng.random(), rng.choice(ends) * 2.0 ** rng.randint(-33, 5),
                                       min(s, 64.0) * rng.random() + 2.0 ** -33]))
            assert div_by(a, b, rb) == rnd(q(a) / q(b)), (a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("sigma", [2.0 ** -21, 2.0 ** -20, 3e-4, 0.05, 0.142, 0.15, 1.7, 2.0 ** 20, 2.0 ** 21])
@pytest.mark.parametrize("scale", [1 / 65535, 2.0 ** -10, 2.0 ** -9, 2.0 ** -30, 2.0 ** -31])
@pytest.mark.parametrize("alpha", [0.25, 1.0])
def test_fused_levels_bit_identical(sigma, scale, alpha, monkeypatch):
    import torch
    from gpu_util import bits, run, to_device

    class Scaled(hp.Pipeline):
        def add_stage(self, kind, inputs, channels, storage=hp.HP_F32, op=0, params=None, **kw):
            if kind == hp.HP_POINTWISE and op == hp.HP_OP_GRAY:
                params = [scale]
            return super().add_stage(kind, inputs, channels, storage, op=op, params=params, **kw)

    monkeypatch.setattr(hp, "Pipeline", Scaled)
    h, w = 45, 130
    img = synth.rgb_u16_gradient_noise(h, w, seed=5)
    img[:, :2, :9] = 0                       # a gray of 0, the smallest ones, and the largest
    img[:, 2:4, :9] = np.arange(9, dtype=np.uint16)
    img[:, 4:6, :9] = 65535
    x = to_device(img, hp.HP_U16)
    p, ids = pipelines.local_laplacian(levels=3, k_levels=8, sigma_r=sigma, alpha=alpha, out_storage=hp.HP_F32)
    plain = run(p, [x], [hp.HP_U16], (3, h, w), hp.HP_F32)
    pipelines.local_laplacian_fused_schedule(p, ids)
    assert p.group_info([(w, h)], p.group_count() - 1).kernel == hp.HP_KERNEL_LL_LEVEL_ROWS
    assert torch.equal(bits(run(p, [x], [hp.HP_U16], (3, h, w), hp.HP_F32)), bits(plain))
