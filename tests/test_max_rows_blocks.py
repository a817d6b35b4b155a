"""The max filter's 4-row x 4-column block form: its selection of prefixes and
suffixes replayed on the CPU, and the kernel on special values, odd strips and
single rows (GPU) against the oracle."""

import numpy as np
import pytest
import torch

import __graft_entry__
from oracle import maxfilter as om
from paper_2012_07145_gb300 import hp


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


@pytest.mark.parametrize("radius", [0, 1, 2, 3, 4])
def test_vertical_blocks_replayed(radius):
    """Row by row as the kernel does it: the maximum of the block's rows so far
    and of the two earlier blocks' suffixes is the maximum of the last
    2 radius + 1 rows (NaN before the first)."""
    rows = np.random.default_rng(radius).random(40)
    X, Y = [np.nan] * 4, [np.nan] * 4
    for i in range(10):
        pre = np.nan
        for j in range(4):
            h = rows[4 * i + j]
            pre = np.fmax(pre, h)
            n, m = 2 * radius - j, pre
            if n >= 4:
                m = np.fmax(m, Y[0])
            if 0 < n < 4:
                m = np.fmax(m, Y[4 - n])
            if n > 4:
                m = np.fmax(m, X[8 - n])
            if n < 0:
                m = h
                for t in range(1, 2 * radius + 1):
                    m = np.fmax(m, X[j - t])
            X[j] = h
            t = 4 * i + j
            assert m == rows[max(0, t - 2 * radius):t + 1].max()
        for j in (2, 1, 0):
            X[j] = np.fmax(X[j], X[j + 1])
        X, Y = Y, X


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("h,w", [(1, 1), (3, 119), (9, 121), (40, 241), (33, 363), (70, 480)])
@pytest.mark.parametrize("radius,shape", [(1, "square"), (2, "vertical"), (3, "square"), (4, "square"), (4, "horizontal"),
                                          (1, "vertical"), (3, "horizontal")])
def test_special_values_and_strip_edges(dtype, h, w, radius, shape):
    """Strips of 120 columns cut at every edge; infinities, the type's
    lowest value and NaN (ignored next to a number)."""
    from gpu_util import run, to_device, to_numpy
    rng = np.random.default_rng(h * 1000 + w + radius)
    img = torch.from_numpy(rng.standard_normal((2, h, w)).astype(np.float32))
    st = hp.HP_F32 if dtype == "f32" else hp.HP_BF16
    if dtype == "bf16":
        img = img.to(torch.bfloat16).float()
    img = img.numpy()
    pick = rng.random(img.shape)
    low = float(torch.finfo(torch.float32 if dtype == "f32" else torch.bfloat16).min)
    img[pick < 0.05] = -np.inf
    img[(pick >= 0.05) & (pick < 0.1)] = np.nan
    img[(pick >= 0.1) & (pick < 0.5)] = low
    img[(pick >= 0.5) & (pick < 0.502)] = np.inf
    rx, ry = (radius if shape != "vertical" else 0), (radius if shape != "horizontal" else 0)
    p = hp.Pipeline([st], [2])
    p.set_output(p.add_stage(hp.HP_MAX_STENCIL, [p.input(0)], 2, st, rx=rx, ry=ry))
    padded = np.pad(img, ((0, 0), (ry, ry), (rx, rx)), mode="edge")
    ref = np.full_like(img, np.nan)
    for dy in range(2 * ry + 1):
        for dx in range(2 * rx + 1):
            ref = np.fmax(ref, padded[:, dy:dy + h, dx:dx + w])
    assert np.array_equal(om.max_filter(np.zeros((h, w)), rx, ry), np.zeros((h, w)))
    for rows in (0, 5):
        p.schedule([0], tile_h=[rows] if rows else None)
        assert p.group_info([(w, h)], 0).kernel == hp.HP_KERNEL_MAX_ROWS
        got = to_numpy(run(p, [to_device(img, st)], [st], (2, h, w), st))
        assert p.device_error() == 0
        assert np.array_equal(got, ref, equal_nan=True)
