"""Rows per run that the streaming max filter takes when the schedule gives none."""

import pytest

import __graft_entry__
from paper_2012_07145_gb300 import hp, pipelines


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


@pytest.mark.parametrize("radius", [1, 2, 3, 4])
@pytest.mark.parametrize("storage,boxed", [(hp.HP_F32, True), (hp.HP_BF16, True), (hp.HP_F16, False), (hp.HP_U8, False),
                                           (hp.HP_U16, False)])
def test_max_filter_run_length(radius, storage, boxed):
    """Inputs that arrive in boxes of 4 rows: a run's input rows are whole boxes.
    The others load row by row: small images take the shortest run, 8 rows."""
    p = pipelines.max_filter(radius, storage=storage, io_storage=storage)
    p.schedule([0, 0])
    for w, h in ((256, 256), (640, 480), (1920, 1080), (64, 20000)):
        rows = p.group_info([(w, h)], 0).tile_h
        assert rows >= 8
        if boxed:
            assert (rows + 2 * radius) % 4 == 0
        elif (w, h) == (256, 256):
            assert rows == 8
