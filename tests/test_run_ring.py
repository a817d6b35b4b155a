"""CPU replay of the TMA ring of a run, as the streaming stencil, max filter,
interpolate level and Harris kernels keep it: one run of rows per warp, a ring
started with the run, every lane testing the box's barrier.

Box i of a run goes to slot i % kRing.  The wait names the parity of the slot's
i // kRing-th phase, kept as a running (slot, phase) pair; box i + kRing is issued
into the slot once box i has been read.  A slot's barrier is modelled by the
phases it has completed.  Beside that, the shared memory that lanes read past
their slot, against the size the library reports for the launch.  Nothing here
touches a GPU; the older replay of rings that run on across units describes the
streaming chain kernel's discipline only."""

import itertools

import pytest

import __graft_entry__
from paper_2012_07145_gb300 import hp, pipelines


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


class Slots:
    def __init__(self, kring):
        self.kring = kring
        self.box = [None] * kring      # the box in the slot
        self.read = [True] * kring
        self.phases = [0] * kring      # phases the slot's barrier has been armed for

    def issue(self, i, slot):
        assert slot == i % self.kring and self.read[slot], ("slot refilled before it was read", i)
        self.box[slot], self.read[slot] = i, False
        self.phases[slot] += 1

    def wait(self, i, slot, parity):
        assert self.box[slot] == i, ("waits for a box that is not in the slot", i, self.box[slot])
        # the phase waited for is the slot's last armed one: an older parity would
        # fall through, a newer one never completes
        assert parity == (self.phases[slot] - 1) & 1, ("parity", i)
        self.read[slot] = True


def replay(nbox, kring, refill=True, flip=True):
    """nbox boxes, as block() / step() of the kernels: the pair (s, phase) runs on."""
    S = Slots(kring)
    for i in range(min(kring, nbox)):
        S.issue(i, i)
    s = phase = 0
    for i in range(nbox):
        S.wait(i, s, phase)
        if i + kring < nbox and refill:
            S.issue(i + kring, s)
        if flip:
            phase ^= s == kring - 1
        s = 0 if s == kring - 1 else s + 1
    assert all(S.read) and sum(S.phases) == nbox, "a box in flight when the warp ends"


@pytest.mark.parametrize("kring", [3, 4])
@pytest.mark.parametrize("nbox", list(range(1, 14)) + [97, 385])
def test_run_ring(nbox, kring):
    replay(nbox, kring)


def test_mistakes_in_the_discipline_are_caught():
    for wrong in (dict(refill=False), dict(flip=False)):
        with pytest.raises(AssertionError):
            replay(8, 3, **wrong)


def test_harris_run():
    """k_harris_rows: boxes of 2 rows, slot and parity from the box number, steps
    below the image without a box."""
    for H, rows in itertools.product((1, 2, 5, 9, 37, 480), (1, 2, 4, 5, 14, 129)):
        for oy in range(0, H, rows):
            y0, ye = max(oy - 2, 0), min(oy + rows, H)
            n = ye - y0 + 2
            n_in = min(y0 + n, H) - y0
            nbox = -(-n_in // 2)
            S = Slots(4)
            for j in range(min(4, nbox)):
                S.issue(j, j)
            j = 0
            while 2 * j < n:
                if 2 * j < n_in:
                    S.wait(j, j % 4, (j // 4) & 1)
                if j + 4 < nbox:
                    S.issue(j + 4, j % 4)
                j += 1
            assert all(S.read) and sum(S.phases) == nbox


# ---- shared memory: mbarriers, then warps x slots, from a 128-byte aligned base ----

BARS = 512


def check_reads(smem, threads, slot_bytes, kring, row_bytes, rows, esize, reads, planes=1):
    """reads(lane): (first, last) element of a box row, counted from the row's start,
    that the lane loads.  The base lies up to 127 bytes into the allocation."""
    warps = threads // 32
    for pad in (0, 16, 112, 127):
        base = pad
        for w, s, row, lane in itertools.product(range(warps), range(kring), range(rows * planes), range(32)):
            at = base + BARS + (w * kring + s) * slot_bytes + row * row_bytes
            first, last = reads(lane)
            assert at + first * esize >= base and at + (last + 1) * esize <= smem, (w, s, row, lane)


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("threads", [32, 128, 256])
def test_stencil_reads(dtype, threads):
    """Four columns and the two on either side; stored lanes stay inside the row."""
    st = {"f32": hp.HP_F32, "f16": hp.HP_F16, "bf16": hp.HP_BF16}[dtype]
    esize = 4 if dtype == "f32" else 2
    p = pipelines.unsharp(storage=st)
    p.schedule([0, 0], threads=[threads])
    info = p.group_info([(1000, 700)], 0)
    assert info.kernel == hp.HP_KERNEL_STENCIL_ROWS and info.threads == threads
    check_reads(info.smem_bytes, threads, 512 * esize, 3, 128 * esize, 4, esize,
                lambda lane: (4 * lane - 2, 4 * lane + 5))
    halo = 1 if esize == 4 else 2
    assert all(0 <= 4 * lane - 2 and 4 * lane + 5 < 128 for lane in range(halo, 32 - halo))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("threads", [32, 128, 256])
def test_max_filter_reads(dtype, threads):
    """Four columns and the four on either side."""
    st = hp.HP_F32 if dtype == "f32" else hp.HP_BF16
    esize, pad, box_w = (4, 0, 128) if dtype == "f32" else (2, 4, 136)
    p = pipelines.max_filter(4, storage=st, io_storage=st)
    p.schedule([0, 0], threads=[threads])
    info = p.group_info([(1000, 700)], 0)
    assert info.kernel == hp.HP_KERNEL_MAX_ROWS and info.threads == threads
    slot = -(-box_w * 4 * esize // 128) * 128
    check_reads(info.smem_bytes, threads, slot, 3, box_w * esize, 4, esize,
                lambda lane: (4 * lane + pad - 4, 4 * lane + pad + 7))
    assert all(pad <= 4 * lane + pad - 4 and 4 * lane + pad + 7 < box_w for lane in range(1, 31))


def test_interpolate_level_reads():
    """The two fine columns of a lane, clamped: inside the box of 68 columns."""
    p = pipelines.interpolate_finest()
    info = p.group_info([(1000, 700), (500, 350)], 0)
    assert info.kernel == hp.HP_KERNEL_INTERP_ROWS
    slot = -(-68 * 2 * 4 * 4 // 128) * 128
    assert info.smem_bytes >= 128 + BARS + info.threads // 32 * 3 * slot
    for W, lane in itertools.product((1, 2, 59, 60, 61, 1000), range(1, 31)):
        for strip in range(-(-((W + 1) // 2) // 30)):
            m = 30 * strip + lane - 1
            if 2 * m <= W - 1:
                for x in (2 * m, min(2 * m + 1, W - 1)):
                    assert 0 <= x - (60 * strip - 4) < 68
