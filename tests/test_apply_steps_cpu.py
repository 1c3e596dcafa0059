"""The record ring of the FP32 / BF16 subdomain sweeps (Section 3.1) on the host: the step
tables that ras_apply_steps hands out (no CUDA call) are played through in the order in
which the kernel's warps free and fill the ring. Step n is read only when the records of
step n + 1 are in, and its place is free only after that, so each step's successor must have
been let in before it, and no step may be copied over one that has not been read. Boxes from
one cell to the largest, cubes, thin and flat ones, several shapes in a handle, schedules
from one cell to several thousand."""
import os

import pytest


@pytest.fixture(scope="module")
def ras():
    from paper_2007_13966_gb300 import build_lib, ras as R
    if not os.path.exists(R.LIB_PATH):
        build_lib.build()
    R.lib()
    return R


def play(ring, rec, steps):
    """What goes wrong when the sweeps run over `steps` (None: nothing)."""
    ns = len(steps) - 1
    place = [(16 * s[2], 16 * s[2] + 4 * s[1] * rec) for s in steps[:ns]]
    if any(a < 0 or a % 16 or b > ring for a, b in place):
        return "outside the ring"
    nxt = 0

    def fill(limit, done):
        nonlocal nxt
        while nxt <= min(limit, ns - 1):
            a, b = place[nxt]
            for t in range(done, nxt):                 # in the ring, not read yet
                if a < place[t][1] and place[t][0] < b:
                    return f"step {nxt} over step {t}"
            nxt += 1

    bad = fill(steps[ns][3], 0)
    for n in range(ns):
        if bad:
            return bad
        if nxt < min(n + 2, ns):
            return f"step {n} waits for step {nxt}"
        bad = fill(steps[n][3], n + 1)
    return bad or (None if nxt == ns else f"step {nxt} never copied")


CHUNKS = (1, 64, 100, 256, 300, 384, 512, 768, 1024, 1536, 2048, 3000)
BOXES = [(n, n, n) for n in range(1, 26)] + [
    (100, 110, 1), (1, 128, 128), (128, 1, 128), (200, 60, 1), (40, 256, 1), (1, 64, 256), (256, 1, 64), (4, 64, 64),
    (64, 4, 64), (64, 64, 4), (3, 30, 100), (31, 33, 15), (33, 31, 16), (17, 20, 19), (20, 20, 18), (2, 90, 90),
    (255, 8, 8), (8, 255, 8), (8, 8, 255), (16, 32, 32), (32, 16, 32), (32, 32, 16), (40, 20, 20), (5, 5, 200)]


@pytest.mark.parametrize("prec", [32, 16])
@pytest.mark.parametrize("box", BOXES)
def test_sweeps_do_not_wait_for_themselves(ras, box, prec):
    for chunk in (0,) + CHUNKS:
        try:
            ring, rec, shapes = ras.apply_steps(box, (1, 1, 1), 0, prec, chunk)
        except ras.RasError:
            assert chunk > 1024                        # refused: the shared memory of a long schedule
            continue
        assert [s[0] for s in shapes] == [box]
        assert play(ring, rec, shapes[0][1]) is None, (chunk, play(ring, rec, shapes[0][1]))


@pytest.mark.parametrize("dims,parts,overlap", [
    ((128, 128, 64), (8, 8, 4), 2), ((60, 220, 85), (4, 14, 6), 2), ((97, 61, 33), (6, 4, 2), 2),
    ((64, 64, 1), (4, 4, 1), 1), ((24, 20, 12), (2, 2, 1), 2), ((17, 13, 9), (3, 3, 2), 2), ((50, 7, 31), (3, 1, 2), 3)])
def test_handles_of_several_shapes(ras, dims, parts, overlap):
    for prec in (32, 16):
        for chunk in (0,) + CHUNKS:
            try:
                ring, rec, shapes = ras.apply_steps(dims, parts, overlap, prec, chunk)
            except ras.RasError:
                assert chunk > 1024
                continue
            for edges, steps in shapes:
                assert play(ring, rec, steps) is None, (edges, prec, chunk)


def test_arguments_are_checked(ras):
    for dims, parts, prec, chunk in [((8, 8, 8), (1, 1, 1), 64, 0), ((26, 26, 26), (1, 1, 1), 32, 0),
                                     ((8, 8, 8), (9, 1, 1), 32, 0), ((8, 8, 8), (1, 1, 1), 32, -1),
                                     ((20, 20, 20), (1, 1, 1), 32, 1 << 20)]:
        with pytest.raises(ras.RasError):
            ras.apply_steps(dims, parts, 0, prec, chunk)
