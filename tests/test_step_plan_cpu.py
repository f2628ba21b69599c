"""The launches of a step and their scratch (csrc/lbcad_plan.h), on the host: every plane is stepped once, and every
plane that a launch's fields kernel writes lies in the scratch of its own box, as the kernels index it (plane z at
(z - sz0) mod nz of the box's place)."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "step_plan")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror",
                    "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2011_00287_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "step_plan_main.cpp"), "-o", exe], check=True)

    def run(boxes, split=False, tighter=0):
        text = "%d %d %d\n%s\n" % (split, tighter, len(boxes), "\n".join("%d %d %d" % tuple(b) for b in boxes))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
        scratch, parts = (int(v) for v in out[0].split())
        rows = [tuple(int(v) for v in line.split()) for line in out[1:-1]]
        return scratch, rows[:parts], rows[parts:]

    return run


def _check(boxes, scratch, parts, place):
    stepped = [[0] * b[2] for b in boxes]
    expect = 0
    for first, ninst, fz, fn, lz, ln, sz0 in parts:
        assert 1 <= ninst <= 28 and (fn == 0) == (ln == 0)
        assert first in (expect, expect - 1)  # the next instance, or another slab of the last one
        if first == expect:
            expect += ninst
        assert first + ninst == expect and (ln == 0 or ninst == 1)
        used = []
        for i in range(first, first + ninst):
            nx, ny, nz = boxes[i]
            at, sites = place[i]
            written = [z % nz for z in range(fz, fz + fn)] if fn else list(range(nz))
            assert -nz <= fz and len(set(written)) == len(written)
            for z in written:
                assert ((z - sz0) % nz + 1) * nx * ny <= sites, (boxes[i], z)
            planes = [z % nz for z in range(lz, lz + ln)] if ln else list(range(nz))
            for z in planes:
                stepped[i][z] += 1
                assert {(z - 1) % nz, z, (z + 1) % nz} <= set(written)
            used.append((at, at + sites))
        used.sort()
        assert used[0][0] >= 0 and used[-1][1] <= scratch
        assert all(a[1] <= b[0] for a, b in zip(used, used[1:]))
    assert expect == len(boxes)
    assert all(n == 1 for s in stepped for n in s)


LARGE = (1000, 1000, 100)  # above 2^26 sites: stepped in slabs


@pytest.mark.parametrize("boxes", [
    [LARGE, (32, 32, 32)], [(32, 32, 32), LARGE], [LARGE, LARGE], [(32, 32, 32), LARGE, (16, 16, 16), (8, 8, 8)],
    [(1024, 520, 127)], [(256, 256, 256)], [(4, 4, 4)] * 57, [(8192, 8192, 16)], [(16384, 8192, 9), (4, 4, 4)],
])
def test_every_launch_stays_in_its_scratch(plan, boxes):
    _check(boxes, *plan(boxes))


def test_random_batches(plan):
    rng = random.Random(5)
    for _ in range(60):
        boxes = [tuple(rng.choice((4, 7, 32, 96, 300, 700, 1200)) for _ in range(3)) for _ in range(rng.randint(1, 40))]
        _check(boxes, *plan(boxes))


@pytest.mark.parametrize("boxes", [[LARGE, (32, 32, 32)], [(64, 48, 40), (9, 7, 6), (5, 4, 4)], [(8192, 8192, 18)],
                                   [(4, 4, 4)], [(1024, 1024, 1024)]])
def test_smaller_scratch_for_more_launches(plan, boxes):
    """Each step down needs no more scratch than the one before, the last no more than three planes of the largest box;
    every one of them steps every plane once, within its scratch."""
    sizes = []
    for tighter in range(14):
        out = plan(boxes, tighter=tighter)
        _check(boxes, *out)
        sizes.append(out[0])
    assert sizes == sorted(sizes, reverse=True)
    assert sizes[-1] == 3 * max(b[0] * b[1] for b in boxes)


def test_split_steps_take_whole_boxes(plan):
    """Sync coupling and Heun have a scratch of their own for each box: only the instances of a launch are bounded."""
    scratch, parts, place = plan([LARGE, (32, 32, 32)] * 15, split=True)
    assert scratch == 0 and [p[:2] for p in parts] == [(0, 28), (28, 2)]
    assert all(p[2:] == (0, 0, 0, 0, 0) for p in parts)
