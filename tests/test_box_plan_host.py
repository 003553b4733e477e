"""The tiling rule of the direct engine (csrc/box_conv.cuh), compiled for the CPU (no GPU): every box
that the engine accepts has a tile, and the tile fits."""
import os
import random
import shutil
import subprocess

import pytest

from tests._direct_shapes import TALL_TILES

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1308_0730_gb300", "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
MAX_SMEM = 226 * 1024


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("box") / "box_plan_check")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                        "--expt-relaxed-constexpr", "-I", CSRC, "-I", INCLUDE,
                        os.path.join(HERE, "native", "box_plan_check.cu"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(cases):
        text = "\n".join(" ".join(str(n) for n in (*dims, *box, ty)) for dims, box, ty in cases)
        r = subprocess.run([out], input=text, capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stderr
        keys = ("ny", "s", "ck", "cy", "cx", "warps", "smem")
        return [None if line == "none" else dict(zip(keys, map(int, line.split()))) for line in r.stdout.splitlines()]

    return run


def accepted(kx, ky, kz):
    """The direct engine's rule: a 32 x 1 x 4 tile with its halo and the taps in 200 KB."""
    return (kx * ky * kz + (31 + kx) * ky * (3 + kz)) * 4 <= 200 * 1024


def longest(fits):
    n = 1
    while fits(n + 2):
        n += 2
    return n


def test_every_accepted_box_has_a_tile(plan):
    rng = random.Random(3)
    boxes = [(longest(lambda n: accepted(n, a, b)), a, b) for a in (1, 3, 5, 9) for b in (1, 3, 5, 9)]
    boxes += [(a, longest(lambda n: accepted(a, n, b)), b) for a in (1, 3, 9) for b in (1, 3, 9)]
    boxes += [(a, b, longest(lambda n: accepted(a, b, n))) for a in (1, 3, 9) for b in (1, 3, 9)]
    boxes += [(6395, 1, 1), (6397, 1, 1), (6501, 1, 1), (8003, 1, 1)]
    while len(boxes) < 400:
        b = tuple(2 * rng.randrange(0, int(10 ** rng.uniform(0.3, 2.2))) + 1 for _ in range(3))
        if accepted(*b):
            boxes.append(b)
    cases = [(tuple(k + rng.randrange(0, 300) for k in box), box, ty) for box in boxes for ty in (8, 4)]
    for (dims, box, ty), p in zip(cases, plan(cases)):
        what = f"{box} taps on {dims}, ty {ty}: {p}"
        assert p is not None, what
        assert p["smem"] <= MAX_SMEM and 1 <= p["cy"] <= box[1] and 1 <= p["ck"] <= box[2], what
        assert p["cx"] == box[0] or (p["cx"] < box[0] and p["cx"] % 4 == 0), what
        nz = p["warps"] // p["s"]
        assert nz >= 1 and -(-dims[2] // nz) <= 65535 and -(-dims[1] // (8 * p["ny"])) <= 65535, what


def test_tile_choice_does_not_change_the_order_of_sums(plan):
    """Splits of the tap planes and pieces of their rows: the same for ty = 8 and ty = 4. (The rows
    staged at a time may differ: their chains run on, tests/test_gpu_direct_heights.py.)"""
    rng = random.Random(5)
    cases = [((200, 80, 40), (101, 41, 3)), ((194, 356, 87), (1, 191, 3)), ((40, 194, 78), (11, 95, 1)),
             ((6600, 1, 1), (6501, 1, 1)), ((7000, 3, 9), (6501, 1, 5)), ((7000, 9, 9), (6501, 3, 3))]  # in pieces
    while len(cases) < 4000:
        box = tuple(2 * rng.randrange(0, int(10 ** rng.uniform(0.3, 2.0))) + 1 for _ in range(3))
        if accepted(*box):
            cases.append((tuple(k + rng.randrange(0, 200) for k in box), box))
    plans = plan([(dims, box, ty) for dims, box in cases for ty in (8, 4)])
    heights = rows = 0
    for (dims, box), a, b in zip(cases, plans[::2], plans[1::2]):
        assert (a["s"], a["cx"]) == (b["s"], b["cx"]), f"{box} taps on {dims}: {a} and {b}"
        # a chain runs on over the stagings of one plane only
        assert all(p["ck"] == 1 or (p["cy"], p["cx"]) == (box[1], box[0]) for p in (a, b)), f"{box} taps on {dims}: {a}, {b}"
        heights += a["ny"] != b["ny"]
        rows += a["cy"] != b["cy"]
    assert heights > 400 and rows > 4  # the two choices do differ in their tiles


def test_shapes_of_the_tall_tiles(plan):
    """The volumes that test_gpu_direct_tall.py runs do take 16-row tiles."""
    plans = plan([(dims, box, 8) for dims, box in TALL_TILES])
    assert all(p["ny"] == 2 for p in plans), plans
    assert {b[0] for _, b in TALL_TILES} >= {3, 5, 7, 9, 11, 13, 15, 17, 19, 21}
    assert {p["s"] for p in plans} >= {1, 4, 8}
    assert plans[-1]["cy"] < TALL_TILES[-1][1][1]
