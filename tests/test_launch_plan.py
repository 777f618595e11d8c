"""The launch plan of the stencil kernels (csrc/plan.h, host arithmetic): every grid that some
tile of a table can launch gets a launch within the grid and shared-memory limits, also where
the preferred tile, the room for receiver blocks or the one-block kernel drop out."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_03032_gb300", "csrc")
NSM = 152

WRAP = """
#include "plan.h"
extern "C" int choose(const double *v, int n, int forced, int nx, int ny, int nz, int nshots,
                      int nsm, int *out) {
    fdsweep::PlanEntry e[8];
    for (int i = 0; i < n; ++i, v += 11)
        e[i] = fdsweep::PlanEntry{(int)v[0], (int)v[1], (int)v[2], (int)v[3], (float)v[4],
                                  (float)v[5], (float)v[6], v[7], (int)v[8], (int)v[9], v[10] != 0};
    const fdsweep::PlanChoice c = fdsweep::choose_plan(e, n, forced, nx, ny, nz, nshots, nsm);
    out[0] = c.zchunk;
    out[1] = c.nzc;
    return c.entry;
}
"""

# bx, by, bz, per_sm, launch, lat, thr, warm-up planes, longest chunk, long chunk, spare
MARCH8 = (64, 8, 0, 5, 3.57, 0.278, 0.162, 1.6, 47000, 0, 0)
MARCH16 = (64, 16, 0, 3, 2.44, 0.299, 0.269, 3.64, 35000, 0, 0)
WIDE = (64, 28, 0, 1, 1.76, 0.609, 0.325, 9.4, 900, 0, 0)
DIRECT = (32, 8, 8, 3, 2.50, 1.41, 1.20, 0, 40000, 0, 0)
SPARE16 = MARCH16[:10] + (1,)
HALF = (64, 16, 0, 3, 5.23, 0.347, 0.290, 4.3, 36000, 8192, 0)
TABLES = {"so4": (MARCH8, MARCH16, DIRECT), "so4 damp field": (MARCH8, DIRECT, SPARE16),
          "wide": (MARCH8, WIDE, DIRECT), "binary16": (HALF,), "fused": (MARCH16,)}


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, lib = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib],
                   check=True)
    fn = ctypes.CDLL(lib).choose

    def run(table, shape, nshots, forced=-1):
        flat = [float(x) for e in table for x in e]
        out = (ctypes.c_int * 2)()
        nz, ny, nx = shape
        i = fn((ctypes.c_double * len(flat))(*flat), len(table), forced, nx, ny, nz, nshots, NSM,
               out)
        return i, out[0], out[1]
    return run


def launchable(e, shape, nshots):
    """Whether the limits alone allow the entry: 65535 blocks in y and z."""
    nz, ny, _ = shape
    chunk = e[2] or e[8]
    return -(-ny // e[1]) <= 65535 and nshots * -(-nz // chunk) <= 65535


def check(table, shape, nshots, got):
    i, zchunk, nzc = got
    nz, ny, nx = shape
    e = table[i]
    assert zchunk >= 1 and nzc == -(-nz // zchunk)
    assert nshots * nzc <= 65535 and -(-ny // e[1]) <= 65535
    assert zchunk == e[2] if e[2] else zchunk <= e[8]


@pytest.mark.parametrize("name,shape,nshots", [
    ("so4", (48461, 2, 4), 30001),             # two chunks per column, no room for receivers
    ("so4 damp field", (48461, 2, 4), 30001),
    ("binary16", (50000, 2, 8), 31000),
    ("so4", (2, 600000, 4), 1),                # too many rows for the 8-row tiles
    ("so4 damp field", (2, 600000, 4), 1),
    ("so4", (3, 5, 7), 65535), ("wide", (901, 9, 9), 60000)])
def test_extreme_grids_have_a_launch(choose, name, shape, nshots):
    table = TABLES[name]
    got = choose(table, shape, nshots)
    assert got[0] >= 0
    check(table, shape, nshots, got)


@pytest.mark.parametrize("name", sorted(TABLES))
def test_a_launch_exists_exactly_where_the_limits_allow_one(choose, name):
    table, rng = TABLES[name], random.Random(7)
    log = lambda hi: int(2 ** rng.uniform(1, hi))  # noqa: E731
    for _ in range(3000):
        shape, nshots = (log(17), log(21), log(12)), log(17) - 1
        got = choose(table, shape, nshots)
        # the one-block kernel alone is not taken beyond two waves
        able = [launchable(e, shape, nshots) for e in table if not e[2]]
        if any(able):
            assert got[0] >= 0
        if got[0] >= 0:
            check(table, shape, nshots, got)
            assert not table[got[0]][10] or sum(able) == 1
        for i, e in enumerate(table):
            f = choose(table, shape, nshots, forced=i)
            assert f[0] == (i if launchable(e, shape, nshots) else -1)
            if f[0] >= 0:
                check(table, shape, nshots, f)


def test_ordinary_grids_leave_room_for_receiver_blocks(choose):
    rng = random.Random(3)
    for _ in range(500):
        shape = tuple(rng.randint(2, 800) for _ in range(3))
        for table in TABLES.values():
            i, zchunk, nzc = choose(table, shape, rng.randint(1, 64))
            assert i >= 0 and nzc * 64 <= 60000
