"""Memory plan of the gradient: checkpoint interval, batch of shots and levels (csrc/plan.h),
and that a call's batches do not depend on how much of the device memory the library's own
pool holds."""
import ctypes
import os
import random
import subprocess

import numpy as np
import pytest

import workloads
from tests.gpu_util import require_cuda, to_dev

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_03032_gb300", "csrc")

WRAP = """
#include "plan.h"
extern "C" void plan(int nsteps, int nshots, long long vol, int every, double total,
                     double available, double fixed, int *out) {
    const fdsweep::GradientPlan p =
        fdsweep::plan_gradient(nsteps, nshots, vol, every, 1 << 30, 8, total, available, fixed);
    const int v[] = {p.K, p.nseg, p.G, p.B, p.nfwd, p.nck};
    for (int i = 0; i < 6; ++i) out[i] = v[i];
}
"""


@pytest.fixture(scope="module")
def fn(tmp_path_factory):
    d = tmp_path_factory.mktemp("gradient_plan")
    src, lib = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib],
                   check=True)
    return ctypes.CDLL(lib).plan


D = ctypes.c_double


@pytest.mark.parametrize("n,nshots,batch", [(32, 64, 64), (32, 128, 128), (40, 128, 128),
                                            (64, 32, 32), (64, 100, 62), (128, 16, 8),
                                            (256, 16, 8), (64, 3, 3), (4, 100000, 16383)])
@pytest.mark.parametrize("every", [0, 8])
def test_small_grids_are_batched_by_their_points(fn, n, nshots, batch, every):
    out = (ctypes.c_int * 6)()
    fn(59, nshots, ctypes.c_longlong(n ** 3), every, D(2.97e11), D(2.9e11), D(24.0 * n ** 3), out)
    assert out[3] == batch


def test_plan_fits_the_memory_it_counts(fn):
    rng = random.Random(2)
    total = 2.97e11
    for _ in range(20000):
        nsteps, nshots = int(2 ** rng.uniform(0, 12)) - 1, int(2 ** rng.uniform(0, 8))
        vol = int(2 ** rng.uniform(8, 31))
        every = rng.choice([0, 0, 1, rng.randint(1, 2 * nsteps + 2)])
        available, fixed = total * rng.uniform(0.01, 1.0), 24.0 * vol
        out = (ctypes.c_int * 6)()
        fn(nsteps, nshots, ctypes.c_longlong(vol), every, D(total), D(available), D(fixed), out)
        K, nseg, G, B, nfwd, nck = out
        assert 1 <= B <= nshots and 1 <= G <= min(K, 8)
        assert B <= 8 or (B - 1) * vol < 1.6e7  # more only of grids that do not fill the device
        assert nseg * K >= nsteps > (nseg - 1) * K if nsteps else nseg == 0
        levels = nfwd + G + 1 + K + 2 + nck
        if B > 1 or G > 1:
            assert B * levels * vol * 4.0 + fixed <= 0.8 * available
        if every == 0 and nseg == 1 and nsteps > 2:  # the whole history is kept
            assert B * (nsteps + 2) * vol * 4.0 <= min(total / 8, available / 4)
        if every:
            assert K == min(every, max(nsteps, 1)) or nsteps == 0
        if B == 1 and G == 1:  # no more than two pairs, the segment and the checkpoints
            assert levels <= 4 + K + 2 + 2 * max(nseg, 1)


@pytest.mark.gpu
def test_batches_do_not_depend_on_the_pool():
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300 import _native
    shape, h, nt, nshots = (96, 96, 96), (10.0, 10.0, 10.0), 121, 8
    m = workloads.slowness_squared(workloads.smooth_random(shape, 3, 5.0, 1.5, 3.0))
    dt = 0.9 * workloads.cfl_dt(h, 3.0)
    rng = np.random.default_rng(4)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    src = f32(rng.uniform(200.0, 700.0, (nshots, 1, 3)))
    rec = f32(rng.uniform(100.0, 800.0, (nshots, 5, 3)))
    args = to_dev(torch, m, src, f32(rng.standard_normal((nshots, nt, 1))), rec,
                  f32(rng.standard_normal((nshots, nt, 5))))

    def launches():
        before = _native.load().fd_launch_count()
        fd.acoustic_gradient(fd.Grid(shape, h), 8, dt, nt, *args, checkpoint_every=60)
        torch.cuda.synchronize()
        return _native.load().fd_launch_count() - before

    want = launches()  # eight shots together, 2.2 GB; the pool keeps them
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - 1500000000, dtype=torch.uint8, device="cuda")
    try:
        got = launches()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert got == want
