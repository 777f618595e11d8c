"""Gradient over a kept history of more than 2 GiB per shot (beyond the largest pitch of a 2-D
copy or fill): every shot starts from rest, also in memory that an earlier call used.
Tolerance: the two runs do the same operations and differ only in the order of the atomic
injections, 1e-6 as for the other gradient comparisons."""
import numpy as np
import pytest

import workloads
from tests.gpu_util import rel_l2, require_cuda, to_dev

pytestmark = pytest.mark.gpu


def test_history_beyond_two_gib_per_shot():
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    shape, h, nt, nshots = (72, 80, 100), (10.0, 10.0, 10.0), 960, 3
    assert (nt + 1) * 4 * 72 * 80 * 100 > 2 ** 31
    m = workloads.slowness_squared(workloads.smooth_random(shape, 3, 5.0, 1.5, 3.0))
    damp = workloads.damping_profile(shape, 8, h, 3.0)
    dt = 0.9 * workloads.cfl_dt(h, 3.0)
    rng = np.random.default_rng(6)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    src = f32(rng.uniform(100.0, 600.0, (nshots, 1, 3)))
    rec = f32(rng.uniform(100.0, 600.0, (nshots, 5, 3)))
    wav = f32(np.stack([workloads.ricker(nt, dt, f0=0.02) * (s + 1) for s in range(nshots)]))
    args = to_dev(torch, m, src, wav[..., None], rec, f32(rng.standard_normal((nshots, nt, 5))))
    g, d = fd.Grid(shape, h), to_dev(torch, damp)[0]
    kept = fd.acoustic_gradient(g, 4, dt, nt, *args, damp=d)
    short = fd.acoustic_gradient(g, 4, dt, nt, *args, damp=d, checkpoint_every=31)
    again = fd.acoustic_gradient(g, 4, dt, nt, *args, damp=d)
    for got in (kept, again):
        assert rel_l2(got.cpu().numpy(), short.cpu().numpy()) <= 1e-6
