"""Every kernel of the two-pass TTI scheme gives the same bits.

Marching and one-block kernels evaluate a point with the same operations in the same
order, so all configurations of a radius agree exactly, on grids smaller than a block, with
cut blocks and with one point beyond a block, for both kinds of derivative."""
import numpy as np
import pytest

import workloads
from tests.gpu_util import require_cuda, to_dev

pytestmark = pytest.mark.gpu

H = (10.0, 9.0, 11.0)


@pytest.mark.parametrize("deriv", ["centred", "staggered"])
@pytest.mark.parametrize("so", [4, 8, 12, 16])
@pytest.mark.parametrize("shape,nshots", [((3, 7, 9), 1), ((17, 9, 33), 2), ((24, 21, 71), 1)])
def test_configurations_agree_bitwise(shape, nshots, so, deriv):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300 import _native
    rng = np.random.default_rng(so)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    m = workloads.slowness_squared(rng.uniform(1.5, 3.0, shape))
    eps, th, ph = f32(rng.uniform(0.1, 0.2, shape)), f32(rng.uniform(-1, 1, shape)), \
        f32(rng.uniform(-3, 3, shape))
    delta = f32(0.5 * eps)
    damp = workloads.damping_profile(shape, 4, H, 3.0)
    nt = 8
    dt = 0.5 * workloads.cfl_dt(H, 3.0, eps_max=0.2)
    ext = np.array([(shape[2] - 1) * H[0], (shape[1] - 1) * H[1], (shape[0] - 1) * H[2]])
    src = f32(np.stack([np.full(3, 0.2), np.full(3, 0.8)])[None].repeat(nshots, 0) * ext)
    rec = f32(rng.uniform(0.0, 1.0, (nshots, 5, 3)) * ext)
    wav = f32(rng.standard_normal((nshots, nt, 2)))
    p0, r0 = (f32(rng.standard_normal((nshots, 2) + shape)) for _ in range(2))
    g = fd.Grid(shape, H)
    d = to_dev(torch, m, eps, delta, th, ph, src, wav, rec, damp, p0, r0)
    outs = []
    try:
        for cfg in list(range(_native.num_tti_configs(so))) + [-1]:
            _native.set_tti_config(so, cfg)
            out = fd.tti_forward(g, so, dt, nt, *d[:8], damp=d[8], p_init=d[9], r_init=d[10],
                                 deriv=deriv, receiver="mean", scheme="two_pass")
            outs.append([o.cpu().numpy() for o in out])
    finally:
        _native.set_tti_config(so, -1)
    for out in outs[1:]:
        for got, ref in zip(out, outs[0]):
            np.testing.assert_array_equal(got, ref)
