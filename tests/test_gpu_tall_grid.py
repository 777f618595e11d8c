"""A grid with more rows than 65535 tiles of eight hold: the plan takes a taller tile.
Tolerance: the repository's 1e-4 for FP32, at every point."""
import numpy as np
import pytest

import oracle
import workloads
from tests.gpu_util import TOL, max_abs_rel, require_cuda, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["axes", "field"])
def test_more_rows_than_eight_row_tiles_hold(layout):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    shape, h, nt = (2, 600000, 4), (10.0, 10.0, 10.0), 4
    rng = np.random.default_rng(12)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    m = workloads.slowness_squared(rng.uniform(1.5, 3.0, shape))
    damp = f32(0.01 * rng.random(shape if layout == "field" else sum(shape)))
    u = f32(rng.standard_normal((1, 2) + shape))
    src, rec, wav = np.zeros((1, 0, 3)), np.zeros((1, 0, 3)), np.zeros((1, nt, 0))
    dt = 0.5 * workloads.cfl_dt(h, 3.0)
    arrays = [m] + [f32(a) for a in (src, wav, rec)]
    _, ref = oracle.acoustic_forward(oracle.make_grid(shape, h), 4, dt, nt, *arrays, damp=damp,
                                     u_init=u, damp_layout=layout)
    d, ui = to_dev(torch, damp, u)
    _, uf = fd.acoustic_forward(fd.Grid(shape, h), 4, dt, nt, *to_dev(torch, *arrays), damp=d,
                                u_init=ui, damp_layout=layout)
    assert max_abs_rel(uf.cpu().numpy(), ref) <= TOL
