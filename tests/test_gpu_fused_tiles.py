"""Both tiles of the fused TTI scheme by their index: 0 (64 x 8), 1 (64 x 16, the built-in
choice) give the same bits, on grids with cut tiles."""
import pytest

from tests.gpu_util import require_cuda, to_dev
from tests.test_gpu_chunks import H
from tests.test_gpu_marching import tti_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("so", [2, 4])
@pytest.mark.parametrize("shape", [(5, 17, 65), (33, 31, 70)])
def test_fused_tiles_agree_bitwise(shape, so):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300 import _native
    p, arrays = tti_problem(shape, 1)
    args = to_dev(torch, *arrays)
    d, u = to_dev(torch, p["damp"], p["u"])
    outs = []
    try:
        for cfg in (0, 1, -1):
            _native.set_tti_config(so, cfg)
            outs.append(fd.tti_forward(fd.Grid(shape, H), so, p["dt"], p["nt"], *args, damp=d,
                                       p_init=u, r_init=u, scheme="fused"))
    finally:
        _native.set_tti_config(so, -1)
    for out in outs[1:]:
        for got, ref in zip(out, outs[0]):
            assert torch.equal(got, ref)
