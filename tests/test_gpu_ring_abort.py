"""A wait that runs out in the acoustic kernel, in every launch configuration (marching rings of
each depth and tile, with and without chunk-edge planes, and the one-block kernel): the call
reports FD_ERR_TIMEOUT, and the next one computes the same bits as before."""
import numpy as np
import pytest

from tests.gpu_util import require_cuda
from tests.test_gpu_failures import _problem, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("so", [2, 4, 8, 12, 16])
def test_every_configuration_gives_up_and_recovers(so):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300 import FdError, _native
    lib = _native.load()
    w = _problem(n=64, so=so, nt=6)
    want = _run(torch, fd, w)
    try:
        for cfg in range(lib.fd_num_acoustic_configs(so)):
            _native.set_acoustic_config(so, cfg)
            lib.fd_set_wait_limit_ns(1)
            try:
                with pytest.raises(FdError) as e:
                    _run(torch, fd, w)
            finally:
                lib.fd_set_wait_limit_ns(0)
            assert e.value.name == "FD_ERR_TIMEOUT", cfg
            got = _run(torch, fd, w)
            np.testing.assert_array_equal(got[0], want[0])
            np.testing.assert_array_equal(got[1], want[1])
    finally:
        _native.set_acoustic_config(so, -1)
