"""Both gradients of the source-to-receiver map from one reverse sweep.

The imaging condition takes several time steps per launch, with a kernel for up to 4 and
8 shots and several batches above; the steps of a segment are a full launch, a remainder
or fewer than a launch takes.  Tolerance: the repository's 1e-4 relative L2 for FP32
against the FP64 oracle; the two entry points run the same operations and differ only in
the order of the atomic injections, 1e-6."""
import numpy as np
import pytest

import oracle
import workloads
from tests.gpu_util import TOL, rel_l2, require_cuda, to_dev

pytestmark = pytest.mark.gpu

H = (10.0, 9.0, 11.0)


@pytest.mark.parametrize("nshots,nt,nsrc,every", [
    (1, 2, 1, 0), (2, 12, 1, 0), (4, 20, 2, 8), (5, 19, 1, 0), (8, 10, 17, 3),
    (9, 18, 1, 0), (16, 11, 1, 5), (17, 13, 1, 0), (3, 1, 1, 0)])
def test_one_sweep_matches_the_separate_calls(nshots, nt, nsrc, every):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300.autograd import acoustic_modeling
    shape, so = (19, 22, 35), 8
    rng = np.random.default_rng(nshots)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    m = workloads.slowness_squared(rng.uniform(1.5, 3.0, shape))
    damp = workloads.damping_profile(shape, 4, H, 3.0)
    dt = 0.9 * workloads.cfl_dt(H, 3.0)
    ext = np.array([(shape[2] - 1) * H[0], (shape[1] - 1) * H[1], (shape[0] - 1) * H[2]])
    src = f32(rng.uniform(0.1, 0.9, (nshots, nsrc, 3)) * ext)
    rec = f32(rng.uniform(0.0, 1.0, (nshots, 6, 3)) * ext)
    wav = f32(rng.standard_normal((nshots, nt, nsrc)))
    dd = f32(rng.standard_normal((nshots, nt, 6)))
    g = fd.Grid(shape, H)
    mt, dampt, srct, wavt, rect, ddt = to_dev(torch, m, damp, src, wav, rec, dd)
    mv, qv = mt.clone().requires_grad_(True), wavt.clone().requires_grad_(True)
    d = acoustic_modeling(mv, qv, g, so, dt, srct, rect, dampt, checkpoint_every=every)
    gm, gq = (t.cpu().numpy() for t in torch.autograd.grad(d, (mv, qv), grad_outputs=ddt))
    sep = fd.acoustic_gradient(g, so, dt, nt, mt, srct, wavt, rect, ddt, damp=dampt,
                               checkpoint_every=every).cpu().numpy()
    adj = fd.acoustic_adjoint(g, so, dt, nt, mt, srct, rect, ddt, damp=dampt).cpu().numpy()
    og = oracle.make_grid(shape, H)
    mref = oracle.acoustic_gradient(og, so, dt, nt, m, src, wav, rec, dd, damp=damp)
    qref = oracle.acoustic_adjoint(og, so, dt, nt, m, src, rec, dd, damp=damp)
    for got, ref, other in ((gm, mref, sep), (gq, qref, adj)):
        if np.any(ref):
            assert rel_l2(got, ref) <= TOL
            assert rel_l2(got, other) <= 1e-6
        else:
            assert not np.any(got) and not np.any(other)
