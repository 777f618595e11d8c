"""Grids whose columns are cut into very short or uneven z chunks, against the FP64 oracle.

The stencil kernels march z chunks whose number follows from the grid (few planes per
chunk on small grids); a chunk starts with planes of its lower neighbour and a grid may
have fewer planes than the stencil reaches.  Tolerance: the repository's 1e-4 relative
L2 for FP32, on wavefields (every point of them: a wrong plane shows) and traces."""
import numpy as np
import pytest

import oracle
import workloads
from tests.gpu_util import TOL, max_abs_rel, rel_l2, require_cuda, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [(3, 70, 9), (17, 9, 130), (41, 33, 66), (131, 10, 18)]
H = (10.0, 9.0, 11.0)


def problem(shape, nshots, eps_max=0.0):
    rng = np.random.default_rng(sum(shape))
    v = rng.uniform(1.5, 3.0, shape)
    ext = np.array([(shape[2] - 1) * H[0], (shape[1] - 1) * H[1], (shape[0] - 1) * H[2]])
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    dt = 0.9 * workloads.cfl_dt(H, 3.0, eps_max=eps_max)
    nt = 9
    u = np.stack([np.stack([workloads.smooth_random(shape, 7 * s + k, 1.5, -1.0, 1.0)
                            for k in range(2)]) for s in range(nshots)])
    return dict(m=workloads.slowness_squared(v),
                damp=workloads.damping_profile(shape, 4, H, 3.0), dt=dt, nt=nt,
                src=f32(rng.uniform(0.1, 0.9, (nshots, 2, 3)) * ext),
                rec=f32(rng.uniform(0.0, 1.0, (nshots, 7, 3)) * ext),
                wav=f32(rng.standard_normal((nshots, nt, 2))), u=f32(u), rng=rng)


@pytest.mark.parametrize("so", [4, 8, 12, 16])
@pytest.mark.parametrize("shape", SHAPES)
def test_acoustic_short_chunks(shape, so):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    p = problem(shape, 2)
    g = fd.Grid(shape, H)
    m, d, sx, sw, rx, u = to_dev(torch, p["m"], p["damp"], p["src"], p["wav"], p["rec"], p["u"])
    og = oracle.make_grid(shape, H)
    rref, uref = oracle.acoustic_forward(og, so, p["dt"], p["nt"], p["m"], p["src"], p["wav"],
                                         p["rec"], damp=p["damp"], u_init=p["u"])
    rec, uf = fd.acoustic_forward(g, so, p["dt"], p["nt"], m, sx, sw, rx, damp=d, u_init=u)
    assert rel_l2(rec.cpu().numpy(), rref) <= TOL
    assert rel_l2(uf.cpu().numpy(), uref) <= TOL
    assert max_abs_rel(uf.cpu().numpy(), uref) <= TOL
    # the 3-D damping variant on the same profiles summed point by point
    nz, ny, nx = shape
    dd = p["damp"]
    field = (dd[nx + ny:][:, None, None] + dd[nx:nx + ny][None, :, None]
             + dd[:nx][None, None, :]).astype(np.float32)
    _, uf = fd.acoustic_forward(g, so, p["dt"], p["nt"], m, sx, sw, rx, u_init=u,
                                damp=torch.from_numpy(field).cuda(), damp_layout="field")
    assert max_abs_rel(uf.cpu().numpy(), uref) <= TOL


@pytest.mark.parametrize("so", [4, 8, 12, 16])
@pytest.mark.parametrize("shape", SHAPES)
def test_tti_short_chunks(shape, so):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    p = problem(shape, 1, eps_max=0.3)
    rng = p["rng"]
    eps = rng.uniform(0.05, 0.3, shape).astype(np.float32)
    delta = (eps * rng.uniform(0.0, 0.9, shape)).astype(np.float32)
    theta = rng.uniform(0.0, np.pi, shape).astype(np.float32)
    phi = rng.uniform(-np.pi, np.pi, shape).astype(np.float32)
    og = oracle.make_grid(shape, H)
    rref, pref, qref = oracle.tti_forward(og, so, p["dt"], p["nt"], p["m"], eps, delta, theta,
                                          phi, p["src"], p["wav"], p["rec"], damp=p["damp"],
                                          p_init=p["u"], r_init=p["u"])
    args = to_dev(torch, p["m"], eps, delta, theta, phi, p["src"], p["wav"], p["rec"])
    d, u = to_dev(torch, p["damp"], p["u"])
    rec, pf, qf = fd.tti_forward(fd.Grid(shape, H), so, p["dt"], p["nt"], *args, damp=d,
                                 p_init=u, r_init=u)
    assert rel_l2(rec.cpu().numpy(), rref) <= TOL
    assert max_abs_rel(pf.cpu().numpy(), pref) <= TOL
    assert max_abs_rel(qf.cpu().numpy(), qref) <= TOL
