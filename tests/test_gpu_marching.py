"""The z-marching kernels on grids for which the plan takes the one-block kernels: every
configuration by its index, per-axis and 3-D damping, short and uneven chunks, fewer planes
than the stencil reaches, and the batch engine's march over slots that are not the first ones.

Configuration 0 of each table marches; it is compared with the FP64 oracle (1e-4, the
repository's FP32 tolerance, at every point), and the others with it bit by bit: all evaluate
a point with the same operations in the same order."""
import numpy as np
import pytest

import oracle
import workloads
from tests.gpu_util import TOL, max_abs_rel, rel_l2, require_cuda, to_dev
from tests.test_gpu_chunks import H, SHAPES, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["axes", "field"])
@pytest.mark.parametrize("so", [2, 4, 8, 12, 16])
@pytest.mark.parametrize("shape", SHAPES)
def test_acoustic_configurations(shape, so, layout):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300 import _native
    p = problem(shape, 2)
    damp = p["damp"]
    if layout == "field":
        damp = (0.05 * workloads.smooth_random(shape, 5, 1.5, 0.0, 1.0)).astype(np.float32)
    og = oracle.make_grid(shape, H)
    rref, uref = oracle.acoustic_forward(og, so, p["dt"], p["nt"], p["m"], p["src"], p["wav"],
                                         p["rec"], damp=damp, u_init=p["u"], damp_layout=layout)
    m, d, sx, sw, rx, u = to_dev(torch, p["m"], damp, p["src"], p["wav"], p["rec"], p["u"])
    outs = []
    try:
        for cfg in list(range(_native.num_acoustic_configs(so))) + [-1]:
            _native.set_acoustic_config(so, cfg)
            rec, uf = fd.acoustic_forward(fd.Grid(shape, H), so, p["dt"], p["nt"], m, sx, sw, rx,
                                          damp=d, u_init=u, damp_layout=layout)
            outs.append((rec.cpu().numpy(), uf.cpu().numpy()))
    finally:
        _native.set_acoustic_config(so, -1)
    rec, uf = outs[0]
    assert rel_l2(rec, rref) <= TOL
    assert max_abs_rel(uf, uref) <= TOL
    for r, f in outs[1:]:
        np.testing.assert_array_equal(f, uf)
        np.testing.assert_array_equal(r, rec)


def tti_problem(shape, nshots):
    p = problem(shape, nshots, eps_max=0.3)
    rng = p["rng"]
    eps = rng.uniform(0.05, 0.3, shape).astype(np.float32)
    delta = (eps * rng.uniform(0.0, 0.9, shape)).astype(np.float32)
    theta = rng.uniform(0.0, np.pi, shape).astype(np.float32)
    phi = rng.uniform(-np.pi, np.pi, shape).astype(np.float32)
    return p, [p["m"], eps, delta, theta, phi, p["src"], p["wav"], p["rec"]]


@pytest.mark.parametrize("so", [4, 8, 12, 16])
@pytest.mark.parametrize("shape", SHAPES)
def test_tti_marching_passes(shape, so):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300 import _native
    p, arrays = tti_problem(shape, 1)
    rref, pref, qref = oracle.tti_forward(oracle.make_grid(shape, H), so, p["dt"], p["nt"],
                                          *arrays, damp=p["damp"], p_init=p["u"], r_init=p["u"])
    d, u = to_dev(torch, p["damp"], p["u"])
    try:
        _native.set_tti_config(so, 0)
        rec, pf, qf = fd.tti_forward(fd.Grid(shape, H), so, p["dt"], p["nt"],
                                     *to_dev(torch, *arrays), damp=d, p_init=u, r_init=u,
                                     scheme="two_pass")
    finally:
        _native.set_tti_config(so, -1)
    assert rel_l2(rec.cpu().numpy(), rref) <= TOL
    assert max_abs_rel(pf.cpu().numpy(), pref) <= TOL
    assert max_abs_rel(qf.cpu().numpy(), qref) <= TOL


@pytest.mark.parametrize("deriv", ["centred", "staggered"])
@pytest.mark.parametrize("so", [2, 4])
@pytest.mark.parametrize("shape", SHAPES)
def test_fused_and_two_pass_schemes_agree_bitwise(shape, so, deriv):
    """The automatic scheme changes from one to the other with the size of the grid."""
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    p, arrays = tti_problem(shape, 2)
    d, u = to_dev(torch, p["damp"], p["u"])
    args = to_dev(torch, *arrays)
    outs = [fd.tti_forward(fd.Grid(shape, H), so, 0.5 * p["dt"], p["nt"], *args, damp=d, p_init=u,
                           r_init=u, deriv=deriv, receiver="mean", scheme=scheme)
            for scheme in ("fused", "two_pass", "auto")]
    for out in outs[1:]:
        for got, ref in zip(out, outs[0]):
            assert torch.equal(got, ref)


@pytest.mark.parametrize("so", [4, 8, 16])
def test_engine_marches_over_the_slots_in_use(so):
    """More blocks than the one-block kernel is taken for, also with the two slots left."""
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    from paper_1807_03032_gb300.serving import Engine
    shape, h, nts = (100, 104, 112), (10.0, 10.0, 10.0), (8, 22, 30)
    m = workloads.slowness_squared(workloads.smooth_random(shape, 3, 5.0, 1.5, 3.0))
    damp = workloads.damping_profile(shape, 8, h, 3.0)
    dt = 0.8 * workloads.cfl_dt(h, 3.0)
    rng = np.random.default_rng(8)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    g, (mt, dpt) = fd.Grid(shape, h), to_dev(torch, m, damp)
    eng = Engine(g, so, dt, mt, dpt, max_slots=3, max_nsrc=1, max_nrec=12)
    shots, outs, slots = [], [], []
    for nt in nts:  # receivers close enough for eight steps
        src = rng.uniform(200.0, 800.0, (1, 3))
        shots.append(to_dev(torch, f32(src), f32(rng.standard_normal((nt, 1))),
                            f32(src + rng.uniform(-30.0, 30.0, (12, 3)))))
        outs.append(torch.empty((nt, 12), device="cuda"))
        slots.append(eng.add_shot(nt, *shots[-1], outs[-1]))
    eng.step(8)
    eng.release(slots[0])  # the other two go on in slots 1 and 2
    for _ in range(11):
        eng.step(2)
    eng.sync()
    eng.close()
    for nt, (s, w, r), out in zip(nts, shots, outs):
        ref, _ = fd.acoustic_forward(g, so, dt, nt, mt, s[None], w[None], r[None], damp=dpt,
                                     return_final=False)
        assert float(ref.abs().max()) > 0
        assert torch.equal(out, ref[0])
