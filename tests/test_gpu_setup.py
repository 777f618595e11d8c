"""The setup kernels (b, damping field factor, TTI a, s and symmetry axis): inputs whose base
address is not 16-byte aligned, rows of every remainder modulo four, and angles over many
turns (range reduction, and its 64-bit path beyond 1000 radians)."""
import numpy as np
import pytest

import oracle
import workloads
from tests.gpu_util import TOL, max_abs_rel, require_cuda, to_dev

pytestmark = pytest.mark.gpu

H = (10.0, 9.0, 11.0)


def shifted(torch, a):
    """The array on the device, one float past a 16-byte boundary."""
    buf = torch.empty(a.size + 5, dtype=torch.float32, device="cuda")
    off = next(k for k in range(1, 5) if (buf.data_ptr() + 4 * k) % 16 == 4)
    v = buf[off:off + a.size].view(a.shape)
    v.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return v


def tti_problem(shape, turns=0.0, seed=3):
    rng = np.random.default_rng(seed)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    m = workloads.slowness_squared(rng.uniform(1.5, 3.0, shape))
    eps = f32(rng.uniform(0.05, 0.3, shape))
    delta = f32(eps * rng.uniform(-0.5, 0.9, shape))
    theta = f32(rng.uniform(-np.pi, np.pi, shape) + turns * rng.integers(-3, 4, shape))
    phi = f32(rng.uniform(-np.pi, np.pi, shape) - turns * rng.integers(-3, 4, shape))
    u = f32(workloads.random_wavefields(shape, seed, sigma=1.5))
    src, wav, rec = np.zeros((1, 0, 3)), np.zeros((1, 4, 0)), np.zeros((1, 0, 3))
    return [m, eps, delta, theta, phi, f32(src), f32(wav), f32(rec)], u


@pytest.mark.parametrize("nx", [16, 17, 18, 19])
def test_unaligned_inputs_give_the_same_bits(nx):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    shape = (11, 9, nx)
    arrays, u = tti_problem(shape)
    g, dt = fd.Grid(shape, H), 0.9 * workloads.cfl_dt(H, 3.0, eps_max=0.3)
    ud = torch.from_numpy(u).cuda()
    a = fd.tti_forward(g, 4, dt, 4, *to_dev(torch, *arrays), p_init=ud, r_init=ud)
    b = fd.tti_forward(g, 4, dt, 4, *[shifted(torch, x) for x in arrays[:5]],
                       *to_dev(torch, *arrays[5:]), p_init=ud, r_init=ud)
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    field = np.abs(u[0, 0]) * np.float32(0.01)
    m, fld = to_dev(torch, arrays[0], field)
    sp = to_dev(torch, *arrays[5:])
    a = fd.acoustic_forward(g, 4, dt, 4, m, *sp, damp=fld, damp_layout="field", u_init=ud)
    b = fd.acoustic_forward(g, 4, dt, 4, shifted(torch, arrays[0]), *sp,
                            damp=shifted(torch, field), damp_layout="field", u_init=ud)
    assert torch.equal(a[1], b[1])


@pytest.mark.parametrize("turns", [2 * np.pi, 40 * np.pi, 200 * np.pi, 3e5])
def test_angles_over_many_turns(turns):
    torch = require_cuda()
    import paper_1807_03032_gb300 as fd
    shape = (12, 10, 21)
    arrays, u = tti_problem(shape, turns)
    dt = 0.9 * workloads.cfl_dt(H, 3.0, eps_max=0.3)
    og = oracle.make_grid(shape, H)
    _, pref, qref = oracle.tti_forward(og, 8, dt, 4, *arrays, p_init=u, r_init=u)
    ud = torch.from_numpy(u).cuda()
    _, p, q = fd.tti_forward(fd.Grid(shape, H), 8, dt, 4, *to_dev(torch, *arrays), p_init=ud,
                             r_init=ud)
    assert max_abs_rel(p.cpu().numpy(), pref) <= TOL
    assert max_abs_rel(q.cpu().numpy(), qref) <= TOL
