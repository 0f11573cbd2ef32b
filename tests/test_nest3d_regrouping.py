"""For equal factors the GPU collects the 3D iteration into one pass per axis (``csrc/solver3d.cpp``), and the
sixth-order iteration on lines into three inverses (``csrc/nest_rows.cuh``).  Here both collected forms, with the
oracle's line inverse, are compared with the oracle's terms."""
import numpy as np
import pytest

from oracle.fch import fch_be_step
from oracle.helmholtz import helmholtz_inverse
from oracle.solver import G, Problem, stage_params
from oracle.split3d import H, Problem3D, fixed_point_map
from paper_1611_04214_gb300.inputs import uniform_noise


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("M", [2, 4, 6])
def test_collected_3d_passes_equal_the_terms(bc, M):
    prob = Problem3D(nx=22, ny=19, nz=17, Lx=3.0, Ly=2.5, Lz=2.0, bc=bc, eps=0.1, M=M)
    sp = stage_params(1e-3, prob.eps)
    assert sp.c_in == sp.c_out
    w, Y = (uniform_noise((17 * 19, 22), 0.7, seed=k).reshape(17, 19, 22) for k in (1, 2))

    def h(f, axis):
        return H(prob, f, sp.c_in, axis)

    g = G(w, sp.lam)
    s, b = h(w, "z"), h(g, "z")
    t, e = h(s, "z"), h(b, "z")
    a3, b3 = t, -2 * s + 4 * t - sp.beta * e
    c3 = -w + 4 * s - 4 * t + sp.beta * (3 * e - b)
    E = Y - h(h(a3, "y"), "y")
    q1, q2 = h(-2 * a3 + h(b3, "y"), "y"), -a3 + h(b3 + h(c3, "y"), "y")
    got = w + E + h(q1 + h(q2, "x"), "x")
    ref = fixed_point_map(prob, Y, w, sp)
    assert np.abs(got - ref).max() < 1e-13 * np.abs(ref).max() * 10


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("M", [2, 6])
def test_collected_sixth_order_iteration_equals_the_terms(bc, M):
    prob = Problem(nx=48, eps=0.18, M=M, tol=1e-30, max_iter=3, bc=bc)
    dt, eta, eps = 0.05, 1.5, 0.18
    vn = 1.0 + uniform_noise((2, 48), 0.3, seed=M)
    a = np.cbrt(dt * eps ** 4)
    c_eta, c_f, c_p = dt * eta * eps ** 4 / a ** 2, dt * eps ** 2 / a ** 2, dt / a

    def h(f):
        return helmholtz_inverse(f, a, prob.hx, bc, M, axis=1)

    v, lap, h2 = vn.copy(), (h(vn) - vn) / a, h(h(vn))
    for _ in range(3):
        f, fp = v * (v * (v - 3) + 2), v * (3 * v - 6) + 2
        p = f * fp - eps ** 2 * fp * lap - eta * eps ** 2 * f
        q = h(c_eta * v - c_f * f + c_p * p) - ((3 + c_eta) * v - c_f * f)
        z = h2 + h(q) - q
        v = h(z)
        lap = (v - z) / a
    r = fch_be_step(prob, vn, dt, eta)
    assert np.abs(v - r.v).max() < 1e-11 * np.abs(r.v).max()
    assert np.abs(lap - r.lap_v).max() < 1e-9 * np.abs(r.lap_v).max()
