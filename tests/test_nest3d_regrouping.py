"""For equal factors the GPU collects the 3D iteration into one pass per axis (``csrc/solver3d.cpp``).  Here the
collected form, with the oracle's line inverse, is compared with the oracle's terms."""
import numpy as np
import pytest

from oracle.solver import G, stage_params
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
