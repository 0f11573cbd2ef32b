"""On periodic grids the GPU collects the 2D sixth-order iteration axis by axis (``csrc/fch2d.cpp``).  Here the collected
form, with the oracle's line inverse, is compared with the oracle's iterates over two steps."""
import numpy as np
import pytest

from oracle.fch import fch2d_be_step
from oracle.helmholtz import helmholtz_inverse
from oracle.solver import Problem
from paper_1611_04214_gb300.inputs import uniform_noise


@pytest.mark.parametrize("M", [2, 4, 6])
def test_collected_iteration_equals_the_terms(M):
    nx, ny, dt, eta, eps, its = 32, 26, 0.05, 1.5, 0.18, 4
    prob = Problem(nx=nx, ny=ny, Lx=2 * np.pi, Ly=1.5 * np.pi, bc="periodic", eps=eps, M=M, tol=1e-30, max_iter=its)
    a = np.cbrt(dt * eps ** 4)
    c_eta, c_f, c_p = dt * eta * eps ** 4 / a ** 2, dt * eps ** 2 / a ** 2, dt / a

    def H(f, axis):
        return helmholtz_inverse(f, a, prob.hx if axis else prob.hy, prob.bc, M, axis=axis)

    u = uniform_noise((ny, nx), 0.3, seed=M)
    W, ref, wref = u + 1.0, u, None
    for _ in range(2):
        vn = u + 1.0
        m2 = H(H(H(H(vn, 0), 0), 1), 1)
        for k in range(its + 1):
            hy = H(W, 0)
            v, h = H(hy, 1), H(W, 1) + hy
            xw, lap = v - h + W, (2 * v - h) / a
            if k == its:
                break
            f, fp = v * (v * (v - 3) + 2), v * (3 * v - 6) + 2
            pp = f * fp - (eps ** 2 * fp * lap + eta * eps ** 2 * f)
            s1, E = (3 + 2 * c_eta) * v - 2 * c_f * f + c_p * pp, xw - 3 * W
            p = (3 + c_eta) * v - c_f * f + E
            q, r, t, z = -(s1 + 2 * p), 2 * s1 + E, -E - xw, m2 + xw - W
            e = z + H(t + H(p, 0), 0)
            b = t + H(2 * p - t + H(q, 0), 0)
            c = p + H(q + H(r, 0), 0)
            W = W + e + H(b + H(c, 1), 1)
        u = v - 1.0
        o = fch2d_be_step(prob, ref + 1.0, dt, eta, wref)
        wref, ref = o.w, o.v - 1.0
        assert np.abs(u - ref).max() < 1e-11
