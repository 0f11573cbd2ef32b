"""For equal factors the GPU collects the 2D iteration into one pass per axis with two inverses
each (``csrc/nest.cuh``).  Here the collected form, with the oracle's line inverse, is compared with
the oracle's term-by-term map, and the ghost values that stand for the shifted wall stencils
with the oracle's wall weights."""
import numpy as np
import pytest

from oracle.helmholtz import helmholtz_inverse
from oracle.solver import G, Problem, fixed_point_map, stage_params
from oracle.weights import local_weights
from paper_1611_04214_gb300.inputs import uniform_noise


@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("M", [2, 4, 6])
def test_collected_passes_equal_the_terms(bc, M):
    prob = Problem(nx=41, ny=34, Lx=3.0, Ly=2.5, bc=bc, eps=0.1, M=M)
    sp = stage_params(1e-3, prob.eps)
    assert sp.c_in == sp.c_out
    v, Y = uniform_noise((34, 41), 0.7, seed=1), uniform_noise((34, 41), 0.7, seed=2)

    def H(f, axis):
        return helmholtz_inverse(f, sp.c_in, prob.hx if axis == 1 else prob.hy, bc, M, axis=axis)

    g = G(v, sp.lam)
    s, b = H(v, 0), H(g, 0)
    t, a = H(s, 0), H(b, 0)
    A = sp.beta * (2 * a - b) - v + 2 * s - t
    B = -sp.beta * a - 2 * (s - t)
    got = v + (Y - t) + H(B + H(A, 1), 1)
    ref = fixed_point_map(prob, Y, v, sp)
    assert np.abs(got - ref).max() < 1e-13 * np.abs(ref).max() * 10


@pytest.mark.parametrize("M", [2, 4, 6])
@pytest.mark.parametrize("nu", [0.05, 0.7, 5.0])
def test_ghost_values_stand_for_the_wall_stencils(M, nu):
    # J^L_j, J^R_j next to the wall from the shifted stencil on nodes 0..M, and from the centred one
    # with the ghosts -1..-M/2 of the polynomial through those nodes
    H = M // 2
    v = uniform_noise((M + 1 + H,), 1.0, seed=M)
    ghost = [sum(v[o] * np.prod([(-q - k) / (o - k) for k in range(M + 1) if k != o]) for o in range(M + 1))
             for q in range(H, 0, -1)]
    ext = np.concatenate([ghost, v])                       # ext[H + j] = node j
    for j in range(H):
        for side in ("L", "R"):
            wall = np.dot(local_weights(nu, [o - j for o in range(M + 1)], side), v[:M + 1])
            mid = np.dot(local_weights(nu, range(-H, H + 1), side), ext[j:j + M + 1])
            assert abs(wall - mid) < 1e-13 * np.abs(ext).max()
