"""GPU: the nested column and row passes (``csrc/nest.cuh``, ``csrc/nest_rows.cuh``) against the
oracle over a fixed number of iterations, at the sizes where their cuts change: columns of whole
chunks in one block, of an odd number of chunks, of chunks of two lengths, over two blocks of a
cluster and over five; rows packed within a warp and over a block, and one value per register."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.solver import OracleSolver, Problem  # noqa: E402
from oracle.vch import VchSolver  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

from _parity import check_fp32, check_fp64  # noqa: E402

# (nx, ny, M)
SHAPES = [(256, 256, 4), (257, 263, 2), (1056, 264, 6), (1001, 520, 4), (256, 2049, 6)]


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    build.build_library()


@functools.lru_cache(maxsize=4)
def _oracle(nx, ny, M, bc):
    u = uniform_noise((ny, nx), 0.05, seed=nx + ny, mean=0.1)
    if bc == "dirichlet":
        u[0, :] = u[-1, :] = -1
        u[:, 0] = u[:, -1] = -1
    u = u.astype(np.float32).astype(np.float64)
    prob = Problem(nx=nx, ny=ny, bc=bc, eps=0.05, M=M, tol=1e-30, max_iter=4)
    out, _ = OracleSolver(prob).step(u, 1e-4, "be")
    return u, out


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("nx,ny,M", SHAPES)
def test_nested_steps_match_oracle(nx, ny, M, bc, precision):
    from paper_1611_04214_gb300.molt import Solver
    u0, ref = _oracle(nx, ny, M, bc)
    with Solver(nx=nx, ny=ny, bc=bc, eps=0.05, quad_order=M, precision=precision, tol=1e-30, max_iter=4) as s:
        s.set_execution("host_loop")
        s.profile_enable(True)
        u = torch.tensor(u0, device="cuda").to(s.dtype)
        s.step(u, 1e-4, "be", raise_on_nonconvergence=False)
        launched = s.profile_collect()
        got = u.double().cpu().numpy()
    assert launched["cols_nested"][1] == launched["rows_nested"][1] == 4, launched
    scale = np.abs(ref + 1).max()
    case = f"nested_{nx}x{ny}_M{M}_{bc}_be_1step_4it"
    if precision == "fp64":
        check_fp64(case + "_fp64", got, ref, 1e-11 * scale)
    else:
        check_fp32(case, got, ref, scale)


@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
def test_nested_vector_steps_match_oracle(bc):
    from paper_1611_04214_gb300.molt import Solver
    nx, ny = 288, 263
    x, y = (np.linspace(0, 1, n, endpoint=bc != "periodic") for n in (nx, ny))
    f = np.sin if bc == "dirichlet" else np.cos
    w = 2 if bc == "periodic" else 1
    p1 = 0.1 * f(np.pi * w * x)[None, :] * f(2 * np.pi * w * y)[:, None]
    p2 = 0.1 * f(2 * np.pi * w * x)[None, :] * f(np.pi * w * y)[:, None]
    u = (-0.5 + p1, -np.sqrt(3) / 2 + p2)
    prob = Problem(nx=nx, ny=ny, bc=bc, eps=0.32, M=4, tol=1e-30, max_iter=5)
    o1, o2, _ = VchSolver(prob).step(u[0], u[1], 5e-4, "be")
    with Solver(nx=nx, ny=ny, bc=bc, eps=0.32, quad_order=4, precision="fp64", tol=1e-30, max_iter=5) as s:
        g = [torch.tensor(a, device="cuda") for a in u]
        s.vch_step(g[0], g[1], 5e-4, "be", raise_on_nonconvergence=False)
    for a, b in zip(g, (o1, o2)):
        check_fp64(f"nested_vch_{nx}x{ny}_{bc}_be_1step_5it_fp64", a.cpu().numpy(), b, 1e-11)
