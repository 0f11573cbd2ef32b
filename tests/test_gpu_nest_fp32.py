"""GPU: FP32 paths of the nested passes against the oracle, held to the FP32 bar of 1e-6 of the field's scale
(tests/_parity.py): the vector model's column pass (column pairs aligned and not, whole chunks and chunks of two lengths,
one block and a cluster), the 3D passes on slabs of an odd number of columns, and the sixth-order
iterations over two iterations."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.fch import Fch2DSolver as OracleFch2D, FchSolver as OracleFch  # noqa: E402
from oracle.solver import Problem  # noqa: E402
from oracle.split3d import Problem3D, Solver3D as Oracle3D  # noqa: E402
from oracle.vch import VchSolver  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

from _parity import check_fp32  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    build.build_library()


@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("nx,ny,M", [(256, 264, 4), (257, 263, 6), (288, 1040, 6), (301, 521, 4)])
def test_nested_vector_fp32(nx, ny, M, bc):
    from paper_1611_04214_gb300.molt import Solver
    its = 4
    x, y = (np.linspace(0, 1, n, endpoint=bc != "periodic") for n in (nx, ny))
    f = np.sin if bc == "dirichlet" else np.cos
    w = 2 if bc == "periodic" else 1
    p1 = 0.1 * f(np.pi * w * x)[None, :] * f(2 * np.pi * w * y)[:, None]
    p2 = 0.1 * f(2 * np.pi * w * x)[None, :] * f(np.pi * w * y)[:, None]
    u = [a.astype(np.float32).astype(np.float64) for a in (-0.5 + p1, -np.sqrt(3) / 2 + p2)]
    prob = Problem(nx=nx, ny=ny, bc=bc, eps=0.32, M=M, tol=1e-30, max_iter=its)
    o1, o2, _ = VchSolver(prob).step(u[0], u[1], 5e-4, "be")
    with Solver(nx=nx, ny=ny, bc=bc, eps=0.32, quad_order=M, precision="fp32", tol=1e-30, max_iter=its) as s:
        s.set_execution("host_loop")
        s.profile_enable(True)
        g = [torch.tensor(a, device="cuda", dtype=torch.float32) for a in u]
        s.vch_step(g[0], g[1], 5e-4, "be", raise_on_nonconvergence=False)
        launched = s.profile_collect()
    assert launched["cols_nested"][1] == launched["rows_nested"][1] == 2 * its, launched
    scale = max(np.abs(o1).max(), np.abs(o2).max())
    for k, (a, b) in enumerate(zip(g, (o1, o2))):
        check_fp32(f"nested_vch_{nx}x{ny}_M{M}_{bc}_be_1step_{its}it_u{k + 1}", a.cpu().numpy(), b, scale)


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("nx,ny,nz,M", [(225, 45, 67, 4), (75, 29, 520, 2), (61, 520, 23, 6)])
def test_nested_3d_odd_columns(nx, ny, nz, M, bc):
    from paper_1611_04214_gb300.molt import Solver3D
    dt, its = 1e-3, 4
    L = dict(Lx=2 * np.pi, Ly=2 * np.pi * ny / nx, Lz=2 * np.pi * nz / nx)
    u0 = uniform_noise((nz * ny, nx), 0.05, seed=nx + nz, mean=0.05).reshape(nz, ny, nx).astype(np.float32)
    prob = Problem3D(nx=nx, ny=ny, nz=nz, bc=bc, eps=0.1, M=M, tol=1e-30, max_iter=its, **L)
    ref, _ = Oracle3D(prob).step(u0.astype(np.float64), dt, "be")
    with Solver3D(nx, ny, nz, bc=bc, eps=0.1, quad_order=M, tol=1e-30, max_iter=its, **L) as s:
        u = torch.tensor(u0, device="cuda")
        before = s.kernel_launches()
        s.step(u, dt, "be", raise_on_nonconvergence=False)
        launched = s.kernel_launches() - before
        got = u.double().cpu().numpy()
    assert launched < 15 * its, launched
    check_fp32(f"nested3d_{nx}x{ny}x{nz}_M{M}_{bc}_be_1step_4it", got, ref, np.abs(ref + 1).max())


@pytest.mark.parametrize("n,lines,M", [(128, 3, 6), (1024, 5, 4), (2048, 2, 6), (333, 7, 6), (1000, 3, 2)])
def test_fused_sixth_order_lines_fp32(n, lines, M):
    from paper_1611_04214_gb300.molt import Fch1D
    its, dt, eps = 2, 0.05, 0.18
    u0 = uniform_noise((lines, n), 0.3, seed=n, mean=-0.1).astype(np.float32).astype(np.float64)
    ref, _ = OracleFch(Problem(nx=n, eps=eps, M=M, tol=1e-30, max_iter=its, bc="periodic"), 1.0).step(u0, dt)
    with Fch1D(n, lines, bc="periodic", eps=eps, eta=1.0, quad_order=M, tol=1e-30, max_iter=its, precision="fp32") as s:
        u = torch.tensor(u0, device="cuda", dtype=torch.float32)
        s.step(u, dt, raise_on_nonconvergence=False)
        got = u.double().cpu().numpy()
    check_fp32(f"fused_fch1d_{n}x{lines}_M{M}_1step_2it", got, ref, np.abs(ref + 1).max())


@pytest.mark.parametrize("nx,ny,M", [(256, 64, 6), (777, 130, 4), (64, 520, 2), (2048, 45, 6), (300, 77, 2)])
def test_nested_sixth_order_grids_fp32(nx, ny, M):
    from paper_1611_04214_gb300.molt import Fch2D
    its, dt, eps = 2, 0.05, 0.18
    L = dict(Lx=2 * np.pi, Ly=2 * np.pi * ny / nx)
    u0 = uniform_noise((ny, nx), 0.3, seed=nx, mean=-0.1).astype(np.float32).astype(np.float64)
    prob = Problem(nx=nx, ny=ny, bc="periodic", eps=eps, M=M, tol=1e-30, max_iter=its, **L)
    ref, _ = OracleFch2D(prob, 1.0).step(u0, dt)
    with Fch2D(nx, ny, bc="periodic", eps=eps, eta=1.0, quad_order=M, tol=1e-30, max_iter=its, precision="fp32", **L) as s:
        u = torch.tensor(u0, device="cuda", dtype=torch.float32)
        s.step(u, dt, raise_on_nonconvergence=False)
        got = u.double().cpu().numpy()
    check_fp32(f"nested_fch2d_{nx}x{ny}_M{M}_1step_2it", got, ref, np.abs(ref + 1).max())
