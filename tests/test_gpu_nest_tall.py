"""GPU: the nested passes on columns of more than 4096 nodes (clusters of 9 to 16 blocks) against the oracle over a
fixed number of iterations: whole chunks and chunks of two lengths, the longest column; rows of 1024 nodes, where
the four passes stay."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.solver import OracleSolver, Problem  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

from _parity import check_fp32  # noqa: E402


@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("nx,ny,M,nested", [(264, 4617, 4, True), (256, 8192, 6, True), (1024, 6152, 2, False)])
def test_tall_columns_match_oracle(nx, ny, M, nested, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Solver
    build.build_library()
    u0 = uniform_noise((ny, nx), 0.05, seed=nx + ny, mean=0.1)
    if bc == "dirichlet":
        u0[0, :] = u0[-1, :] = -1
        u0[:, 0] = u0[:, -1] = -1
    u0 = u0.astype(np.float32).astype(np.float64)
    prob = Problem(nx=nx, ny=ny, bc=bc, eps=0.05, M=M, tol=1e-30, max_iter=3)
    ref, _ = OracleSolver(prob).step(u0, 1e-4, "be")
    with Solver(nx=nx, ny=ny, bc=bc, eps=0.05, quad_order=M, precision="fp32", tol=1e-30, max_iter=3) as s:
        s.set_execution("host_loop")
        s.profile_enable(True)
        u = torch.tensor(u0, device="cuda").to(s.dtype)
        s.step(u, 1e-4, "be", raise_on_nonconvergence=False)
        launched = s.profile_collect()
        got = u.double().cpu().numpy()
    assert ("cols_nested" in launched and launched["cols_nested"][1] == 3) == nested, launched
    check_fp32(f"nested_tall_{nx}x{ny}_M{M}_{bc}_be_1step_3it", got, ref, np.abs(ref + 1).max())
