"""GPU: the FP32 rounding of the nested passes beside that of single sweeps, on white noise with small node spacings: the
same spacing and step on 256 rows, which the nested passes take, and on 255, which run by single sweeps.  An
inverse of either form rounds its recurrences once a node; the nested one adds at most three roundings
of that size per chunk of eight nodes (the chunk's aggregate, its start correction, its first value): its
error may be sqrt(11/8) times the other's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.solver import OracleSolver, Problem  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402


@pytest.mark.parametrize("M", [2, 4, 6])
@pytest.mark.parametrize("spacing", [2 * np.pi / 1500, 2 * np.pi / 2048])
def test_nested_rounding_is_that_of_single_sweeps(spacing, M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Solver
    build.build_library()
    nx, its, dt, eps = 1056, 6, 1e-4, 0.05
    rms = {}
    for ny in (255, 256):
        L = dict(Lx=spacing * nx, Ly=spacing * ny)
        err = []
        for seed in range(2):
            u0 = uniform_noise((ny, nx), 0.05, seed=seed, mean=0.1).astype(np.float32).astype(np.float64)
            prob = Problem(nx=nx, ny=ny, bc="periodic", eps=eps, M=M, tol=1e-30, max_iter=its, **L)
            ref, _ = OracleSolver(prob).step(u0, dt, "be")
            with Solver(nx=nx, ny=ny, bc="periodic", eps=eps, quad_order=M, precision="fp32", tol=1e-30, max_iter=its, **L) as s:
                s.set_execution("host_loop")
                s.profile_enable(True)
                u = torch.tensor(u0, device="cuda", dtype=torch.float32)
                s.step(u, dt, "be", raise_on_nonconvergence=False)
                nested = "cols_nested" in s.profile_collect()
                err.append(u.double().cpu().numpy() - ref)
            assert nested == (ny == 256)
        rms[ny] = np.sqrt(np.mean(np.square(err)))
    print("rms error", rms)
    assert rms[256] <= np.sqrt(11 / 8) * rms[255], rms
