"""GPU: FP32 SDC2 on lines and grids over some tens of steps against the oracle (fixed iterations).  The corrected
level's right side is formed by the inverses that its iteration runs, so that the rounding of their weights cancels and
a step does not drift; the bar is the FP32 one, 1e-6 of max|u + 1| (tests/_parity.py).  The Dirichlet states here sit
near the wall value (max|u + 1| = 0.4), where backward Euler is 1.8 to 2.2e-6 off as well: they are guarded at 4e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.solver import OracleSolver, Problem  # noqa: E402

from _parity import check_fp32  # noqa: E402


# node spacings small beside the kernel's decay length, where a rounded decay weighs most
@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("nx,ny,steps", [(1000, 1, 40), (4096, 1, 40), (512, 264, 6)])
def test_sdc2_fp32_does_not_drift(nx, ny, steps, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Solver
    build.build_library()
    its, dt, eps = 6, 1e-4, 0.05
    x, y = (np.linspace(0, 1, n, endpoint=bc != "periodic") if n > 1 else np.zeros(1) for n in (nx, ny))
    if bc == "dirichlet":
        u0 = -1 + 0.4 * np.sin(np.pi * x)[None, :] * (np.sin(np.pi * y)[:, None] if ny > 1 else 1.0)
        u0[:, 0] = u0[:, -1] = -1
        if ny > 1:
            u0[0, :] = u0[-1, :] = -1
    else:
        u0 = 0.3 + 0.05 * np.cos(2 * np.pi * x)[None, :] * np.cos(2 * np.pi * y)[:, None]
    u0 = u0.astype(np.float32).astype(np.float64)
    o = OracleSolver(Problem(nx=nx, ny=ny, bc=bc, eps=eps, M=4, tol=1e-30, max_iter=its))
    ref = u0
    with Solver(nx=nx, ny=ny, bc=bc, eps=eps, quad_order=4, precision="fp32", tol=1e-30, max_iter=its) as s:
        u = torch.tensor(u0, device="cuda", dtype=torch.float32)
        for _ in range(steps):
            s.step(u, dt, "sdc2", raise_on_nonconvergence=False)
            ref, _ = o.step(ref, dt, "sdc2")
        got = u.double().cpu().numpy().reshape(ref.shape)
    check_fp32(f"sdc2_{nx}x{ny}_{bc}_{steps}steps_{its}it", got, ref, np.abs(ref + 1).max(),
               known_miss=(4.0, "rounding of the stored variable beside a small max|v|") if bc == "dirichlet" else None)
