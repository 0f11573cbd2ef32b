"""GPU: the sixth-order iteration on periodic lines in one kernel (``nest_fch_kernel``) against the oracle over a
fixed number of iterations: packed lines within a warp and over a block, one value per register in chunks of one
length and of two, fewer lines than a block holds.  FP64: 1e-11 of max|v|, the bar of the separate sweeps.
FP32: an evaluation of the map is accurate to about 8 ulp of max|v| and contracts, so k of them and the
right side stay within (k + 1) 8 ulp."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.fch import FchSolver as OracleFch  # noqa: E402
from oracle.solver import Problem  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

from _parity import ULP32, check_fp64  # noqa: E402

CASES = [(128, 3, 6, "fp32"), (1024, 5, 4, "fp32"), (2048, 2, 6, "fp32"), (333, 7, 6, "fp32"), (1000, 3, 2, "fp32"),
         (256, 5, 6, "fp64"), (777, 3, 4, "fp64"), (1024, 2, 2, "fp64")]


@pytest.mark.parametrize("n,lines,M,precision", CASES)
def test_fused_iteration_matches_oracle(n, lines, M, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Fch1D
    build.build_library()
    its, dt, eps = 8, 0.05, 0.18
    u0 = uniform_noise((lines, n), 0.3, seed=n, mean=-0.1).astype(np.float32).astype(np.float64)
    prob = Problem(nx=n, eps=eps, M=M, tol=1e-30, max_iter=its, bc="periodic")
    o = OracleFch(prob, 1.0)
    ref = u0
    with Fch1D(n, lines, bc="periodic", eps=eps, eta=1.0, quad_order=M, tol=1e-30, max_iter=its, precision=precision) as s:
        u = torch.tensor(u0, device="cuda").to(torch.float32 if precision == "fp32" else torch.float64)
        for _ in range(2):                       # the second step starts from the carried Lap v
            s.step(u, dt, raise_on_nonconvergence=False)
            ref, _ = o.step(ref, dt)
        launched = s.kernel_launches()
        got = u.double().cpu().numpy()
    assert launched < 2 * 14 * its, launched     # the separate sweeps take 14 and more an iteration
    scale = np.abs(ref + 1).max()
    if precision == "fp64":
        check_fp64(f"fused_fch1d_{n}x{lines}_M{M}_2steps_8it_fp64", got, ref, 1e-11 * scale)
    else:
        err = np.abs(got - ref).max()
        assert err <= 2 * (its + 1) * 8 * ULP32 * scale, (err, scale)
