"""GPU: the stage loop of a single line in one block (``csrc/nest_line.cuh``) against the oracle over a fixed number
of iterations: every number of nodes per thread and the lines at their limits, chunks of one length and of two,
the shortest and the longest line, equal and different factors.  FP64: 1e-11 of max|v|.  FP32: k
evaluations of the map and the right side at 8 ulp of max|v| each."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.solver import OracleSolver, Problem, stage_params  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

from _parity import ULP32, check_fp64  # noqa: E402

CASES = [(32, 6), (77, 2), (256, 4), (1024, 6), (1025, 4), (2048, 2), (2049, 6), (4096, 4)]   # n, M


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("dt", [1e-4, 5e-3])
@pytest.mark.parametrize("n,M", CASES)
def test_line_loop_matches_oracle(n, M, dt, bc, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Solver
    build.build_library()
    its, eps = 5, 0.05
    sp = stage_params(dt, eps)
    assert (sp.c_in == sp.c_out) == (dt < 1e-3)
    u0 = uniform_noise((1, n), 0.05, seed=n, mean=0.1)
    if bc == "dirichlet":
        u0[:, 0] = u0[:, -1] = -1
    u0 = u0.astype(np.float32).astype(np.float64)
    prob = Problem(nx=n, ny=1, bc=bc, eps=eps, M=M, tol=1e-30, max_iter=its)
    ref, _ = OracleSolver(prob).step(u0, dt, "be")
    with Solver(nx=n, ny=1, bc=bc, eps=eps, quad_order=M, precision=precision, tol=1e-30, max_iter=its) as s:
        u = torch.tensor(u0, device="cuda").to(s.dtype)
        before = s.kernel_launches()
        s.step(u, dt, "be", raise_on_nonconvergence=False)
        launched = s.kernel_launches() - before
        got = u.double().cpu().numpy().reshape(ref.shape)
    assert launched < 3 * its, launched           # two sweeps and a check an iteration, separately
    scale = np.abs(ref + 1).max()
    if precision == "fp64":
        check_fp64(f"line_{n}_M{M}_{bc}_dt{dt:g}_be_5it_fp64", got, ref, 1e-11 * scale)
    else:
        err = np.abs(got - ref).max()
        assert err <= (its + 1) * 8 * ULP32 * scale, (err, scale)
