"""GPU: the 2D sixth-order iteration in nested passes (``csrc/fch2d.cpp``) against the oracle over a fixed number of
iterations and two steps (W carried): rows packed within a warp and over a block and one value per register,
columns of whole chunks, of two lengths, and over two blocks of a cluster.  FP64: 1e-11 of max|v|.  FP32:
the fields of the y pass are up to 9 max|v|, so one evaluation is accurate to about 9 times 8 ulp of it, and
k of them and the right side, in two steps, stay within 2 (k + 1) 72 ulp."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.fch import Fch2DSolver as Oracle2D  # noqa: E402
from oracle.solver import Problem  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

from _parity import ULP32, check_fp64  # noqa: E402

CASES = [(256, 64, 6), (777, 130, 4), (64, 520, 2), (2048, 45, 6), (300, 77, 2)]   # nx, ny, M


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny,M", CASES)
def test_nested_sixth_order_steps_match_oracle(nx, ny, M, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Fch2D
    build.build_library()
    its, dt, eps = 6, 0.05, 0.18
    L = dict(Lx=2 * np.pi, Ly=2 * np.pi * ny / nx)
    u0 = uniform_noise((ny, nx), 0.3, seed=nx, mean=-0.1).astype(np.float32).astype(np.float64)
    prob = Problem(nx=nx, ny=ny, bc="periodic", eps=eps, M=M, tol=1e-30, max_iter=its, **L)
    o = Oracle2D(prob, 1.0)
    ref = u0
    with Fch2D(nx, ny, bc="periodic", eps=eps, eta=1.0, quad_order=M, tol=1e-30, max_iter=its, precision=precision, **L) as s:
        u = torch.tensor(u0, device="cuda").to(torch.float32 if precision == "fp32" else torch.float64)
        for _ in range(2):
            s.step(u, dt, raise_on_nonconvergence=False)
            ref, _ = o.step(ref, dt)
        launched = s.kernel_launches()
        got = u.double().cpu().numpy()
    assert launched < 2 * 14 * its, launched     # the sweeps alone would be more
    scale = np.abs(ref + 1).max()
    if precision == "fp64":
        check_fp64(f"nested_fch2d_{nx}x{ny}_M{M}_2steps_6it_fp64", got, ref, 1e-11 * scale)
    else:
        err = np.abs(got - ref).max()
        assert err <= 2 * (its + 1) * 72 * ULP32 * scale, (err, scale)
