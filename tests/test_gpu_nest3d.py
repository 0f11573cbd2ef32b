"""GPU: the 3D iteration in one nested pass per axis (``csrc/solver3d.cpp``) against the 3D oracle over a fixed
number of iterations, at the sizes where the cuts change: whole chunks and chunks of two lengths on every
axis, y and z columns over two blocks of a cluster, one value per register along x; and a line of 113 nodes, which
cannot be cut into chunks of 16 and 15 and keeps the separate sweeps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.split3d import Problem3D, Solver3D as Oracle3D  # noqa: E402
from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

from _parity import check_fp32  # noqa: E402

SHAPES = [(64, 64, 64, 4), (64, 57, 520, 4), (214, 520, 47, 6), (113, 45, 51, 2)]   # nx, ny, nz, M


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("nx,ny,nz,M", SHAPES)
def test_nested_3d_steps_match_oracle(nx, ny, nz, M, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Solver3D
    build.build_library()
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
    assert (launched < 15 * its) == (nx != 113), launched          # the sweeps alone would be more
    check_fp32(f"nested3d_{nx}x{ny}x{nz}_M{M}_{bc}_be_1step_4it", got, ref, np.abs(ref + 1).max())
