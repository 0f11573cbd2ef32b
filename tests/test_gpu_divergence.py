"""GPU: an iteration that overflows ends as not converged, on every path (the cubic of an overflowing field turns a whole
line into NaN within one iteration, so that no finite or infinite value is left beside it and the residual over
numbers is zero); independent lines go on beside one that has overflowed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402

NOT_CONVERGED = -2
BIG = 40.0     # |u| far outside the wells: the lagged cubic grows without bound


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    build.build_library()


def _field(shape, precision, seed=3):
    rows = int(np.prod(shape[:-1]))
    u = BIG * uniform_noise((rows, shape[-1]), 1.0, seed=seed).reshape(shape)
    return torch.tensor(u, device="cuda").to(torch.float32 if precision == "fp32" else torch.float64)


def _check(info, *fields):
    assert not all(torch.isfinite(f).all().item() for f in fields)      # (it did overflow)
    assert info.status == NOT_CONVERGED, (info.status, info.iters, info.residual)


# lines in one block and by sweeps; grids in nested passes and by sweeps
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("mode", ["graph", "host_loop"])
@pytest.mark.parametrize("nx,ny,bc,dt", [(256, 1, "periodic", 1e-3), (4096, 1, "dirichlet", 1e-3), (5000, 1, "neumann", 1e-3),
                                         (256, 264, "neumann", 1e-3), (96, 72, "periodic", 1e-3),
                                         (1024, 40, "neumann", 0.02)])
def test_diverged_steps_are_reported(nx, ny, bc, dt, mode, precision):
    from paper_1611_04214_gb300.molt import Solver
    with Solver(nx=nx, ny=ny, bc=bc, eps=0.1, quad_order=4, precision=precision, tol=1e-6, max_iter=60) as s:
        s.set_execution(mode)
        u = _field((ny, nx), precision)
        _check(s.step(u, dt, "be", raise_on_nonconvergence=False), u)


@pytest.mark.parametrize("nx,ny", [(256, 264), (96, 72), (1024, 40), (300, 1)])
def test_diverged_vector_steps_are_reported(nx, ny):
    from paper_1611_04214_gb300.molt import Solver
    with Solver(nx=nx, ny=ny, bc="neumann", eps=0.32, quad_order=4, precision="fp32", tol=1e-6, max_iter=60) as s:
        u1, u2 = _field((ny, nx), "fp32", 1), _field((ny, nx), "fp32", 2)
        _check(s.vch_step(u1, u2, 5e-4, "be", raise_on_nonconvergence=False), u1, u2)


def test_diverged_instances_of_a_batch_are_reported():
    from paper_1611_04214_gb300.molt import Batch
    inst = [(40, 56, 2.0, 2.0, 0.1), (96, 72, 3.0, 2.0, 0.06)]
    with Batch(inst, bc="neumann", quad_order=4, tol=1e-6, max_iter=200) as b:
        parts = [0.01 * uniform_noise((56, 40), 1.0, seed=1), BIG * uniform_noise((72, 96), 1.0, seed=2)]
        u = torch.tensor(b.pack([p.astype(np.float32) for p in parts]), device="cuda")
        info = b.step(u, [1e-4, 1e-3], "be", raise_on_nonconvergence=False)
    assert info.instance_status == [0, NOT_CONVERGED], info


@pytest.mark.parametrize("shape", [(64, 64, 64), (45, 51, 113)])
def test_diverged_3d_steps_are_reported(shape):
    from paper_1611_04214_gb300.molt import Solver3D
    nz, ny, nx = shape
    with Solver3D(nx, ny, nz, bc="periodic", eps=0.1, quad_order=4, tol=1e-6, max_iter=60) as s:
        u = _field(shape, "fp32")
        _check(s.step(u, 1e-3, "be", raise_on_nonconvergence=False), u)


# one line of several diverges while the others converge
@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_diverged_sixth_order_lines_are_reported(bc, precision):
    from paper_1611_04214_gb300.molt import Fch1D
    with Fch1D(512, 5, bc=bc, eps=0.18, quad_order=4, tol=1e-5, max_iter=400, precision=precision) as s:
        u = torch.full((5, 512), -1.0, device="cuda", dtype=torch.float32 if precision == "fp32" else torch.float64)
        u[2] = _field((1, 512), precision)[0]
        _check(s.step(u, 0.05, raise_on_nonconvergence=False), u)


# ... and finish their iterations as they do without it
@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_lines_go_on_beside_a_diverged_one(bc, precision):
    from paper_1611_04214_gb300.molt import Fch1D
    x = torch.linspace(0, 2 * np.pi, 512, dtype=torch.float64)
    rows = torch.stack([-1 + 0.01 * (k + 1) * torch.cos(x) for k in range(5)])
    out = []
    for bad in (False, True):
        with Fch1D(512, 5, bc=bc, eps=0.18, quad_order=4, tol=1e-30, max_iter=25, precision=precision) as s:
            u = rows.to(torch.float32 if precision == "fp32" else torch.float64).cuda()
            if bad:
                u[2] = _field((1, 512), precision)[0]
            info = s.step(u, 0.05, raise_on_nonconvergence=False)
            out.append((u.cpu(), info.iters))
    assert not torch.isfinite(out[1][0][2]).any() and out[0][1] == out[1][1] == [25]
    keep = [0, 1, 3, 4]
    assert torch.equal(out[0][0][keep], out[1][0][keep])


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_diverged_2d_sixth_order_steps_are_reported(bc, precision):
    from paper_1611_04214_gb300.molt import Fch2D
    with Fch2D(128, 96, bc=bc, eps=0.18, quad_order=4, tol=1e-5, max_iter=400, precision=precision) as s:
        u = _field((96, 128), precision)
        _check(s.step(u, 0.05, raise_on_nonconvergence=False), u)


# a candidate that overflows is rejected, and the step size falls until one does not
@pytest.mark.parametrize("estimator", ["richardson", "sdc2", "bdf2"])
def test_adaptive_step_rejects_an_overflowing_candidate(estimator):
    from paper_1611_04214_gb300.molt import Solver
    with Solver(nx=256, ny=1, bc="periodic", eps=0.1, quad_order=4, precision="fp64", tol=1e-6, max_iter=60) as s:
        u = _field((1, 256), "fp64")
        out = s.step_adaptive(u, 1e-3, 1e3, 1e-14, 1e-3, gamma=2.0, estimator=estimator)
    assert torch.isfinite(u).all() and out["rejections"] > 0 and np.isfinite(out["eta"]), out


@pytest.mark.parametrize("estimator", ["richardson", "bdf2"])
def test_adaptive_vector_step_rejects_an_overflowing_candidate(estimator):
    from paper_1611_04214_gb300.molt import Solver
    with Solver(nx=256, ny=1, bc="neumann", eps=0.32, quad_order=4, precision="fp64", tol=1e-6, max_iter=60) as s:
        u1, u2 = _field((1, 256), "fp64", 1) / 4, _field((1, 256), "fp64", 2) / 4
        out = s.vch_step_adaptive(u1, u2, 5e-4, 1e3, 1e-16, 5e-4, gamma=2.0, estimator=estimator)
    assert torch.isfinite(u1).all() and torch.isfinite(u2).all()
    assert out["rejections"] > 0 and np.isfinite(out["eta"]), out
