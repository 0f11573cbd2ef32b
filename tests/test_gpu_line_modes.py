"""GPU: single lines that one block steps (``csrc/nest_line.cuh``) under the host-driven loop and under profiling: the
host launches every iteration and reads its residual back, the profile names the kernels, and the fields
and iteration counts are those of the device-driven loop bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04214_gb300.inputs import uniform_noise  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bc,scheme", [("neumann", "be"), ("periodic", "sdc2"), ("dirichlet", "sdirk2")])
@pytest.mark.parametrize("n", [33, 256, 4096])
def test_line_host_loop_and_profile(n, bc, scheme, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_04214_gb300 import build
    from paper_1611_04214_gb300.molt import Solver
    build.build_library()
    u0 = uniform_noise((1, n), 0.05, seed=n, mean=0.1)
    if bc == "dirichlet":
        u0[:, 0] = u0[:, -1] = -1
    out = {}
    for mode in ("graph", "host_loop", "profile"):
        with Solver(nx=n, ny=1, bc=bc, eps=0.1, quad_order=4, precision=precision, tol=1e-9, max_iter=400) as s:
            s.set_execution("host_loop" if mode == "host_loop" else "graph")
            s.profile_enable(mode == "profile")
            u = torch.tensor(u0, device="cuda").to(s.dtype)
            before = s.kernel_launches()
            info = [s.step(u, 2e-3, scheme) for _ in range(2)]
            out[mode] = (u.cpu().numpy(), [i.iters for i in info], [i.residual for i in info], s.kernel_launches() - before,
                         s.profile_collect())
    iters = sum(sum(i) for i in out["graph"][1])
    for mode in ("host_loop", "profile"):
        assert np.array_equal(out[mode][0], out["graph"][0]), mode
        assert out[mode][1:3] == out["graph"][1:3], mode
        assert out[mode][3] >= iters, mode                       # a launch an iteration
    assert out["graph"][3] < iters
    stages = sum(len(i) for i in out["graph"][1])
    kernels = out["profile"][4]
    assert kernels["line"][1] == iters and kernels["line_rhs"][1] == stages, kernels
    assert kernels["line"][0] > 0.0
