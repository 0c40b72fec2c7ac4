"""The FP64 residual of the acceptance (structure-aware FK, split sin / cos,
off-diagonal error rotations) where its branches change: at the start itself
(no step taken), from the manifold to far from it, angles on both sides of the
split table's range, a TSR offset that is not the identity, links with and
without CoM offsets.  The oracle evaluates the same configurations in FP64;
both round O(1) intermediates (1e-15 per operation at most, a few hundred of
them in a chain), so they agree to 1e-12 of max(1, residual)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc  # noqa: E402
from paper_2604_13323_gb300 import workloads as W  # noqa: E402
from tests.gpu_util import f32_exact  # noqa: E402

pytestmark = pytest.mark.gpu


def _workload(name):
    n = 192
    if name in ("tray", "peg", "tsr"):
        return W.arm_task_workload(name, n=n)
    if name == "arm":
        return W.arm_workload(n=n)
    if name == "dual":
        return W.dual_arm_workload(total=10, n_random=n)
    if name == "rod":
        return W.dual_rod_workload(n=n)
    wl = W.humanoid_workload(n=n, hull=name == "hull")
    if name == "offset":   # TSR offsets, a dense CoM offset on the head, none elsewhere on the neck
        Q = W._rt(W.random_rotation(np.random.default_rng(3)), (0.02, -0.01, 0.03))
        for c in wl.constraints[:2]:
            c.Q = Q
        wl.robot.com[wl.extra["names"].index("head")] = (0.01, 0.02, -0.03)
        wl.robot.com[wl.extra["names"].index("neck_yaw")] = 0.0
    return wl


@pytest.mark.parametrize("name", ["arm", "tray", "peg", "tsr", "dual", "rod", "humanoid", "hull", "offset"])
@pytest.mark.parametrize("iters", [0, 2, 30])
def test_reported_residual_is_the_oracles(name, iters):
    from paper_2604_13323_gb300 import build, mcproj
    build.build()
    wl = _workload(name)
    q0 = f32_exact(wl.q)
    q0[:, :32] *= np.linspace(0.5, 6.0, 32)[None, :].astype(np.float32)   # past the table's +-4 rad
    q0 = f32_exact(q0)
    P = mcproj.Projector(wl.robot, wl.constraints)
    p = W.Params(tol=wl.params.tol, max_iters=iters, lam=wl.params.lam)
    out, fl, it, rs = P.project(torch.tensor(q0, dtype=torch.float32, device="cuda"), p)
    torch.cuda.synchronize()
    out, rs = out.double().cpu().numpy(), rs.cpu().numpy()
    O = orc.Oracle(wl.robot, wl.constraints)
    for i in range(out.shape[1]):
        r = np.linalg.norm(O.residual(out[:, i]))
        assert abs(r - rs[i]) <= 1e-12 * max(1.0, r, np.abs(out[:, i]).max()), (i, r, rs[i])
