"""The collision check on both sides of the sizes where its number of lanes per
configuration changes (8 to 4 at 16 warps on an SM, 4 to 1 at 20): the verdicts
of the one-lane kernel, which a call that asks for the number of tests takes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2604_13323_gb300 import workloads as W  # noqa: E402
from tests.gpu_util import f32_exact  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["arm", "rod", "dual", "humanoid"])
@pytest.mark.parametrize("n_obs", [33, 1024])
def test_verdicts_at_the_lines(name, n_obs):
    from paper_2604_13323_gb300 import build, mcproj
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lines = (12 * 32 * sms // 8, 16 * 32 * sms // 8, 20 * 32 * sms // 4)
    n_max = lines[-1] + 1
    wl = {"arm": lambda: W.arm_workload(n=n_max), "rod": lambda: W.dual_rod_workload(n=n_max),
          "dual": lambda: W.dual_arm_workload(total=10, n_random=n_max), "humanoid": lambda: W.humanoid_workload(n=n_max)}[name]()
    rng = np.random.default_rng(5)
    P = mcproj.Projector(wl.robot, wl.constraints, W.Obstacles(
        spheres=W._sphere_obstacles(rng, n_obs, (-2.0, -2.0, -1.0), (2.5, 2.0, 2.2), 0.005, 0.02), aabbs=np.zeros((0, 6))))
    q = torch.tensor(f32_exact(wl.q), dtype=torch.float32, device="cuda")
    one = P.check(q, pairs=torch.zeros(n_max, dtype=torch.int32, device="cuda"))
    assert n_obs < 100 or 0.0 < one.float().mean().item() < 1.0   # (few of the small scene's are hit)
    for n in lines:
        for k in (n, n + 1):
            assert torch.equal(P.check(q[:, :k].contiguous()), one[:k]), k
