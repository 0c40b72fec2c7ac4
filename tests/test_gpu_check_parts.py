"""The collision check with 8 or 4 lanes per configuration (batches that leave
the SMs idle) against the one-lane kernel, which a call that asks for the
number of tests takes: the same verdicts at the sizes where the rule changes,
for ragged batches, link counts below and above the lanes, scenes with and
without chunks and boxes, and spheres fixed to the world."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2604_13323_gb300 import workloads as W  # noqa: E402
from tests.gpu_util import f32_exact  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mcproj():
    from paper_2604_13323_gb300 import build, mcproj as m
    build.build()
    m.load_library()
    return m


@pytest.mark.parametrize("name", ["arm", "dual", "humanoid"])
@pytest.mark.parametrize("n_obs,n_box", [(0, 2), (1, 0), (33, 1), (200, 6)])
def test_parts_return_the_one_lane_verdicts(mcproj, name, n_obs, n_box):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    room = 8 * 32 * sms
    sizes = (1, 15, 17, 257, room // 8, room // 8 + 1, room // 4, room // 4 + 1)
    n_max = max(sizes)
    wl = {"arm": lambda: W.arm_workload(n=n_max), "dual": lambda: W.dual_arm_workload(total=10, n_random=n_max),
          "humanoid": lambda: W.humanoid_workload(n=n_max)}[name]()
    rng = np.random.default_rng(5)
    lo = rng.uniform((0.3, -1.0, 0.0), (1.0, 0.7, 1.2), size=(n_box, 3))
    obst = W.Obstacles(spheres=W._sphere_obstacles(rng, n_obs, (-0.5, -1.5, 0.0), (2.0, 1.5, 2.0), 0.05, 0.15),
                       aabbs=np.concatenate([lo, lo + rng.uniform(0.05, 0.4, size=(n_box, 3))], axis=1))
    rb = wl.robot   # two spheres fixed to the world, one link without spheres
    rb.sphere_link[rb.sphere_link == rb.sphere_link[0]] = -1
    rb.sphere[rb.sphere_link == -1, :3] += (-3.0, 0.0, 0.0)
    P = mcproj.Projector(rb, wl.constraints, obst)
    q = torch.tensor(f32_exact(wl.q), dtype=torch.float32, device="cuda")
    for n in sizes:
        qn = q[:, :n].contiguous()
        one = P.check(qn, pairs=torch.zeros(n, dtype=torch.int32, device="cuda"))
        assert torch.equal(P.check(qn), one), n
        if n_obs >= 33 and n >= 257:
            assert one.float().mean().item() > 0.0
