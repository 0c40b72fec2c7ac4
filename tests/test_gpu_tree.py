"""The humanoid's tree kernel (one lane per configuration) where its launch
shape changes: one warp, one warp per SM, two warps per block, full blocks
with and without refill.  A configuration's result depends on nothing else in
its launch, so pieces of a large batch projected on their own return the same
bits, and the outputs are valid points of the manifold."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc  # noqa: E402
from paper_2604_13323_gb300 import workloads as W  # noqa: E402
from tests.gpu_util import f32_exact  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mcproj():
    from paper_2604_13323_gb300 import build, mcproj as m
    build.build()
    m.load_library()
    return m


@pytest.mark.parametrize("hull", [False, True])
@pytest.mark.parametrize("per_sm", [0, 1, 2, 7, 15])
def test_launch_shapes_agree(mcproj, per_sm, hull):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = max(33, 32 * sms * per_sm + 1)   # per_sm warps on every SM and one configuration more
    wl = W.humanoid_workload(n=n, hull=hull)
    q0 = f32_exact(wl.q)
    P = mcproj.Projector(wl.robot, wl.constraints)
    q = torch.tensor(q0, dtype=torch.float32, device="cuda")
    big = P.project(q, wl.params)
    for lo, hi in ((0, 1), (0, 31), (n - 33, n)):
        part = P.project(q[:, lo:hi].contiguous(), wl.params)
        for a, b in zip(part, big):
            assert torch.equal(a, b[..., lo:hi])
    fl, rs = big[1].cpu().numpy(), big[3].cpu().numpy()
    conv = (fl & mcproj.F_CONVERGED) != 0
    assert conv.mean() > 0.99
    assert (rs[conv] < wl.params.tol).all()
    O = orc.Oracle(wl.robot, wl.constraints)
    qg = big[0].double().cpu().numpy()
    for i in range(0, n, max(1, n // 64)):   # the reported residual is the FP64 residual of the output
        r = np.linalg.norm(O.residual(qg[:, i]))
        assert abs(r - rs[i]) <= 1e-12 * max(1.0, r)
