"""The dual arm's step out of registers (at most 12 warps on an SM) and out of
shared memory (more): the same bits on both sides of the rule's line, as a
batch, with the fused check, and on segments, with configurations that are not
finite, that leave by MaxDistance or the cap, or that need the FP64 re-solve."""
import dataclasses

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


def _line():
    return 12 * 32 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("kw", [{}, {"max_step": 0.7}, {"max_iters": 3}, {"pivot_fp64": 3e-4}, {"lam": 0.0},
                                {"alpha": 0.5, "max_iters": 60}, {"tol": 2e-7}])
@pytest.mark.parametrize("fused", [0, 1])
def test_batches_agree(mcproj, kw, fused):
    n = _line()
    wl = W.dual_arm_workload(total=10, n_random=n + 1)
    p = dataclasses.replace(wl.params, **kw)
    q = torch.tensor(f32_exact(wl.q), dtype=torch.float32, device="cuda")
    q[2, 5], q[9, 40], q[13, n - 1] = float("nan"), float("inf"), 1e30
    P = mcproj.Projector(wl.robot, wl.constraints, wl.obstacles)
    for tpb in (64, 128, 256):
        P.set_tuning(tpb, 8 if tpb < 256 else 4, 32, fused, 1)
        many = P.project_check(q, p)                                # shared memory
        few = [P.project_check(q[:, :m].contiguous(), p) for m in (1, 33, n)]   # registers
        for r in few:
            for x, y in zip(r, many):
                assert torch.equal(x.nan_to_num(7.0), y[..., :x.shape[-1]].nan_to_num(7.0)), (tpb, x.shape)
        P.set_tuning(tpb, 1, 32, fused, 1)                          # few warps: registers, with refill
        for x, y in zip(P.project_check(q, p), many):
            assert torch.equal(x.nan_to_num(7.0), y.nan_to_num(7.0)), tpb


def test_segments_agree(mcproj):
    n = _line()
    wl = W.dual_arm_workload(total=n + 200)
    ex = wl.extra
    P = mcproj.Projector(wl.robot, wl.constraints)
    starts = P.project(torch.tensor(ex["raw_start"], dtype=torch.float32, device="cuda"), wl.params)[0]
    delta = torch.tensor(ex["raw_dir"] * ex["step"], dtype=torch.float32, device="cuda")
    length = torch.tensor(ex["lengths"], dtype=torch.int32, device="cuda")
    total = int(ex["lengths"].sum())
    assert total > n
    keep = int(np.searchsorted(np.cumsum(ex["lengths"]), n, side="right"))   # whole segments within the line
    m = int(ex["lengths"][:keep].sum())
    many = P.project_segments(starts, delta, length, wl.params, total=total)
    few = P.project_segments(starts[:, :keep].contiguous(), delta[:, :keep].contiguous(), length[:keep].contiguous(),
                             wl.params, total=m)
    for x, y in zip(few, many):
        assert torch.equal(x, y[..., :m])
