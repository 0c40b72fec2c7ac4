"""Segment offsets: uneven segments whose numbers lie at the edges of the
scan's tiles (4,096 lengths), with empty ones among them, give the points of
the same segments projected as a plain batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2604_13323_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_seg", [1, 31, 33, 1024, 4095, 4096, 4097, 9001])
def test_segment_points_are_the_batchs(n_seg):
    from paper_2604_13323_gb300 import build, mcproj
    build.build()
    wl = W.sphere_workload(n_pairs=1)
    rng = np.random.default_rng(n_seg)
    length = rng.integers(0, 4, n_seg).astype(np.int32)
    length[-1] = 2
    start = rng.standard_normal((3, n_seg))
    delta = 0.05 * rng.standard_normal((3, n_seg))
    P = mcproj.Projector(wl.robot, wl.constraints)
    st, de = (torch.tensor(x, device="cuda") for x in (start, delta))
    ln = torch.tensor(length, device="cuda")
    seg = np.repeat(np.arange(n_seg), length)
    t = np.arange(length.sum()) - np.repeat(np.cumsum(length) - length, length)
    # the library rounds start + t * delta once, the batch twice
    si = torch.tensor(seg, device="cuda")
    pts = st[:, si] + torch.tensor(t, device="cuda") * de[:, si]
    ref = P.project(pts, wl.params)
    for rep in range(3):   # launched directly, then captured, then replayed
        got = P.project_segments(st, de, ln, wl.params)
        torch.cuda.synchronize()
        assert torch.equal(got[1], ref[1])
        # a rounding of a coordinate of size 4, projected
        assert (got[0] - ref[0]).abs().max().item() <= 1e-14
