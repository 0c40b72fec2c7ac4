"""Path length, gradient and step for the joint numbers that have a compiled
kernel (7, 14) and for another (36), at the edges of a warp's 32 segments."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2604_13323_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
U = 2.0 ** -24   # FP32 unit roundoff


def _robot(d):
    return {7: lambda: W.arm_workload(n=1), 14: lambda: W.dual_arm_workload(total=10),
            36: lambda: W.humanoid_workload(n=1)}[d]()


@pytest.mark.parametrize("d", [7, 14, 36])
@pytest.mark.parametrize("n_paths,n_way", [(1, 2), (3, 32), (5, 33), (2, 34), (131, 65)])
def test_path_kernels_match_fp64(d, n_paths, n_way):
    from paper_2604_13323_gb300 import build, mcproj
    build.build()
    wl = _robot(d)
    P = mcproj.Projector(wl.robot, wl.constraints)
    rng = np.random.default_rng(1000 * d + n_way)
    Q = rng.uniform(-2, 2, (d, n_paths * n_way)).astype(np.float32)
    if n_way > 3:
        Q[:, 2] = Q[:, 1]   # a segment of no length
    L, G = P.path_length_grad(torch.tensor(Q, device="cuda"), n_paths, n_way)
    X = Q.astype(np.float64).reshape(d, n_paths, n_way)
    E = np.diff(X, axis=2)
    n = np.linalg.norm(E, axis=0)
    unit = E / np.where(n > 0, n, 1)
    ref = np.zeros_like(X)
    ref[:, :, 1:] += unit
    ref[:, :, :-1] -= unit
    # a unit vector's component: difference 1, norm^2 (d + 1) / 2, rsqrt 4,
    # product 1 roundings; two of them and their difference (at most 2)
    assert np.abs(G.cpu().numpy().reshape(ref.shape) - ref).max() <= (d + 15) * U
    # a norm: 1 + (d + 1) / 2 + 1 roundings; a lane's sum and the warp's five
    Lref = n.sum(axis=1)
    assert (np.abs(L.cpu().numpy() - Lref) <= (d / 2 + 9 + n_way / 32) * U * Lref).all()
    D = rng.standard_normal(Q.shape).astype(np.float32)
    for eta, cap in ((0.1, 0.0), (0.1, 0.05)):
        Y = torch.tensor(Q, device="cuda")
        P.path_step(Y, torch.tensor(D, device="cuda"), n_paths, n_way, eta, cap)
        s = float(np.float32(eta)) * D.astype(np.float64).reshape(X.shape)
        if cap:
            m = np.abs(s).max(axis=0)
            s = s * np.where(m > cap, float(np.float32(cap)) / m, 1.0)
        s[:, :, [0, -1]] = 0
        want = X - s
        # the step: eta g, its maximum, the quotient, scale and product 5 roundings; the sum 1
        got = Y.cpu().numpy().reshape(X.shape)
        assert (np.abs(got - want) <= 5 * U * np.abs(s) + U * np.abs(want) + 1e-12).all()
        assert np.array_equal(got[:, :, [0, -1]], Q.reshape(X.shape)[:, :, [0, -1]])
