"""Two contexts on two host threads, each on its own stream, whose calls need
different amounts of shared memory of the same kernel (the batch size or the
scene decides): every call succeeds and returns what it returns alone.  One
captured graph that holds both sizes."""
import threading

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


def _scene(n_obs):
    rng = np.random.default_rng(7)
    return W.Obstacles(spheres=W._sphere_obstacles(rng, n_obs, (-2.0, -2.0, -1.0), (2.5, 2.0, 2.2), 0.02, 0.06),
                       aabbs=np.zeros((0, 6)))


def _calls(mcproj, name):
    """Two calls of one entry point, the second with more shared memory."""
    def dev(a):
        return torch.tensor(f32_exact(a), dtype=torch.float32, device="cuda")

    if name == "tree":       # warps per block
        wl = W.humanoid_workload(n=20000)
        wl.params.max_iters = 0   # the launches matter, not the steps
        out = []
        for n in (33, 20000):
            P, q = mcproj.Projector(wl.robot, wl.constraints), dev(wl.q[:, :n])
            out.append(lambda P=P, q=q, s=None: P.project(q, wl.params, stream=s))
        return out
    if name == "check":      # four lanes per configuration: 66 KB and the scene
        n = 16 * 32 * torch.cuda.get_device_properties(0).multi_processor_count // 8 + 1
        wl = W.humanoid_workload(n=n)
        out = []
        for k in (8, 1000):
            P, q = mcproj.Projector(wl.robot, wl.constraints, _scene(k)), dev(wl.q)
            out.append(lambda P=P, q=q, s=None: (P.check(q, stream=s),))
        return out
    if name == "fused":      # the dual arm's step keeps its Jacobian in shared memory
        wl = W.dual_arm_workload(total=10, n_random=2000)
        wl.params.max_iters = 0
        out = []
        for k in (8, 1000):
            P, q = mcproj.Projector(wl.robot, wl.constraints, _scene(k)), dev(wl.q)
            P.set_tuning(128, 4, 32, 1, 1)
            out.append(lambda P=P, q=q, s=None: P.project_check(q, wl.params, stream=s))
        return out
    wl = W.extend_workload(n_ext=1, n=8)   # extend: above 48 KB from 1,000 obstacles
    ex = wl.extra
    out = []
    for k in (1000, 1024):
        P = mcproj.Projector(wl.robot, wl.constraints, _scene(k))
        qs = P.project(dev(ex["raw_start"]), wl.params)[0]
        qt, ep = dev(ex["target"]), dev(ex["eps"])
        out.append(lambda P=P, qs=qs, qt=qt, ep=ep, s=None: P.extend(qs, qt, ep, wl.params, ex["r"], ex["delta"], stream=s))
    return out


class _Recorder:
    """The library, keeping the last call and its arguments."""

    def __init__(self, lib):
        self._lib = lib

    def __getattr__(self, name):
        fn = getattr(self._lib, name)

        def call(*args):
            if name != "mcp_last_error":
                self.last = (fn, args)
            return fn(*args)
        return call


@pytest.mark.parametrize("name", ["tree", "check", "fused", "extend"])
def test_two_threads(mcproj, name):
    rec = _Recorder(mcproj.load_library())
    plain = mcproj.Projector.__init__

    def init(self, *a, **k):
        plain(self, *a, lib=rec, **k)
    with pytest.MonkeyPatch.context() as mp:
        mp.setattr(mcproj.Projector, "__init__", init)
        calls = _calls(mcproj, name)
    streams = [torch.cuda.Stream() for _ in calls]
    outs, ref, raw = [], [], []
    for c, s in zip(calls, streams):
        outs.append(c(s=s))
        torch.cuda.synchronize()
        raw.append(rec.last)
        ref.append([t.clone() for t in outs[-1]])
    bad = [0, 0]
    go = threading.Barrier(2)

    def loop(k):
        fn, args = raw[k]
        go.wait()
        for i in range(8000):
            bad[k] += fn(*args) != mcproj.MCP_OK
            if i % 500 == 499:
                streams[k].synchronize()

    threads = [threading.Thread(target=loop, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert bad == [0, 0]
    for got, want in zip(outs, ref):
        for x, y in zip(got, want):
            assert torch.equal(x, y)


def test_one_graph_holds_both_sizes(mcproj):
    calls = _calls(mcproj, "tree")
    ref = [[t.clone() for t in c()] for c in calls]
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            outs = [c(s=s) for c in (calls[1], calls[0])]
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    for got, want in zip(outs, ref[::-1]):
        for x, y in zip(got, want):
            assert torch.equal(x, y)
