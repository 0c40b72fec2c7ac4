"""When the segment projection uses its captured graph, and that the graph does
what the direct launches do: a call that comes twice in a row (the same
outputs, inputs, parameters) is captured, and replayed while it repeats or
comes back; other calls are launched directly.  A context created with
MCP_TEST_FAIL_CUDA="graph launch" reports an error exactly where the graph is
used (after it has run)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2604_13323_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mcproj():
    from paper_2604_13323_gb300 import build, mcproj as m
    build.build()
    m.load_library()
    return m


def _case(n_seg):
    wl = W.sphere_workload(n_pairs=1)
    rng = np.random.default_rng(n_seg)
    length = rng.integers(0, 4, n_seg).astype(np.int32)
    length[-1] = 2
    x = [torch.tensor(a, device="cuda") for a in
         (rng.standard_normal((3, n_seg)), 0.05 * rng.standard_normal((3, n_seg)), length)]
    return wl, x, int(length.sum())


def _outputs(total):
    return dict(out=torch.empty((3, total), dtype=torch.float64, device="cuda"),
                flags=torch.empty(total, dtype=torch.uint8, device="cuda"),
                iters=torch.empty(total, dtype=torch.uint8, device="cuda"),
                resid=torch.empty(total, dtype=torch.float64, device="cuda"))


def _fill(o):
    o["out"].fill_(7.0)
    o["resid"].fill_(7.0)
    o["flags"].fill_(128)
    o["iters"].fill_(255)


@pytest.mark.parametrize("n_seg", [1, 33, 4095, 4096, 4097, 9001])
def test_captured_and_replayed_calls_write_what_the_direct_one_does(mcproj, n_seg):
    wl, (st, de, ln), total = _case(n_seg)
    P = mcproj.Projector(wl.robot, wl.constraints)
    o = _outputs(total)
    for rep in range(5):   # direct, captured, replayed; then replayed on new contents
        if rep == 3:
            st.mul_(1.25)
            de.neg_()
            ln.copy_(ln.flip(0))
        fresh = mcproj.Projector(wl.robot, wl.constraints).project_segments(st, de, ln, wl.params, total=total)
        _fill(o)
        got = P.project_segments(st, de, ln, wl.params, total=total, **o)
        torch.cuda.synchronize()
        for a, b in zip(got, fresh):
            assert torch.equal(a, b), rep


def test_which_calls_use_the_graph(mcproj, monkeypatch):
    wl, (st, de, ln), total = _case(33)
    monkeypatch.setenv("MCP_TEST_FAIL_CUDA", "graph launch")
    P = mcproj.Projector(wl.robot, wl.constraints)
    monkeypatch.delenv("MCP_TEST_FAIL_CUDA")
    A, B = _outputs(total), _outputs(total)

    def graph(o):
        try:
            P.project_segments(st, de, ln, wl.params, total=total, **o)
        except mcproj.MCPError as e:
            assert e.status == mcproj.MCP_ERR_CUDA
            return True
        return False

    #       first; again; other; back (the graph is A's); again; other twice; back (the graph is B's now)
    calls = [A, A, B, A, A, B, B, A, B]
    want = [False, True, False, True, True, False, True, False, True]
    assert [graph(o) for o in calls] == want
    # alternating calls never capture; a load in between starts over
    Q = [_outputs(total) for _ in range(2)]
    assert [graph(Q[i % 2]) for i in range(4)] == [False] * 4
    assert [graph(A), graph(A)] == [False, True]
    P.load_constraints(wl.constraints)
    assert [graph(A), graph(A)] == [False, True]
