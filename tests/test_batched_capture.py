"""spin_invert_batched while the caller captures its stream: what a captured
call does is done when the graph is replayed, so it may not change what the
library takes for done."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spin():
    import paper_1801_04723_gb300 as s

    s.build()
    s.lib()
    return s


def batch(seed, orders=(48, 96, 96, 160)):
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    out = []
    for n in orders:
        A = torch.rand((n, n), generator=g, dtype=torch.float64, device="cuda:0").mul_(2.0).sub_(1.0)
        A.diagonal().add_(float(n))
        out.append(A)
    return out


def inverses(As):
    return [torch.linalg.inv(a) for a in As]


def close(Xs, refs):
    return all(torch.allclose(x, r, rtol=1e-9, atol=1e-14) for x, r in zip(Xs, refs))


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
def test_refused_capture_leaves_no_trace(spin, mode):
    """Other matrices of the plan's orders under capture: the call is refused,
    and the next direct call with them inverts them."""
    first, other = batch(1), batch(2)
    x1, x2 = [torch.zeros_like(a) for a in first], [torch.zeros_like(a) for a in other]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        spin.invert_batched(first, outs=x1)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with pytest.raises(Exception):
        with torch.cuda.graph(graph, stream=s, capture_error_mode=mode):
            spin.invert_batched(other, outs=x2, blocking=False)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        _, status = spin.invert_batched(other, outs=x2)
    torch.cuda.synchronize()
    assert status.tolist() == [0] * len(other)
    assert close(x2, inverses(other)) and close(x1, inverses(first))
