"""Inner products of double doubles over long spreads (7 and 8 pieces): three CTAs an SM,
so that 400 products take the time of 300."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def microseconds(f, n=20):
    """A call's time, n of them replayed from a graph (the host's calls left out)."""
    f()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(n):
            f()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    out = []
    for _ in range(9):
        a.record()
        graph.replay()
        b.record()
        b.synchronize()
        out.append(a.elapsed_time(b) / n * 1e3)
    return sorted(out)[4]


@pytest.mark.parametrize("spread,S", [(28, 7), (36, 8)])
def test_three_an_sm(mw, cuda, spread, S):
    nsm = torch.cuda.get_device_properties(cuda).multi_processor_count
    g = torch.Generator(device=cuda)
    g.manual_seed(5)

    def sym(shape):
        return torch.rand(shape, dtype=torch.float64, device=cuda, generator=g) * 2 - 1

    def vectors():
        X = torch.empty((2, 3 * nsm - 8, 200), dtype=torch.float64, device=cuda)
        X[0] = torch.exp2(sym(X.shape[1:]) * spread)
        X[0, :, 0], X[0, :, 1] = 2.0 ** spread, 2.0 ** -spread
        X[1] = X[0] * sym(X.shape[1:]) * 2.0 ** -54
        return X
    A, B = vectors(), vectors()
    plan = mw.plan_dot(A, B)
    assert plan.S_A == S

    def time(count):
        C = torch.empty((2, count), dtype=torch.float64, device=cuda)
        return microseconds(lambda: mw.mw_dot_batched(A[:, :count], B[:, :count], plan, C=C, check=False))
    two, three = time(2 * nsm - 8), time(3 * nsm - 8)
    # one entry a thread: a CTA's time is latency, so a second round of CTAs takes near
    # twice the time of one and a fuller first round hardly more
    assert three <= 1.4 * two
