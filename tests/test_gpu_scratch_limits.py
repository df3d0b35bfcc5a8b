"""Calls whose fast way's scratch does not fit the GPU's free memory take the
plain way: parallel gradient segments the walk in turn, a product model's
scalars the step-by-step kernels.  Direct calls, a graph replay and the
caller's own capture, with all but a part of the memory taken by another
allocation.  The results agree with those of the fast way within the
gradient's 1e-3 |g| + 1e-4 max|g|; the log-likelihood does not depend on the
way."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32, PROD = 1, 2, 3
MB = 1 << 20


def exposures(gp):
    # 12 series of 60000 exposures, states of 5: 5760 chunks of 250 events.
    # Needed beside the event stream: about 180 MB; parallel segments: 160 MB more
    rng = np.random.default_rng(8)
    n, s = 60000, 12
    t = np.concatenate([np.cumsum(rng.exponential(1.0, n)) for _ in range(s)])
    dur = rng.uniform(0.05, 0.5, n * s) * np.minimum(np.diff(t, append=t[-1] + 1) % 1e3, 1.0)
    y = rng.standard_normal(n * s).astype(np.float32)
    off = np.arange(s + 1) * n
    theta = np.array([[1.0, 0.63, 3.0, 0.5, 5.0, 0.1]] * s) * np.linspace(1, 1.1, s)[:, None]
    return (lambda **kw: gp.Model((SHO, M32), off, t, t + dur, y, np.full(n * s, 0.1, np.float32),
                                  **kw)), theta


def instants(gp):
    # 12 series of 60000 instants: the scalars with their tangents take 104 MB
    rng = np.random.default_rng(9)
    n, s = 60000, 12
    t = np.concatenate([np.cumsum(rng.exponential(1.0, n)) for _ in range(s)])
    y = rng.standard_normal(n * s).astype(np.float32)
    off = np.arange(s + 1) * n
    theta = np.array([[1.0, 0.13, 1.0, 1.26, 10.0, 0.5, 5.0, 0.1]] * s)
    theta *= np.linspace(1, 1.1, s)[:, None]
    return (lambda **kw: gp.Model((PROD, M32), off, t, t, y, np.full(n * s, 0.1, np.float32),
                                  **kw)), theta


class Filled:
    """All of the GPU's free memory but ``leave`` bytes taken."""

    def __init__(self, gp, leave):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        # graphs that ended keep their memory for later ones until asked for it
        ctypes.CDLL(gp.LIB_PATH).cudaDeviceGraphMemTrim(0)
        free = torch.cuda.mem_get_info()[0]
        self.t = torch.empty(max(free - leave, 0), dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *a):
        del self.t
        torch.cuda.empty_cache()


def captured(m, theta):
    ll = torch.empty(theta.shape[0], dtype=torch.float64, device="cuda")
    g = torch.empty(theta.shape, dtype=torch.float32, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        m.loglik_grad(theta, out=ll, grad=g)
    graph.replay()
    torch.cuda.synchronize()
    return ll, g


@pytest.mark.parametrize("make,leave,fast", [(exposures, 2048, True), (exposures, 200, False),
                                             (instants, 2048, True), (instants, 96, False)])
@pytest.mark.parametrize("how", ["direct", "graph", "capture"])
def test_plain_way_where_memory_is_short(make, leave, fast, how):
    import paper_2601_02527_gb300 as gp
    build, th = make(gp)
    theta = torch.tensor(th, dtype=torch.float32, device="cuda")
    ref = build()
    n0 = gp.launch_count()
    ll0, g0 = (x.cpu().numpy().astype(np.float64) for x in ref.loglik_grad(theta))
    n_ref = gp.launch_count() - n0
    ref.close()
    m = build()
    if how != "direct":
        m.loglik(theta)  # the error flags exist before any capture
    with Filled(gp, leave * MB):
        n0 = gp.launch_count()
        if how == "direct":
            ll, g = m.loglik_grad(theta)
        elif how == "graph":
            ll, g = m.loglik_grad(theta, batched=True)
        else:
            ll, g = captured(m, theta)
        torch.cuda.synchronize()
        # the fast way's two kernels more (segments: the information and the
        # adjoints; scalars: the scalars and the elements from them)
        assert gp.launch_count() - n0 == n_ref - (0 if fast else 2)
    assert m.last_error() == (-1, 0)
    ll, g = ll.cpu().numpy(), g.cpu().numpy().astype(np.float64)
    m.close()
    assert np.array_equal(ll, ll0)
    assert np.all(np.abs(g - g0) <= 1e-3 * np.abs(g0) + 1e-4 * np.abs(g0).max(1, keepdims=True))
