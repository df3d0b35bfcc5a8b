"""The product gradient in other units of time: times scaled by 2^k, rates by
2^-k, lengths by 2^k.  The log-likelihood is the same and each gradient
component scales by its parameter's unit, to the gradient's 1e-3 |g| +
1e-4 max|g| (pivots of the combination may fall differently).  One length
scale makes the plain term's rate a power of two."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROD, SHO, M32 = 3, 1, 2
SQRT3 = float(np.float32(1.7320508))


@pytest.mark.parametrize("k", [-20, 20, 24])
@pytest.mark.parametrize("terms,th,unit", [
    ((PROD,), [1.0, 0.0013, 1.0, 0.126, 0.3, 0.1], [0, -1, 0, -1, 0, 0]),
    ((PROD, M32), [1.0, 0.013, 1.0, 1.26, 10.0, 0.5, 5.0, 0.1], [0, -1, 0, -1, 0, 0, 1, 0]),
    ((PROD, M32), [1.0, 0.25, 0.5, 2.0, 10.0, 0.5, SQRT3, 0.1], [0, -1, 0, -1, 0, 0, 1, 0]),
    ((PROD, SHO), [1.0, 0.13, 1.0, 1.26, 10.0, 0.5, 0.63, 0.4, 0.1],
     [0, -1, 0, -1, 0, 0, -1, 0, 0])])
def test_gradient_in_units_of_time(terms, th, unit, k):
    import paper_2601_02527_gb300 as gp
    rng = np.random.default_rng(13)
    n = 900
    gap = rng.exponential(1.0, n)
    gap[[100, 500]] = 30.0, 200.0
    t = np.cumsum(gap)
    y = rng.standard_normal(n).astype(np.float32)
    th = np.array(th, np.float32)
    out = []
    for cache, u in ((1, 1.0), (0, 1.0), (0, 2.0 ** k)):
        size = u ** np.array(unit, float)
        m = gp.Model(terms, [0, n], t * u, t * u, y, np.full(n, 0.1, np.float32), step_cache=cache)
        ll, g = m.loglik_grad(torch.tensor((th * size).astype(np.float32)[None], device="cuda"))
        assert m.last_error() == (-1, 0)
        out.append((ll.item(), g[0].cpu().numpy().astype(np.float64) * size))
    (l0, g0), *rest = out
    # components have units of their own: each against what the parameter's own
    # size makes of it
    rel = g0 * th
    for l1, g1 in rest:
        assert abs(l1 - l0) <= 1e-6 * abs(l0)
        assert np.all(np.abs(g1 * th - rel) <= 1e-3 * np.abs(rel) + 1e-4 * np.abs(rel).max())
