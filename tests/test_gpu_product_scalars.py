"""Product models with the step scalars formed for all steps at once against
the kernels that form them step by step (step_cache = 1): the same FP32
arithmetic for the log-likelihood, hence the same bits, and the gradient within its 1e-3 |g| + 1e-4 max|g|.  Chunk lengths around
the steps a block takes (8), empty chunks, repeated times, overdamped and
critically damped factors, both kinds of plain term, shared sets."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROD, SHO, M32 = 3, 1, 2
BASE = {(PROD,): [1.0, 0.13, 1.0, 1.26, 10.0], (PROD, M32): [1.0, 0.13, 1.0, 1.26, 10.0, 0.5, 5.0],
        (PROD, SHO): [1.0, 0.13, 0.5, 1.26, 0.3, 0.5, 0.63, 0.4]}


@pytest.mark.parametrize("terms", list(BASE))
@pytest.mark.parametrize("chunk,sets", [(0, 0), (7, 0), (8, 2), (33, 0)])
def test_scalars_at_once(terms, chunk, sets):
    import paper_2601_02527_gb300 as gp
    assert gp.SHO_PRODUCT == PROD
    rng = np.random.default_rng(9)
    sizes = [1, 31, 257, 1500]
    off = np.concatenate([[0], np.cumsum(sizes)])
    gaps = [rng.exponential(1.0, n) for n in sizes]
    gaps[2][10:14] = 0.0
    gaps[3][100] = 400.0
    t = np.concatenate([np.cumsum(g) for g in gaps])
    y = rng.standard_normal(off[-1]).astype(np.float32)
    yerr = rng.uniform(0.05, 0.2, off[-1]).astype(np.float32)
    rows = sets if sets else len(sizes)
    b = np.array(BASE[terms] + [0.1])
    th = (b * np.exp(0.1 * rng.standard_normal((rows, len(b))))).astype(np.float32)
    th[0] = b  # Q = 1/2 exactly where the base has it
    theta = torch.tensor(th, device="cuda")
    out = []
    for cache in (0, 1):
        m = gp.Model(terms, off, t, t, y, yerr, chunk_len=chunk, step_cache=cache)
        only = m.loglik(theta, per_series=not sets).cpu().numpy()
        ll, g = m.loglik_grad(theta, per_series=not sets)
        assert m.last_error() == (-1, 0)
        assert np.array_equal(only, ll.cpu().numpy())
        out.append((only, g.cpu().numpy().astype(np.float64)))
    (l0, g0), (l1, g1) = out
    assert np.array_equal(l0, l1)
    assert np.all(np.abs(g0 - g1) <= 1e-3 * np.abs(g1) + 1e-4 * np.abs(g1).max(1, keepdims=True))
