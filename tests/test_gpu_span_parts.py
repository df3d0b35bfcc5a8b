"""Spans that are not whole warps of 32 chunks (a short series over several
ranks, or any range a caller picks): the spans' elements fold to the unsplit
log-likelihood, 1e-4 max(|L|, 0.1 N), whatever ran on the GPU before.  A batch
of other parameters runs before each span, so that shared memory holds their
tables."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2
THETA = {(SHO,): [1.0, 0.63, 3.0, 0.1], (SHO, M32): [1.0, 0.63, 3.0, 0.5, 5.0, 0.1],
         (SHO, SHO): [1.0, 0.63, 0.8, 0.5, 3.1, 0.8, 0.1]}


def build(gp, terms, layout, n, series=1):
    rng = np.random.default_rng(31)
    t = np.arange(n * series) + rng.uniform(0, 0.4, n * series)
    y = rng.standard_normal(n * series).astype(np.float32)
    return gp.Model(terms, np.arange(series + 1) * n, t, t + 0.5, y,
                    np.full(n * series, 0.1, np.float32), layout=layout)


@pytest.mark.parametrize("terms,layout", [((SHO,), 0), ((SHO, M32), 0), ((SHO, SHO), 1)])
@pytest.mark.parametrize("sets", [1, 3])
@pytest.mark.parametrize("cuts", [[0, 16, 32], [0, 1, 32], [0, 11, 12, 27, 32]])
def test_partial_warps(terms, layout, sets, cuts):
    import paper_2601_02527_gb300 as gp
    n = 400
    m = build(gp, terms, layout, n)
    assert m.info["n_chunks"] == 32
    base = np.array(THETA[terms])
    theta = torch.tensor(base * np.linspace(1, 1.5, sets)[:, None], dtype=torch.float32,
                         device="cuda")
    ref = m.loglik(theta, per_series=False).cpu().numpy()
    other = build(gp, terms, layout, 40, 2000)
    wrong = torch.tensor(np.tile(3.0 * base, (2000, 1)), dtype=torch.float32, device="cuda")
    spans = []
    for c0, c1 in zip(cuts, cuts[1:]):
        other.loglik(wrong)
        spans.append(m.span_element(theta, c0, c1, per_series=False))
    got = m.span_loglik(torch.stack(spans)).cpu().numpy()
    assert m.last_error() == (-1, 0)
    assert np.all(np.abs(got - ref) <= 1e-4 * np.maximum(np.abs(ref), 0.1 * n)), (got, ref)
