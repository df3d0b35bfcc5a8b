"""The element pass and the gradient walk take the warps of chunks by length;
results do not depend on where a series stands.  Series of very different
lengths, each alone and within a batch in two orders: the same chunks, so the
log-likelihoods are the same bits, and the gradients too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2


@pytest.mark.parametrize("terms,sets", [((SHO,), 0), ((SHO, M32), 0), ((SHO,), 3)])
def test_order_of_series(terms, sets):
    import paper_2601_02527_gb300 as gp
    rng = np.random.default_rng(3)
    sizes = [3, 5000, 40, 900, 9000, 1, 20000, 300]
    np_ = 3 * len(terms) + 1 - (M32 in terms)
    base = np.array([1.0, 0.63, 3.0, 0.5, 5.0])[:np_ - 1]
    rows = sets if sets else len(sizes)
    th = np.concatenate([base * np.exp(0.2 * rng.standard_normal((rows, np_ - 1))),
                         np.full((rows, 1), 0.1)], 1).astype(np.float32)
    t = [np.cumsum(rng.exponential(1.0, n)) for n in sizes]
    dur = [rng.uniform(0.05, 0.5, n) * np.diff(x, append=x[-1] + 1) for n, x in zip(sizes, t)]
    y = [rng.standard_normal(n).astype(np.float32) for n in sizes]

    def run(pick):
        off = np.concatenate([[0], np.cumsum([sizes[i] for i in pick])])
        cat = [np.concatenate([a[i] for i in pick]) for a in (t, dur, y)]
        m = gp.Model(terms, off, cat[0], cat[0] + cat[1], cat[2],
                     np.full(off[-1], 0.1, np.float32), combine=1)
        theta = torch.tensor(th if sets else th[pick], device="cuda")
        ll, g = m.loglik_grad(theta, per_series=not sets)
        n = len(pick)
        return (ll.cpu().numpy().reshape(-1, n), g.cpu().numpy().reshape(-1, n, np_))

    whole = run(list(range(len(sizes))))
    back = run(list(range(len(sizes)))[::-1])
    for k in range(2):
        assert np.array_equal(whole[k], back[k][:, ::-1])
    for i in range(len(sizes)):
        one = run([i])
        for k in range(2):
            assert np.array_equal(whole[k][:, i], one[k][:, 0])
