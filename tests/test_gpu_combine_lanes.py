"""The combination with 16 lanes (or a warp) per element against one thread:
the same operations in the same order, so the same bits.  A series (or set)
alone takes the first, among many others the second."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2
THETA = {(SHO,): [1.0, 0.63, 3.0, 0.1], (SHO, M32): [1.0, 0.63, 3.0, 0.5, 5.0, 0.1],
         (SHO, SHO): [1.0, 0.63, 0.8, 0.5, 3.1, 0.8, 0.1]}
# state dimensions 5, 6, 7, 4
SHAPES = [((SHO,), 0, 3), ((SHO, SHO), 1, 1), ((SHO, M32), 0, 3), ((SHO, M32), 0, 0)]


def series(rng, n, slots):
    if slots == 0:
        t = np.cumsum(rng.exponential(1.0, n))
        return t, t.copy(), np.zeros(n, np.int32)
    inst = (np.arange(n) % slots).astype(np.int32)
    t_s, t_e = np.zeros(n), np.zeros(n)
    for k in range(slots):
        m = inst == k
        dur = rng.uniform(0.2, 2.0, m.sum())
        t_e[m] = np.cumsum(dur + rng.exponential(0.5, m.sum()))
        t_s[m] = t_e[m] - dur
    return t_s, t_e, inst


def build(gp, rng, terms, layout, slots, sizes):
    parts = [series(rng, n, slots) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)])
    t_s, t_e, inst = (np.concatenate([p[i] for p in parts]) for i in range(3))
    # the first series' values do not depend on the others
    y = np.random.default_rng(6).standard_normal(off[-1]).astype(np.float32)
    return gp.Model(terms, off, t_s, t_e, y, np.full(off[-1], 0.1, np.float32),
                    inst if slots else None, layout=layout)


@pytest.mark.parametrize("terms,layout,slots", SHAPES)
@pytest.mark.parametrize("others", [400, 10000])  # past the scan's line, past the fold's
def test_series_alone_and_among_others(terms, layout, slots, others):
    import paper_2601_02527_gb300 as gp
    out = []
    for sizes in ([9000], [9000] + [1] * others):
        m = build(gp, np.random.default_rng(4), terms, layout, slots, sizes)
        theta = torch.tensor([THETA[terms]] * len(sizes), dtype=torch.float32, device="cuda")
        ll, g = m.loglik_grad(theta)
        out.append((ll[0].item(), g[0].cpu().numpy().astype(np.float64)))
    (l0, g0), (l1, g1) = out
    assert l0 == l1
    assert np.all(np.abs(g0 - g1) <= 1e-3 * np.abs(g1) + 1e-4 * np.abs(g1).max())


@pytest.mark.parametrize("terms,layout,slots", SHAPES)
def test_long_series_one_set_and_many(terms, layout, slots):
    # more than 16 warps of chunks: the warp totals are scanned in tiles
    import paper_2601_02527_gb300 as gp
    n = 70000 if slots else 140000
    m = build(gp, np.random.default_rng(5), terms, layout, slots, [n])
    th = np.array([THETA[terms]] * 600) * np.linspace(1.0, 1.2, 600)[:, None]
    theta = torch.tensor(th, dtype=torch.float32, device="cuda")
    many = m.loglik(theta, per_series=False)
    for k in (0, 7):
        assert m.loglik(theta[k:k + 1], per_series=False)[0].item() == many[k].item()
