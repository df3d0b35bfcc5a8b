"""The gradient with one thread per segment against the walk of a chunk's
segments in turn (the sequential combination keeps it) and against the oracle,
for ragged series: empty and one-segment chunks, segments shorter than the
interval, chunks of one series that differ in length.  Tolerances: the
gradient's 1e-3 |g| + 1e-4 max|g|, the conditioned values' 1e-3 of the largest
mean and 2e-3 var + 2e-4 of the largest variance."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2
THETA = {(SHO,): [1.0, 0.63, 3.0, 0.1], (SHO, M32): [1.0, 0.63, 3.0, 0.5, 5.0, 0.1],
         (SHO, SHO): [1.0, 0.63, 0.3, 0.5, 3.1, 0.8, 0.1]}
SIZES = [1, 7, 513, 1200, 6000]


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


@pytest.mark.parametrize("terms,layout,slots,sets", [
    ((SHO,), 0, 0, 0), ((SHO,), 0, 1, 0), ((SHO,), 0, 3, 2), ((SHO, M32), 0, 0, 3),
    ((SHO, M32), 0, 1, 0), ((SHO, SHO), 1, 1, 0), ((SHO, SHO), 0, 3, 0)])
@pytest.mark.parametrize("ck", [32, 64])
def test_segments(terms, layout, slots, sets, ck):
    import paper_2601_02527_gb300 as gp
    oracle.build()
    rng = np.random.default_rng(11)
    parts = [series(rng, n, slots) for n in SIZES]
    off = np.concatenate([[0], np.cumsum(SIZES)])
    t_s, t_e, inst = (np.concatenate([p[i] for p in parts]) for i in range(3))
    inst = inst if slots else None
    y = rng.standard_normal(off[-1]).astype(np.float32)
    yerr = rng.uniform(0.05, 0.2, off[-1]).astype(np.float32)
    rows = sets if sets else len(SIZES)
    th = (np.array(THETA[terms]) * np.exp(0.2 * rng.standard_normal((rows, len(THETA[terms])))))
    th = th.astype(np.float32)
    theta = torch.tensor(th, device="cuda")
    out = []
    for combine in (0, 1):
        m = gp.Model(terms, off, t_s, t_e, y, yerr, inst, layout=layout, ckpt_interval=ck,
                     combine=combine)
        ll, g = m.loglik_grad(theta, per_series=not sets)
        _, cond = m.condition(theta, per_series=not sets)
        assert m.last_error() == (-1, 0)
        out.append((ll.cpu().numpy(), g.cpu().numpy().astype(np.float64),
                    cond.cpu().numpy().astype(np.float64)))
    (_, g0, c0), (_, g1, c1) = out
    scale = np.abs(g1).max(axis=1, keepdims=True)
    assert np.all(np.abs(g0 - g1) <= 1e-3 * np.abs(g1) + 1e-4 * scale)
    assert np.all(np.abs(c0 - c1)[..., 0] <= 1e-3 * np.abs(c1[..., 0]).max())
    assert np.all(np.abs(c0 - c1)[..., 1] <= 2e-3 * c1[..., 1] + 2e-4 * c1[..., 1].max())
    for i in (2, 3):
        a, b = off[i], off[i + 1]
        _, ref = oracle.loglik(list(terms), layout, t_s[a:b], t_e[a:b], y[a:b].astype(np.float64),
                               yerr[a:b].astype(np.float64),
                               th[0 if sets else i].astype(np.float64),
                               instrument=None if inst is None else inst[a:b], grad=True)
        assert np.all(np.abs(g0[i] - ref) <= 1e-3 * np.abs(ref) + 1e-4 * np.abs(ref).max())
