"""The plain FP64 filter against the oracle at the edges of its batches of 32
events and for every compiled shape.  Both are FP64 filters of the same
recursion: |L_gpu - L_or| <= 1e-9 max(|L_or|, 0.1 N)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2
THETA = {(SHO,): [1.0, 0.63, 3.0, 0.1], (SHO, M32): [1.0, 0.63, 3.0, 0.5, 5.0, 0.1],
         (SHO, SHO): [1.0, 0.63, 0.3, 0.5, 3.1, 0.8, 0.1]}


def series(rng, n, slots, instants):
    """n measurements: instants (slots = 0), or exposures of ``slots`` instruments
    that overlap one another, ``instants`` of them shrunk to instants."""
    if slots == 0:
        t = np.cumsum(rng.exponential(1.0, n))
        return t, t.copy(), None
    inst = np.arange(n) % slots
    t_s = np.zeros(n)
    t_e = np.zeros(n)
    for k in range(slots):
        m = inst == k
        dur = rng.uniform(0.2, 2.0, m.sum())
        t_e[m] = np.cumsum(dur + rng.exponential(0.5, m.sum()))
        t_s[m] = t_e[m] - dur
    t_e[:instants] = t_s[:instants]
    return t_s, t_e, inst.astype(np.int32)


@pytest.mark.parametrize("terms,layout,slots,instants", [
    ((SHO,), 0, 0, 0), ((SHO,), 0, 1, 0), ((SHO,), 0, 2, 3), ((SHO,), 0, 3, 0),
    ((SHO, M32), 0, 0, 0), ((SHO, M32), 0, 1, 0), ((SHO, SHO), 0, 2, 0), ((SHO, SHO), 0, 3, 5),
    ((SHO, SHO), 1, 1, 0), ((SHO, SHO), 1, 1, 4)])
def test_batches(terms, layout, slots, instants):
    import paper_2601_02527_gb300 as gp
    oracle.build()
    rng = np.random.default_rng(5)
    sizes = [1, 8, 15, 16, 17, 31, 32, 33, 64, 200]
    parts = [series(rng, n, slots, min(instants, n - 1)) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)])
    t_s, t_e = (np.concatenate([p[i] for p in parts]) for i in (0, 1))
    inst = None if slots == 0 else np.concatenate([p[2] for p in parts])
    y = rng.standard_normal(off[-1]).astype(np.float32)
    yerr = rng.uniform(0.05, 0.2, off[-1]).astype(np.float32)
    th = np.array([THETA[terms]], np.float32)
    m = gp.Model(terms, off, t_s, t_e, y, yerr, inst, layout=layout, precision=64)
    ll = m.loglik(torch.tensor(th, device="cuda"), per_series=False).cpu().numpy()
    assert m.last_error() == (-1, 0)
    for i, n in enumerate(sizes):
        a, b = off[i], off[i + 1]
        ref = oracle.loglik(list(terms), layout, t_s[a:b], t_e[a:b], y[a:b].astype(np.float64),
                            yerr[a:b].astype(np.float64), th[0].astype(np.float64),
                            instrument=None if inst is None else inst[a:b])
        assert abs(ll[i] - ref) <= 1e-9 * max(abs(ref), 0.1 * n), (n, ll[i], ref)
