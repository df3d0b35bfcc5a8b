"""The log-likelihood of product models on both sides of the rule by which their
step scalars are formed at once: the same bits as step by step (step_cache =
1), overdamped rows among them.  The route is read from the launches: at once
takes two more."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROD, SHO, M32 = 3, 1, 2
BASE = {(PROD,): [1.0, 0.13, 1.0, 1.26, 10.0], (PROD, M32): [1.0, 0.13, 1.0, 1.26, 10.0, 0.5, 5.0],
        (PROD, SHO): [1.0, 0.13, 0.5, 1.26, 0.3, 0.5, 0.63, 0.4]}


@pytest.mark.parametrize("terms", list(BASE))
@pytest.mark.parametrize("events,sets", [(2, 0), (30, 0), (32, 0), (62, 2), (64, 0), (200, 3),
                                         (64, 400)])
def test_routes_of_the_loglik(terms, events, sets):
    import paper_2601_02527_gb300 as gp
    rng = np.random.default_rng(19)
    # the longest chunk has `events` events (an even number: chunks end at even ones)
    sizes = [32 * events, 5, 17 * events]
    off = np.concatenate([[0], np.cumsum(sizes)])
    t = np.cumsum(rng.exponential(1.0, off[-1]))
    y = rng.standard_normal(off[-1]).astype(np.float32)
    rows = sets if sets else len(sizes)
    th = np.array(BASE[terms] + [0.1]) * np.exp(0.1 * rng.standard_normal((rows, len(BASE[terms]) + 1)))
    th[0, 2] = 0.3  # overdamped
    theta = torch.tensor(th, dtype=torch.float32, device="cuda")
    out, n = [], []
    for cache in (0, 1):
        m = gp.Model(terms, off, t, t, y, np.full(off[-1], 0.1, np.float32), step_cache=cache)
        n0 = gp.launch_count()
        out.append(m.loglik(theta, per_series=not sets).cpu().numpy())
        n.append(gp.launch_count() - n0)
        assert m.last_error() == (-1, 0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    least, per_sm = (64, 2) if len(terms) == 1 else (32, 4)
    at_once = events >= least and 3 * max(sets, 1) <= per_sm * sms
    assert n[0] - n[1] == (2 if at_once else 0)
    assert np.array_equal(out[0], out[1])
