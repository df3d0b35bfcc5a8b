"""Which gradient calls walk a chunk's segments in parallel, seen from the
launches: two more than the walk in turn (the information at the segments'
ends and the adjoints there)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2
THETA = {(SHO,): [1.0, 0.63, 3.0, 0.1], (SHO, M32): [1.0, 0.63, 3.0, 0.5, 5.0, 0.1]}


def build(gp, terms, n, **kw):
    rng = np.random.default_rng(21)
    t = np.cumsum(rng.exponential(1.0, n))
    dur = rng.uniform(0.05, 0.5, n) * np.diff(t, append=t[-1] + 1)
    y = rng.standard_normal(n).astype(np.float32)
    yerr = rng.uniform(0.05, 0.2, n).astype(np.float32)
    m = gp.Model(terms, [0, n], t, t + dur, y, yerr, **kw)
    return m, (t, t + dur, y.astype(np.float64), yerr.astype(np.float64))


def launches(gp, f):
    n0 = gp.launch_count()
    out = f()
    return gp.launch_count() - n0, out


@pytest.mark.parametrize("terms", list(THETA))
@pytest.mark.parametrize("prec", [32, 64])
def test_fp64_combination_walks_in_turn(terms, prec):
    # 1000 exposures: chunks of up to 64 events, two segments.  With the combination
    # in FP64 every segment starts from what was walked back from the FP64
    # adjoint at the chunk's end, as with segments too short for threads of
    # their own (ckpt_interval = 16).
    import paper_2601_02527_gb300 as gp
    oracle.build()
    theta = torch.tensor([THETA[terms]], dtype=torch.float32, device="cuda")
    m, data = build(gp, terms, 1000, combine_precision=prec)
    turn, _ = build(gp, terms, 1000, combine_precision=prec, ckpt_interval=16)
    n, (ll, g) = launches(gp, lambda: m.loglik_grad(theta))
    n1, _ = launches(gp, lambda: turn.loglik_grad(theta))
    assert n == n1 + (2 if prec == 32 else 0)
    nc, _ = launches(gp, lambda: m.condition(theta))
    nc1, _ = launches(gp, lambda: turn.condition(theta))
    assert nc == nc1 + (2 if prec == 32 else 0)
    ref_ll, ref = oracle.loglik(list(terms), 0, *data, np.array(THETA[terms], np.float32)
                                .astype(np.float64), grad=True)
    assert abs(ll.item() - ref_ll) <= 1e-4 * max(abs(ref_ll), 100.0)
    g = g[0].cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 1e-3 * np.abs(ref) + 1e-4 * np.abs(ref).max())


@pytest.mark.parametrize("full,length,parallel", [(5, 64, True), (8, 64, False), (1, 48, True),
                                                  (1, 46, False)])
def test_equal_chunks_past_the_line_walk_in_turn(full, length, parallel):
    # states of 3, `full` warps per SM of chunks of `length` events each
    import paper_2601_02527_gb300 as gp
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, rows = 16 * length, full * sms
    t = np.arange(n * rows) + 0.1
    y = np.random.default_rng(3).standard_normal(n * rows).astype(np.float32)
    theta = torch.tensor([THETA[(SHO,)]] * rows, dtype=torch.float32, device="cuda")
    n_launch = []
    for ck in (32, 16):
        m = gp.Model((SHO,), np.arange(rows + 1) * n, t, t + 0.5, y,
                     np.full(n * rows, 0.1, np.float32), chunk_len=64, ckpt_interval=ck)
        assert m.info["n_chunks"] == 32 * rows
        n_launch.append(launches(gp, lambda: m.loglik_grad(theta))[0])
    assert n_launch[0] - n_launch[1] == (2 if parallel else 0)
