"""Both directions of the combination with several lanes per element against
one thread: a series (or parameter set) alone takes the first, among many
others the second.  The same operations in the same order, so the gradient,
which reads the backward direction's result, is the same bits where both calls
walk their segments alike (segments of 16 events are walked in turn; of 32, in
threads of their own up to 6 warps of chunks per SM)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2
THETA = {(SHO,): [1.0, 0.63, 3.0, 0.1], (SHO, M32): [1.0, 0.63, 3.0, 0.5, 5.0, 0.1],
         (SHO, SHO): [1.0, 0.63, 0.8, 0.5, 3.1, 0.8, 0.1]}
# state dimensions 5, 6, 7, 4
SHAPES = [((SHO,), 0, 3), ((SHO, SHO), 1, 1), ((SHO, M32), 0, 3), ((SHO, M32), 0, 0)]


def build(gp, terms, layout, slots, sizes, **kw):
    # the first series' values do not depend on the others
    rng, rng_y = np.random.default_rng(23), np.random.default_rng(24)
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = off[-1]
    t = np.arange(n) + rng.uniform(0, 0.3, n)
    y = rng_y.standard_normal(n).astype(np.float32)
    # slots exposures open at a time
    t_e = t + (0.0 if slots == 0 else slots - 0.5)
    return gp.Model(terms, off, t, t_e, y, np.full(n, 0.1, np.float32), layout=layout, **kw)


@pytest.mark.parametrize("terms,layout,slots", SHAPES)
@pytest.mark.parametrize("others,ck", [(400, 32), (400, 16), (10000, 16)])
def test_series_alone_and_among_others(terms, layout, slots, others, ck):
    import paper_2601_02527_gb300 as gp
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert 2 * (others + 1) > sms  # past the line of the scan by 16 lanes
    out = []
    for sizes in ([9000], [9000] + [1] * others):
        m = build(gp, terms, layout, slots, sizes, ckpt_interval=ck)
        assert m.info["n_slots"] == slots
        theta = torch.tensor([THETA[terms]] * len(sizes), dtype=torch.float32, device="cuda")
        ll, g = m.loglik_grad(theta)
        assert m.last_error() == (-1, 0)
        out.append((ll[0].item(), g[0].cpu().numpy()))
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("terms,layout,slots", SHAPES)
def test_long_series_one_set_and_many(terms, layout, slots):
    # more than 16 warps of chunks: the warp totals are scanned in tiles
    import paper_2601_02527_gb300 as gp
    m = build(gp, terms, layout, slots, [70000 if slots else 140000], ckpt_interval=16)
    assert m.info["n_chunks"] > 16 * 32
    th = np.array([THETA[terms]] * 600) * np.linspace(1.0, 1.2, 600)[:, None]
    theta = torch.tensor(th, dtype=torch.float32, device="cuda")
    many, g = m.loglik_grad(theta, per_series=False)
    for k in (0, 7):
        one, g1 = m.loglik_grad(theta[k:k + 1], per_series=False)
        assert one[0].item() == many[k].item()
        assert torch.equal(g1[0], g[k])
