"""The host-buffer call with the event stream re-sent in several series groups
against the device call: the same bits, whatever the groups.  The number of
groups is read from the launches: a group has a re-layout, a record expansion
and an element pass of its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHO, M32 = 1, 2


def build(gp, terms, sizes, **kw):
    rng = np.random.default_rng(17)
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = off[-1]
    gap = rng.exponential(1.0, n) + 0.05
    t = np.cumsum(gap)
    dur = rng.uniform(0.1, 0.9, n) * np.append(gap[1:], 1.0)
    # values and noise differ from group to group
    y = (rng.standard_normal(n) + np.linspace(-2, 2, n)).astype(np.float32)
    yerr = rng.uniform(0.05, 0.2, n).astype(np.float32)
    return gp.Model(terms, off, t, t + dur, y, yerr, **kw)


def check(gp, m, th, per_series, groups):
    theta = torch.tensor(th, device="cuda")
    n0 = gp.launch_count()
    ll, g = m.loglik_grad(theta, per_series=per_series)
    n1 = gp.launch_count()
    for _ in range(2):
        n2 = gp.launch_count()
        ll_h, g_h = m.loglik_grad_host(th, per_series=per_series, reupload_events=True)
        assert gp.launch_count() - n2 == n1 - n0 + 3 * groups - 1
        assert np.array_equal(ll.cpu().numpy().ravel(), ll_h.ravel())
        assert np.array_equal(g.cpu().numpy().reshape(g_h.shape), g_h)
    # the stream that the groups left on the device
    again = m.loglik_grad(theta, per_series=per_series)
    assert torch.equal(again[0], ll) and torch.equal(again[1], g)


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def test_many_short_series_in_four_groups():
    import paper_2601_02527_gb300 as gp
    rng = np.random.default_rng(1)
    n = 4 * sms() * 128 // 32 + 40
    m = build(gp, (SHO, SHO), rng.integers(1, 50, n), layout=1)
    th = np.array([1.0, 0.63, 0.8, 0.5, 3.1, 0.8, 0.1]) * np.linspace(1, 1.3, n)[:, None]
    check(gp, m, th.astype(np.float32), True, 4)


def test_groups_with_parallel_segments():
    # states of 3 walk segments in parallel up to 12 warps of chunks per SM;
    # two groups begin at 8 (a series of up to 8192 events owns one warp)
    import paper_2601_02527_gb300 as gp
    rng = np.random.default_rng(2)
    n = 9 * sms()
    sizes = rng.integers(1, 40, n)
    sizes[::37] = rng.integers(1100, 3000, len(sizes[::37]))
    m = build(gp, (SHO,), sizes)
    th = (np.array([1.0, 0.63, 3.0, 0.1]) * np.linspace(1, 1.3, n)[:, None]).astype(np.float32)
    check(gp, m, th, True, 2)


def test_shared_sets_in_two_groups():
    import paper_2601_02527_gb300 as gp
    rng = np.random.default_rng(3)
    m = build(gp, (SHO, M32), rng.integers(1, 50, 2 * sms() * 128 // 32 + 8))
    th = np.array([1.0, 0.63, 3.0, 0.5, 5.0, 0.1]) * np.linspace(1, 1.3, 3)[:, None]
    check(gp, m, th.astype(np.float32), False, 2)


def test_a_long_series_alone_is_no_group():
    # the first quarter and half of the events are those of a series of 800 chunks
    import paper_2601_02527_gb300 as gp
    n = 8 * sms() * 128 // 32
    m = build(gp, (SHO,), [20 * n] + [20] * n)
    th = (np.array([1.0, 0.63, 3.0, 0.1]) * np.linspace(1, 1.3, n + 1)[:, None])
    check(gp, m, th.astype(np.float32), True, 2)
