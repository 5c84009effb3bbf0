"""3D scenes of few tiles run wide CTAs, one or two per SM.  The class follows the particles: set to, or
spread over, more tiles the scene (or a batch's composition) takes the shapes of larger scenes, with the
same bits; and while it runs the wide CTAs, nothing is tried for them or put in the tuner's cache."""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S
from tests.parity_utils import mean_x0_seed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_1810_01054_gb300 import mpm
    return mpm


@pytest.fixture(scope="module")
def ctx(M):
    c = M.Context(0)
    yield c
    c.close()


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _tiles(spec, x):
    t = np.floor(np.asarray(x, np.float64) / spec.dx - 0.5).astype(int) // 4
    return len(np.unique(t, axis=0))


def _grads(sc, T, k):
    sc.rollout(T, k)
    return list(sc.get_state()) + list(sc.backward(mean_x0_seed(sc.N, 3)))  # a batch request's loss


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def _bodies(N, n_grid):
    """A compact body and the same particles over more than two tiles per SM."""
    opt = dict(v_scale=0.2, f_scale=0.02, n_groups=3, amp=2.0, bc_width=3, dt=5e-4, center=[0.45, 0.45, 0.45])
    compact, spread = (S.blob(3, 64, N, 121, radius_cells=r, **opt).copy(n_grid=n_grid) for r in (6.0, 22.0))
    assert _tiles(compact, compact.x0) <= _sms() < 2 * _sms() < _tiles(spread, spread.x0)
    return compact, spread


def test_the_tuner_leaves_wide_kernels_alone_until_the_body_is_spread(M, ctx):
    N, grid = 9000, (72, 60, 64)
    compact, spread = _bodies(N, grid)
    key = (3, N, 18 * 15 * 16, _sms())
    assert M.tune_cache_lookup(*key) is None
    sc = M.Scene(ctx, compact)
    assert all(sc.launch(k)[2] for k in range(4))  # nothing to try
    for _ in range(3):
        _grads(sc, 24, 1)
    assert M.tune_cache_lookup(*key) is None  # and nothing stored

    def spread_pass(T=24, k=1):
        sc.set_state(spread.x0, spread.v0, spread.C0, spread.F0, step=0)
        return _grads(sc, T, k)

    first = spread_pass(5, 2)  # begins with the wide CTAs
    assert not any(sc.launch(k)[2] for k in range(4))  # more tiles were seen
    _same(spread_pass(5, 2), first)
    want = spread_pass()
    for _ in range(2):
        _same(spread_pass(), want)
    assert all(sc.launch(k)[2] for k in range(4))
    assert M.tune_cache_lookup(*key) == [sc.launch(k)[:2] if k != M.TK_ADJ_GATHER else (sc.launch(k)[0], 256)
                                         for k in range(4)]
    _same(spread_pass(5, 2), first)
    # a compact scene of that key does not take the shapes, one created spread does
    again, wide = M.Scene(ctx, compact), M.Scene(ctx, spread)
    assert [wide.launch(k) for k in range(4)] == [sc.launch(k) for k in range(4)]
    assert all(again.launch(k)[2] for k in range(4))
    for s in (sc, again, wide):
        s.close()


def test_a_body_that_falls_apart_keeps_its_bits(M, ctx):
    """Alone, looked at now and then, and in a batch beside another scene: the class changes on the way."""
    s = S.blob(3, 64, 8000, 122, radius_cells=5.0, n_groups=3, amp=1.0, bc_width=3, dt=1e-4, gravity=(0, 0, 0))
    rate = 400.0  # the body's radius grows by 4 % of its first size a step
    v = rate * (np.asarray(s.x0) - np.asarray(s.x0).mean(0))
    s = s.copy(v0=v, C0=np.broadcast_to(rate * np.eye(3), (8000, 3, 3)).copy())
    T = 60
    sc = M.Scene(ctx, s)
    sc.set_tuning(M.TUNE_OFF)
    want = _grads(sc, T, 1)  # one call: wide CTAs to its end
    assert _tiles(s, s.x0) <= _sms() < 2 * _sms() < _tiles(s, want[0])
    sc.close()
    for mode in (M.TUNE_OFF, M.TUNE_AUTO):
        sc = M.Scene(ctx, s)
        sc.set_tuning(mode)
        for _ in range(T // 10):
            sc.step(10)
            got = sc.get_state()
        _same(got, want[:4])
        sc.set_state(s.x0, s.v0, s.C0, s.F0, step=0)
        _same(_grads(sc, T, 7), want)
        sc.close()
    a, other = M.Scene(ctx, s), M.Scene(ctx, S.blob(3, 24, 500, 123, radius_cells=4.0, dt=1e-4))
    batch = M.Batch(ctx, 3)
    slots = [batch.admit(a, T, True), batch.admit(other, 3 * T, False)]
    while not all(batch.poll(sl) for sl in slots):
        batch.tick(3)
        ctx.sync()  # the tiles of the step have arrived when the next tick looks
    _same(list(a.get_state()) + list(a.gradients()), want)
    batch.close()
    for x in (a, other):
        x.close()
