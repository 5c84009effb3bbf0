"""Tile bins against the sort: scenes of at most 4096 tiles keep a list per tile that the step itself
appends to, larger ones sort their particles by tile every step.  The same particles in a grid on
either side of that line give the same bits (the grids differ only at walls nothing is near), over
forward steps, checkpointed rollouts and their reverse passes.
"""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S

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


def _body(dim, edge, ctrl, n):
    """A blob that spans several tiles, on a fine grid (dx = 1/64), moving so that particles change
    tiles, far from the high wall of the first axis."""
    s = S.blob(dim, 64, 2500 if dim == 2 else 3000, 61, radius_cells=9.0 if dim == 2 else 6.0, v_scale=1.0,
               c_scale=1.0, f_scale=0.03, center=[0.4] * dim, ctrl_type=ctrl, hidden=8, n_groups=3, amp=2.0,
               bc_width=3, dt=2e-3)
    v = np.array(s.v0)
    v[:, 0] += 3.0  # 0.4 cells a step
    return s.copy(n_grid=n, v0=v, tile_edge=edge if dim == 2 else 0)


# grids of 4096 tiles and just above, by dimension and tile edge
GRIDS = {(2, 4): ((256, 256), (260, 256)), (2, 8): ((512, 512), (520, 512)), (3, 4): ((64, 64, 64), (68, 64, 64))}


@pytest.mark.parametrize("ctrl", [S.CTRL_SIN, S.CTRL_TABLE, S.CTRL_MLP, S.CTRL_COM])
@pytest.mark.parametrize("shape", list(GRIDS))
def test_bins_give_the_bits_of_the_sort(M, ctx, shape, ctrl):
    dim, edge = shape
    res = []
    for n in GRIDS[shape]:
        spec = _body(dim, edge, ctrl, n)
        got = []
        for steps, k in ((11, 1), (11, 4), (3, 2)):  # graph lengths 8 + 3 and 3; segments of 4, 4, 3
            sc = M.Scene(ctx, spec)
            sc.rollout(steps, k)
            got += list(sc.get_state())
            seed = np.zeros((sc.N, dim))
            seed[:, 0] = 1.0 / sc.N
            got += list(sc.backward(seed))
            sc.step(2)  # goes on from the rollout's end after its reverse pass
            got += list(sc.get_state())
            sc.close()
        res.append(got)
    assert np.abs(res[0][1] - _body(dim, edge, ctrl, GRIDS[shape][0]).v0).max() > 0.01
    for a, b in zip(*res):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("dim", [2, 3])
def test_steps_after_a_forward_only_batch_request(M, ctx, dim):
    """A batch advances the scene's particles with lists of its own; stepping the scene afterwards
    starts from the state the batch left."""
    spec = _body(dim, 4, S.CTRL_SIN, (128, 96) if dim == 2 else (48, 48, 48))
    alone = M.Scene(ctx, spec)
    alone.step(13)
    want = alone.get_state()
    alone.close()
    sc = M.Scene(ctx, spec)
    batch = M.Batch(ctx, dim)
    slot = batch.admit(sc, 9, False)
    while not batch.poll(slot):
        batch.tick(4)
    batch.release(slot)
    sc.step(4)
    for a, b in zip(want, sc.get_state()):
        assert np.array_equal(a, b)
    batch.close()
    sc.close()


@pytest.mark.parametrize("N", [1500, 12000, 30000])  # a few, under and over 512 particles a tile
def test_cta_sizes_of_3d_scenes_give_the_same_bits(M, ctx, N):
    """A 3D scene of at most a tile per SM runs wide CTAs, a batch of two to three such scenes (at most
    two tiles per SM) a wider adjoint gather, a larger one the CTAs of large scenes: the results are the
    same bits."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    spec = S.blob(3, 48, N, 62, radius_cells=8.0, v_scale=0.3, c_scale=0.5, f_scale=0.03, n_groups=7, amp=2.0,
                  bc_width=3, dt=5e-4)
    t = np.floor(np.asarray(spec.x0) / spec.dx - 0.5).astype(int) // 4
    tiles = len(np.unique((t[:, 0] * 12 + t[:, 1]) * 12 + t[:, 2]))
    counts = (1, sms // tiles + 1, 2 * sms // tiles + 1)
    assert tiles <= sms < counts[1] * tiles <= 2 * sms < counts[2] * tiles
    T = 6
    want = None
    for B in counts:
        scenes = [M.Scene(ctx, spec) for _ in range(B)]
        batch = M.Batch(ctx, 3)
        slots = [batch.admit(sc, T, True) for sc in scenes]
        while not all(batch.poll(sl) for sl in slots):
            batch.tick(4)
        for sc in scenes:
            got = sc.get_state() + sc.gradients()
            want = want or got
            for a, b in zip(got, want):
                assert np.array_equal(a, b)
        batch.close()
        for sc in scenes:
            sc.close()
    assert np.abs(want[-1]).max() > 0


def test_scenes_beyond_the_bins_room_sort(M, ctx):
    """A context's scenes hold 16 GiB of tile bins between them (128 MB for 64^3 cells, the control
    words beside); the next scene sorts, takes less memory and gives the same bits."""
    import torch
    spec = _body(3, 4, S.CTRL_SIN, (64, 64, 64))
    free = [torch.cuda.mem_get_info()[0]]
    scenes = []
    for _ in range(130):
        scenes.append(M.Scene(ctx, spec))
        free.append(torch.cuda.mem_get_info()[0])
    took = [a - b for a, b in zip(free, free[1:])]
    assert min(took[:127]) - max(took[128:]) > 100 << 20
    for sc in scenes[1:-1]:
        sc.close()
    got = []
    for sc in (scenes[0], scenes[-1]):
        sc.rollout(5, 2)
        seed = np.ones((sc.N, 3))
        got.append(sc.get_state() + sc.backward(seed))
        sc.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
