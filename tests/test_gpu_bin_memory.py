"""What tile bins take: every set counts against the context's bound, the further sets of a reverse pass
come from what its memory budget leaves, and where the bound, the budget or the device has no room the
scene, its reverse pass or the batch does without, with the same bits."""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def M():
    from paper_1810_01054_gb300 import mpm
    return mpm


@pytest.fixture()
def ctx(M):
    c = M.Context(0)
    yield c
    c.close()


def _spec(dim=3, ctrl=S.CTRL_SIN):
    """A moving blob in a grid of 4096 tiles (3D, 134 MB a set; 2D 34 MB)."""
    n = (64, 64, 64) if dim == 3 else (256, 256)
    s = S.blob(dim, 64, 3000, 101, radius_cells=6.0 if dim == 3 else 9.0, v_scale=1.0, c_scale=1.0, f_scale=0.03,
               center=[0.4] * dim, ctrl_type=ctrl, hidden=8, n_groups=3, amp=2.0, bc_width=3, dt=2e-3)
    v = np.array(s.v0)
    v[:, 0] += 3.0  # 0.4 cells a step: particles change tiles
    return s.copy(n_grid=n, v0=v, tile_edge=4 if dim == 2 else 0)


def _pass(sc, spec, T, k, budget=0):
    sc.set_state(spec.x0, spec.v0, spec.C0, spec.F0, step=0)
    sc.rollout(T, k, budget)
    return list(sc.get_state()) + list(sc.backward(np.full((sc.N, sc.dim), 1.0 / sc.N)))


def _same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_every_set_is_counted_and_given_back(M, ctx):
    import torch
    spec = _spec()
    free = torch.cuda.mem_get_info()[0]
    sc = M.Scene(ctx, spec)
    one = ctx.bin_bytes()[0]
    assert 128 * MB <= one <= 136 * MB
    _pass(sc, spec, 9, 3)  # the reverse pass takes two further sets
    assert ctx.bin_bytes()[0] == 3 * one
    assert free - torch.cuda.mem_get_info()[0] >= 3 * one
    batch = M.Batch(ctx, 3)
    slot = batch.admit(sc, 3, True)
    while not batch.poll(slot):
        batch.tick(4)
    assert ctx.bin_bytes()[0] > 3 * one
    batch.release(slot)
    batch.close()
    assert ctx.bin_bytes()[0] == 3 * one
    sc.close()
    assert ctx.bin_bytes()[0] == 0


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("ctrl", [S.CTRL_SIN, S.CTRL_MLP])
def test_bounds_that_hold_some_of_the_sets_give_the_same_bits(M, ctx, dim, ctrl):
    """No set, the scene's alone, and one and both of its reverse pass's (a controller that reads the
    state takes only the recompute's)."""
    spec = _spec(dim, ctrl)
    sc = M.Scene(ctx, spec)
    one = ctx.bin_bytes()[0]
    shapes = ((11, 4), (11, 1), (3, 2))  # segments of 4, 4, 3; every state; segments of 2 and 1
    want = [_pass(sc, spec, T, k) for T, k in shapes]
    sc.close()
    for sets in range(4):
        ctx.set_bin_bytes(sets * one + one // 2)
        sc = M.Scene(ctx, spec)
        for (T, k), ref in zip(shapes, want):
            _same(_pass(sc, spec, T, k), ref)
            assert ctx.bin_bytes()[0] <= sets * one
        assert ctx.bin_bytes()[0] == min(sets, 3 if ctrl == S.CTRL_SIN else 2) * one
        sc.close()


def test_a_budget_counts_the_further_sets(M, ctx):
    import torch
    spec = _spec()
    sc = M.Scene(ctx, spec)
    one, size = ctx.bin_bytes()[0], sc.info()["state_bytes"]
    T, k = 12, 3
    store = (4 + 2 * (k - 1)) * size
    want = _pass(sc, spec, T, k, store)
    assert ctx.bin_bytes()[0] == one
    free = torch.cuda.mem_get_info()[0]
    for budget, sets in ((store, 1), (store + one, 2), (store + 2 * one, 3), (store, 1), (0, 3), (T * size, 1)):
        _same(_pass(sc, spec, T, k if budget != T * size else 0, budget), want)
        assert ctx.bin_bytes()[0] == sets * one, (budget, sets)
        # nothing of that size beside the sets
        assert abs(free - torch.cuda.mem_get_info()[0] - (sets - 1) * one) < one // 2, (budget, sets)
    _same(_pass(sc, spec, T, k), want)
    assert ctx.bin_bytes()[0] == 3 * one
    _same(_pass(sc, spec, T, 0, 4 * size), want)  # the multi-level store
    assert ctx.bin_bytes()[0] == one
    sc.close()


@pytest.mark.parametrize("dim", [2, 3])
def test_batches_beyond_the_bound_sort(M, ctx, dim):
    spec = _spec(dim)
    res = []
    for most in (None, 0):
        if most is not None:
            ctx.set_bin_bytes(most)
        scenes = [M.Scene(ctx, spec) for _ in range(2)]
        batch = M.Batch(ctx, dim)
        slots = [batch.admit(sc, 7, g) for sc, g in zip(scenes, (True, False))]
        while not all(batch.poll(sl) for sl in slots):
            batch.tick(3)
        held = ctx.bin_bytes()[0]
        assert held == 0 if most == 0 else held > 0
        res.append(list(scenes[0].get_state()) + list(scenes[0].gradients()) + list(scenes[1].get_state()))
        batch.close()
        for sc in scenes:
            sc.close()
        assert ctx.bin_bytes()[0] == 0
    _same(*res)


def test_bins_the_device_cannot_hold_are_not_counted(M, ctx):
    import torch
    spec = _spec()
    sc = M.Scene(ctx, spec)
    want = _pass(sc, spec, 6, 2)
    sc.close()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 112 * MB, dtype=torch.uint8, device="cuda")
    try:
        sc = M.Scene(ctx, spec)  # its 134 MB of bins do not fit, the rest does
        assert ctx.bin_bytes()[0] == 0
        sc.set_state(spec.x0, spec.v0, spec.C0, spec.F0, step=0)
        sc.step(6)
        _same(list(sc.get_state()), want[:4])
        sc.close()
    finally:
        del fill
        torch.cuda.empty_cache()


def test_out_of_memory_is_answered_once(M, ctx):
    """A call that found no device memory leaves no error behind for the next one."""
    import torch
    spec = _spec()
    sc = M.Scene(ctx, spec)
    sc.step(2)
    sc.get_state()
    T = 64 * MB // sc.info()["state_bytes"]
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 16 * MB, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(M.MPMError) as e:
            sc.rollout(T, 1)  # 64 MB of states
        assert e.value.status == -2
    finally:
        del fill
        torch.cuda.empty_cache()
    want = _pass(sc, spec, 6, 2)
    other = M.Scene(ctx, spec)
    _same(_pass(other, spec, 6, 2), want)
    other.close()
    sc.close()


def test_a_batch_that_ran_out_of_memory_goes_on_when_there_is_some(M, ctx):
    """A composition that does not fit is answered with MPM_ERR_OOM; the same call later allocates anew."""
    import torch
    spec = _spec()
    ctx.set_bin_bytes(0)
    scenes = [M.Scene(ctx, spec) for _ in range(3)]
    batch = M.Batch(ctx, 3)
    slot = batch.admit(scenes[0], 5, False)  # the batch's arrays are sized for one scene
    while not batch.poll(slot):
        batch.tick(5)
    want = list(scenes[0].get_state())
    batch.release(slot)
    slots = [batch.admit(sc, 5, False) for sc in scenes[1:]]
    torch.cuda.empty_cache()
    # two scenes' node blocks are 28 MB twice, one scene's (given back first) 14 MB twice
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 16 * MB, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(M.MPMError) as e:
            batch.tick(5)
        assert e.value.status == -2
    finally:
        del fill
        torch.cuda.empty_cache()
    while not all(batch.poll(sl) for sl in slots):
        batch.tick(5)
    for sc in scenes[1:]:
        _same(list(sc.get_state()), want)
    batch.close()
    for sc in scenes:
        sc.close()


def test_requests_that_finished_close_though_the_next_composition_does_not_fit(M, ctx):
    """A tick in which a short request ends before a longer one's next phase finds no memory: the first is
    done and can be released, which lets the second go on."""
    import torch
    spec = _spec()
    ctx.set_bin_bytes(0)
    alone = M.Scene(ctx, spec)
    alone.step(3)
    want = list(alone.get_state())
    alone.close()
    short, long = M.Scene(ctx, spec), M.Scene(ctx, spec)
    batch = M.Batch(ctx, 3)
    a, b = batch.admit(short, 3, False), batch.admit(long, 6, True)
    batch.tick(1)  # the forward half's arrays
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 16 * MB, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(M.MPMError) as e:
            batch.tick(20)  # the reverse half's node blocks take 28 MB
        assert e.value.status == -2
        assert batch.poll(a) and not batch.poll(b)
        _same(list(short.get_state()), want)
        batch.release(a)
        short.close()
    finally:
        del fill
        torch.cuda.empty_cache()
    while not batch.poll(b):
        batch.tick(5)
    single = M.Scene(ctx, spec)
    single.rollout(6, 1)
    seed = np.zeros((single.N, 3))
    seed[:, 0] = 1.0 / single.N
    ref = list(single.get_state()) + list(single.backward(seed))
    _same(list(long.get_state()) + list(long.gradients()), ref)
    batch.close()
    for sc in (long, single):
        sc.close()


def test_bins_yield_to_what_a_scene_cannot_do_without(M, ctx):
    """A scene whose other arrays fit beside no bins is created without them; a rollout's states take the
    memory of the reverse pass's further sets."""
    import torch
    spec = _spec()
    sc = M.Scene(ctx, spec)
    want = _pass(sc, spec, 6, 2)
    held, size = ctx.bin_bytes()[0], sc.info()["state_bytes"]  # three sets

    def fill(leave):
        torch.cuda.empty_cache()
        return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")

    hold = fill(16 * MB)
    T = 64 * MB // size
    got = _pass(sc, spec, T, 1)  # 64 MB of states
    del hold
    torch.cuda.empty_cache()
    assert ctx.bin_bytes()[0] < held
    other = M.Scene(ctx, spec)
    _same(_pass(other, spec, T, 1), got)
    other.close()
    _same(_pass(sc, spec, 6, 2), want)
    sc.close()
    hold = fill(150 * MB)  # the bins alone would fit (134 MB), not with the 40 MB of the rest
    try:
        sc = M.Scene(ctx, spec)
        assert ctx.bin_bytes()[0] == 0
        sc.step(6)
        _same(list(sc.get_state()), want[:4])
        sc.close()
    finally:
        del hold
        torch.cuda.empty_cache()
