"""Scenes and batches of at most 2048 tiles that have no tile bins: the tile scan is part of the scatter, so
the sort is one launch a step (three beyond), and the results are the bits of the bins."""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _spec(dim, grid, edge, ctrl=S.CTRL_SIN):
    s = S.blob(dim, 64, 2500, 111, radius_cells=9.0 if dim == 2 else 6.0, v_scale=1.0, c_scale=1.0, f_scale=0.03,
               center=[0.35] * dim, ctrl_type=ctrl, hidden=8, n_groups=3, amp=2.0, bc_width=3, dt=2e-3)
    v = np.array(s.v0)
    v[:, 0] += 3.0  # 0.4 cells a step: particles change tiles
    return s.copy(n_grid=grid, v0=v, tile_edge=edge if dim == 2 else 0)


# (dim, grid, tile edge, launches of the sort): 768, 2048 and 2080 tiles in 2D; 1728 and 2197 in 3D
GRIDS = [(2, (128, 96), 4, 1), (2, (256, 128), 4, 1), (2, (512, 256), 8, 1), (2, (260, 128), 4, 3),
         (3, (48, 48, 48), 4, 1), (3, (52, 52, 52), 4, 3)]


@pytest.mark.parametrize("ctrl", [S.CTRL_SIN, S.CTRL_MLP])
@pytest.mark.parametrize("dim,grid,edge,sorts", GRIDS)
def test_one_sort_launch_and_the_bits_of_the_bins(dim, grid, edge, sorts, ctrl):
    from paper_1810_01054_gb300 import mpm as M
    spec = _spec(dim, grid, edge, ctrl)
    res = []
    for most in (None, 0):
        ctx = M.Context(0)
        if most is not None:
            ctx.set_bin_bytes(most)
        sc = M.Scene(ctx, spec)
        sc.set_tuning(M.TUNE_OFF)
        got = []
        for T, k in ((11, 1), (11, 4), (3, 2)):
            sc.rollout(T, k)
            got += list(sc.get_state()) + list(sc.backward(np.full((sc.N, dim), 1.0 / sc.N)))
        n0 = M.launch_count()
        sc.step(8)
        launches = M.launch_count() - n0
        got += list(sc.get_state())
        # P2G and G2P, the state-reading controller's two, and the sort (with bins one selection a call)
        tiles = 2 + (2 if ctrl == S.CTRL_MLP else 0)
        assert launches == 8 * (tiles + sorts) if most == 0 else launches == 8 * tiles + 1
        sc.close()
        batch_of = [M.Scene(ctx, spec) for _ in range(2)]  # a batch of twice the tiles
        batch = M.Batch(ctx, dim)
        slots = [batch.admit(s, 9, True) for s in batch_of]
        while not all(batch.poll(sl) for sl in slots):
            batch.tick(4)
        for s in batch_of:
            got += list(s.get_state()) + list(s.gradients())
        batch.close()
        ctx.close()
        res.append(got)
    for a, b in zip(*res):
        assert np.array_equal(a, b)
