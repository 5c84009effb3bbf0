"""Launches with more CTAs than occupied tiles: most CTAs of P2G, G2P and the adjoint gather get no tile
and leave with what they requested on arrival.  The same body gives the same bits whether its grid is
binned (at most 4096 tiles) or sorted, and a tile over capacity is reported and harms no later scene."""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
def test_a_body_of_few_tiles_among_idle_ctas(dim):
    import torch
    from paper_1810_01054_gb300 import mpm as M
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blob = dict(radius_cells=3.0, v_scale=0.5, c_scale=0.5, f_scale=0.02, n_groups=64, amp=2.0, bc_width=3,
                center=[0.4] * dim, dt=1e-3)
    grids = [(256, 256), (260, 256)] if dim == 2 else [(64, 64, 64), (68, 64, 64)]
    spec = S.blob(dim, 64, 400, 91, **blob).copy(tile_edge=4 if dim == 2 else 0)
    t = np.floor(np.asarray(spec.x0) / spec.dx - 0.5).astype(int) // 4
    assert len(np.unique(t, axis=0)) < sms // 4
    dense = S.blob(dim, 64, 9000, 92, **dict(blob, radius_cells=0.4))  # one or two tiles, over capacity
    dense = dense.copy(tile_edge=4 if dim == 2 else 0)
    seed = np.full((400, dim), 1.0 / 400)
    ctx = M.Context(0)
    res = []
    for n in grids:
        for _ in range(2):
            sc = M.Scene(ctx, spec.copy(n_grid=n))
            sc.rollout(9, 4)
            res.append(list(sc.get_state()) + list(sc.backward(seed)))
            sc.close()
            over = M.Scene(ctx, dense.copy(n_grid=n))
            over.rollout(3, 1)
            with pytest.raises(M.MPMError) as e:
                over.backward(np.full((9000, dim), 1.0 / 9000))
            assert e.value.status == -8
            over.close()
    ctx.close()
    assert np.abs(res[0][-1]).max() > 0
    for r in res[1:]:
        for a, b in zip(res[0], r):
            assert np.array_equal(a, b)
