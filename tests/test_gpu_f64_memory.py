"""The FP64 form's second pair of grids is a convenience: a scene, or a rollout's history, that the device
holds only without it still runs, with the same results (its grids are summed by atomics: FP64 rounding,
orders below the 1e-12 allowed)."""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S
from tests.parity_utils import rel_l2

pytestmark = pytest.mark.gpu


def test_without_room_for_the_second_pair():
    import torch
    from paper_1810_01054_gb300 import mpm as M
    MB = 1 << 20
    spec = S.blob(3, 100, 3000, 141, radius_cells=8.0, v_scale=0.3, c_scale=0.5, f_scale=0.03, bc_width=3, dt=5e-4,
                  ctrl_type=S.CTRL_TABLE, hidden=5, n_groups=2)
    pair = 8 * 8 * 100 ** 3  # 61 MiB of grids
    T = 5
    rng = np.random.default_rng(142)  # seeds of every part: under a uniform one dL/dC and dL/dF are zero
    seeds = [rng.normal(size=(3000, 3)), rng.normal(size=(3000, 3)), rng.normal(size=(3000, 3, 3)),
             rng.normal(size=(3000, 3, 3))]
    ctx = M.Context(0)

    def result(sc, T=T):
        sc.rollout(T)
        return list(sc.get_state()) + list(sc.backward(*seeds))

    def same(a, b):
        for x, y in zip(a, b):
            assert rel_l2(x, y) <= 1e-12

    sc = M.Scene64(ctx, spec)
    want = result(sc)
    sc.close()
    fills = []

    def leave(room):
        torch.cuda.empty_cache()
        fills.append(torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda"))

    try:
        leave(pair + pair // 2)  # one pair fits
        sc = M.Scene64(ctx, spec)
        same(result(sc), want)
        fills.clear()
        torch.cuda.empty_cache()
        same(result(sc), want)
        sc.close()
        sc = M.Scene64(ctx, spec)  # both pairs
        same(result(sc), want)
        long = pair * 3 // 4 // (24 * 8 * 3000)  # a history of 46 MiB
        leave(16 * MB)
        sc.rollout(long)  # takes the second pair's memory
        same(list(sc.get_state(T)), want[:4])
        same(result(sc), want)
        sc.close()
    finally:
        fills.clear()
        torch.cuda.empty_cache()
    ctx.close()
