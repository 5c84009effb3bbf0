"""A batch without a memory budget keeps every state of a gradient request while the context's scenes hold
at most 4 GiB of such states between them; a scene holds its states after its request has left."""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def test_states_held_after_their_requests_count():
    import torch
    from paper_1810_01054_gb300 import mpm as M
    MB = 1 << 20
    N, T = 100000, 50
    spec = S.blob(2, 128, N, 131, radius_cells=50.0, n_groups=1, dt=1e-4, bc_width=3)
    ctx = M.Context(0)
    scenes = [M.Scene(ctx, spec) for _ in range(20)]
    one = T * scenes[0].info()["state_bytes"]  # 229 MB: 17 scenes' states fit
    most = 4 * 1024 * MB // one
    assert 2 < most < 19 and one < 256 * MB
    batch = M.Batch(ctx, 2)

    def run(sc):
        free = torch.cuda.mem_get_info()[0]
        slot = batch.admit(sc, T, True)
        while not batch.poll(slot):
            batch.tick(T)
        batch.release(slot)
        return free - torch.cuda.mem_get_info()[0], list(sc.get_state()) + list(sc.gradients())

    runs = [run(sc) for sc in scenes]
    kept = [took > 0.9 * one for took, _ in runs]
    assert kept == [True] * most + [False] * (20 - most)
    for _, got in runs[1:]:
        for a, b in zip(got, runs[0][1]):
            assert np.array_equal(a, b)
    scenes[0].close()  # its states are free again: the next scene may keep its own
    assert run(scenes[-1])[0] > 0.5 * one
    again = run(scenes[1])  # and a scene that holds its states goes on with them
    assert again[0] < MB
    batch.close()
    for sc in scenes[1:]:
        sc.close()
    ctx.close()
