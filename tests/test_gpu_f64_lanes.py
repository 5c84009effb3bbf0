"""The FP64 form's particle kernels give three lanes of a warp to a particle in small scenes (up to 32
particles an SM) and a thread beyond; both against the FP64 oracle around the line and at partly
filled warps (ten particles a warp).  FP64 on both sides: the tolerance is the parity tests' 1e-9,
orders above the summation-order differences (1e-13) and below any dropped term (1e-6)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1810_01054_gb300 import scenes as S
from tests.parity_utils import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("count", ["1", "9", "10", "11", "32", "line", "line+1"])
def test_lanes_against_oracle(dim, count):
    import torch
    from paper_1810_01054_gb300 import mpm as M
    line = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    N = {"line": line, "line+1": line + 1}.get(count) or int(count)
    spec = S.blob(dim, 48, N, 71, radius_cells=14.0 if dim == 2 else 8.0, v_scale=0.3, c_scale=0.5, f_scale=0.03,
                  ctrl_type=S.CTRL_TABLE, hidden=3, n_groups=2, amp=2.0, dt=1e-3)
    ctx = M.Context(0)
    sc = M.Scene64(ctx, spec)
    T = 3
    sc.rollout(T)
    rng = np.random.default_rng(72)
    seeds = [rng.normal(size=(N, dim)), rng.normal(size=(N, dim)), rng.normal(size=(N, dim, dim)),
             rng.normal(size=(N, dim, dim))]
    got = list(sc.get_state()) + list(sc.backward(*seeds))
    sc.close()
    ctx.close()
    osc = O.Scene(spec)
    traj = osc.rollout(T)
    want = [t[T] for t in traj[:4]] + list(osc.backward(traj, seeds))
    for k, (a, b) in enumerate(zip(got, want)):
        assert rel_l2(a, np.asarray(b).reshape(np.shape(a))) <= 1e-9, k
