"""Controller parameters set right before a call are the ones that call uses, whatever stream the
context has and wherever the array lives: the upload is ordered with the kernels that read it and with
the work that produces a device array."""
import numpy as np
import pytest

from paper_1810_01054_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _late(torch, values):
    """A device tensor whose values the current stream writes only behind some milliseconds of work."""
    t = torch.full((len(values),), 7.0, device="cuda")
    src = torch.as_tensor(np.asarray(values, np.float32), device="cuda")
    a = torch.randn(4096, 4096, device="cuda")
    torch.cuda.current_stream().synchronize()
    for _ in range(8):
        a = torch.mm(a, a).clamp_(-1.0, 1.0)
    t.copy_(src)
    return t


@pytest.mark.parametrize("ctrl", [S.CTRL_SIN, S.CTRL_BASIS, S.CTRL_MLP, S.CTRL_TABLE, S.CTRL_COM])
@pytest.mark.parametrize("stream", ["private", "side", "default"])
def test_upload_is_ordered_with_its_readers(ctrl, stream):
    import torch
    from paper_1810_01054_gb300 import mpm as M
    spec = S.blob(2, 32, 900, 81, radius_cells=6.0, v_scale=0.5, c_scale=0.5, f_scale=0.02, ctrl_type=ctrl,
                  hidden=8, n_groups=3, amp=2.0, dt=5e-4)
    rng = np.random.default_rng(82)
    sets = [rng.normal(size=np.asarray(spec.ctrl_params).size).astype(np.float32) for _ in range(3)]
    T, seed = 7, np.full((spec.n_particles, 2), 1.0 / spec.n_particles)

    def result(sc):
        sc.rollout(T, 3)
        return list(sc.get_state()) + list(sc.backward(seed))

    side = torch.cuda.Stream()
    ctx = M.Context(0, stream={"private": None, "side": side, "default": torch.cuda.default_stream()}[stream])
    want = []
    for p in sets:
        fresh = M.Scene(ctx, spec, params=p)
        want.append(result(fresh))
        fresh.close()
    assert any(not np.array_equal(a, b) for a, b in zip(want[0], want[1]))
    sc = M.Scene(ctx, spec)
    with torch.cuda.stream(side if stream == "side" else torch.cuda.default_stream()):
        for p, ref in list(zip(sets, want)) * 2:
            for source in ("host", "device"):
                sc.set_state(spec.x0, spec.v0, spec.C0, spec.F0, step=0)
                sc.step(5)  # work in flight when the parameters change
                t = p.copy() if source == "host" else _late(torch, p)
                sc.set_state(spec.x0, spec.v0, spec.C0, spec.F0, step=0)
                sc.set_params(t)
                t[:] = 1e3  # the caller's array is its own again
                for a, b in zip(result(sc), ref):
                    assert np.array_equal(a, b), source
    sc.close()
    ctx.close()
