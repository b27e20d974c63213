"""The training kernel at the edges of its 128-row tiles, and graph replays
against direct launches (50 Adam steps per replay)."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2403_17261_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 127, 128, 129, 4097])
def test_gradient_at_tile_edges(rows):
    import mlp_bounds as B
    from paper_2403_17261_gb300 import ovl
    sim = ovl.Simulation(S.resting_sphere())
    f, t = S.synthetic_rows(rows + 3, seed=rows)
    sim.log_reserve(rows + 3)
    sim.log_append(f, t)
    th = S.mlp_init_params(seed=2, bias_scale=0.2, bf16_exact=True)
    sim.mlp_set_params(th)
    loss, g = sim.mlp_grad(2, rows)
    X, T = f[2:2 + rows].astype(np.float64), t[2:2 + rows].astype(np.float64)
    L_ref, g_ref = M.grad(th.astype(np.float64), X, T)
    r = np.abs(g.astype(np.float64) - g_ref) / B.grad_tolerance(th.astype(np.float64), X, T)
    assert r.max() <= 1.0, (int(r.argmax()), float(r.max()))
    # the same forward values summed in FP32 and in FP64
    assert abs(loss - sim.mlp_loss(2, rows)) <= 1e-5 * loss
    sim.close()


def test_replay_equals_direct():
    """100 steps (two replays) and the same 100 steps in calls below the replay's length, on one full batch"""
    from paper_2403_17261_gb300 import ovl
    f, t = S.synthetic_rows(300, seed=5)
    out = []
    for calls in ((100,), (40, 60)):
        sim = ovl.Simulation(S.resting_sphere())
        sim.log_reserve(300)
        sim.log_append(f, t)
        sim.mlp_set_params(S.mlp_init_params(seed=4))
        loss = np.concatenate([sim.mlp_train(0, 300, 300, k, sampling=0) for k in calls])
        out.append((sim.mlp_params(), loss))
        sim.close()
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32))
    assert np.array_equal(out[0][1].view(np.uint32), out[1][1].view(np.uint32))
    assert out[0][1][-1] < out[0][1][0]
