"""The packed operands follow the parameters: set, trained, loaded."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _sim(theta=None):
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    sim = ovl.Simulation(S.resting_sphere())
    f, t = S.synthetic_rows(700)
    sim.log_reserve(700)
    sim.log_append(f, t)
    if theta is not None:
        sim.mlp_set_params(theta)
    return sim, f


def _seen(sim, f):
    g = sim.mlp_grad(0, 700)
    return [np.float64(sim.mlp_loss(0, 700)), *(np.asarray(x) for x in g), sim.mlp_forward(f[:130])]


@pytest.mark.parametrize("steps", [0, 1, 120])
def test_operands_are_the_parameters(steps):
    from paper_2403_17261_gb300 import scenes as S
    sim, f = _sim(S.mlp_init_params(seed=5))
    sim.mlp_train(0, 700, 300, steps, seed=3)
    got = _seen(sim, f)
    fresh, _ = _sim(sim.mlp_params())                       # the trained parameters, set anew
    loaded, _ = _sim(S.mlp_init_params(seed=6))
    loaded.load(sim.save())
    for other in (fresh, loaded):
        for a, b in zip(got, _seen(other, f)):
            assert np.array_equal(a, b)
    sim.mlp_set_params(S.mlp_init_params(seed=7))           # and other parameters after training
    again, _ = _sim(S.mlp_init_params(seed=7))
    for a, b in zip(_seen(sim, f), _seen(again, f)):
        assert np.array_equal(a, b)
    for s in (sim, fresh, loaded, again):
        s.close()
