"""The pair search against brute force: one thread and eight threads per body,
hash tables so small that columns wrap, neighbours beyond the list in shared
memory, several scenes in one table, static bodies."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _cloud(n, seed, box, lo, hi, static=0, big=None):
    from paper_2403_17261_gb300 import scenes as S
    rng = np.random.default_rng(seed)
    pos = rng.uniform(-box, box, (n, 3))
    r = rng.uniform(lo, hi, n)
    if big is not None:
        pos[0], r[0] = 0.0, big
    im = np.ones(n)
    im[n - static:] = 0.0
    return S._single("cloud", pos, r, im, [[0, 0, 1, -0.5 * box], [1, 0, 0, -0.7 * box]], mu=0.5, dt=1 / 60, flags=1, gamma=0,
                     beta=2, n_sets=1, set_of_body=np.zeros(n), iters=0)


def _brute(sc, margin):
    f = np.float32
    x, r, n = sc.state[:, :3].astype(f), sc.radius.astype(f), sc.n_bodies
    out = []
    for a in range(n):
        dyn = sc.inv_mass[a] > 0
        b = np.arange(a + 1, n)
        d = x[b] - x[a]
        d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        rs = (r[a] + r[b]) + f(margin)
        hit = (d2 <= rs * rs) & (sc.scene_of_body[b] == sc.scene_of_body[a]) & (dyn | (sc.inv_mass[b] > 0))
        out += [(a, int(k)) for k in b[hit]]
        if dyn:
            for k, p in enumerate(sc.planes.astype(f)):
                if sc.plane_scene[k] == sc.scene_of_body[a]:
                    g = (((p[0] * x[a, 0] + p[1] * x[a, 1]) + p[2] * x[a, 2]) - p[3]) - r[a]
                    if g <= f(margin):
                        out.append((a, n + k))
    return np.array(out, np.int32).reshape(-1, 2)


@pytest.mark.parametrize("make", [
    lambda S: _cloud(1, 0, 1.0, 0.1, 0.2),
    lambda S: _cloud(2, 1, 0.2, 0.1, 0.2),
    lambda S: _cloud(5, 2, 0.3, 0.1, 0.2),
    lambda S: _cloud(700, 3, 2.5, 0.1, 0.3, static=60),
    lambda S: _cloud(3000, 4, 3.0, 0.08, 0.1, big=2.0),    # a body with over 128 neighbours
    lambda S: S.concat_scenes("two", [_cloud(400, 5, 1.5, 0.1, 0.2), _cloud(300, 6, 1.5, 0.05, 0.2)], iters=0),
])
@pytest.mark.parametrize("copies", [1, 0])
def test_pairs(make, copies):
    """copies = 0: the scene beside 40,000 bodies far apart, so that one thread per body searches"""
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    sc = make(S)
    want = _brute(sc, 0.05)
    n = sc.n_bodies
    if not copies:
        m = 40000
        pos = np.stack([10.0 * np.arange(m), np.full(m, 500.0), np.zeros(m)], axis=1)
        far = S._single("far", pos, np.full(m, 0.1), np.ones(m), np.zeros((0, 4)), mu=0.5, dt=1 / 60, flags=1, gamma=0, beta=2,
                        n_sets=1, set_of_body=np.zeros(m), iters=0)
        parts = [sc, far]
        merged = S.concat_scenes("both", parts, iters=0)
        merged.scene_of_body = np.concatenate([sc.scene_of_body, np.full(m, sc.n_scenes)]).astype(np.int32)
        for k in ("scene_mu", "scene_dt", "scene_flags", "scene_gamma", "scene_beta", "n_sets"):
            setattr(merged, k, np.concatenate([getattr(sc, k), getattr(far, k)]))
        merged.plane_scene = sc.plane_scene.copy()
        want = np.where(want >= n, want + m, want)
        sc = merged
    sim = ovl.Simulation(sc, dict(lb_activate=0, lb_deact_every=0))
    sim.set_state(sc.state)
    sim.load_balance(0)          # contacts and graph of the state, nothing else
    try:
        sim.step(iters=0)
    except ovl.OvlError as e:    # bodies in deep overlap may exceed a worker's colours; the contacts stand
        assert e.code == ovl.OVL_ERR_CAPACITY
    got = sim.contacts()[0]
    assert np.array_equal(got, want)
    sim.close()
