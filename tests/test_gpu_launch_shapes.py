"""Launches whose CTAs share an SM: the kernel they take and that it computes
the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pile(side, rng):
    """side x side x 3 spheres, two workers"""
    from paper_2403_17261_gb300 import scenes as S
    pos = S._lattice_pile(side, side, 3, 1.0, 0.5, 0.01, rng)
    n = pos.shape[0]
    return S._single("p", pos, np.full(n, 0.5), np.ones(n), [[0, 0, 1, 0]], mu=0.5, dt=1 / 60, flags=1, gamma=1, beta=4, n_sets=2,
                     set_of_body=(np.arange(n) * 2) // n)


def _batch(n_scenes, iters=8):
    """small piles of uneven sizes"""
    from paper_2403_17261_gb300 import scenes as S
    rng = S.SplitMix64(3)
    sc = S.concat_scenes("batch", [_pile(2 + k % 5, rng) for k in range(n_scenes)], iters=iters)
    sc.state[:, 7:13] = rng.uniform(6 * sc.n_bodies, -0.3, 0.3).reshape(-1, 6).astype(np.float32)
    return sc


def _run(sc, par, steps=2):
    from paper_2403_17261_gb300 import ovl
    sim = ovl.Simulation(sc, par)
    for _ in range(steps):
        sim.step()
    out, st = sim.state(), sim.stats()
    sim.close()
    return out.view(np.uint32), st


@pytest.mark.parametrize("par,masses", [
    (dict(pgs_cluster=1), False),                     # 512 threads: twice as many CTAs without the masses
    (dict(pgs_cluster=2), False),
    (dict(pgs_threads=256), False),
    (dict(pgs_cluster=1, pgs_threads=32), True),      # registers for all that are there
])
def test_shared_sms(par, masses):
    sc = _batch(350)
    ref, st = _run(sc, {})
    assert st["solve_ctas_masses"] == st["solve_ctas"]
    out, st = _run(sc, par)
    assert np.array_equal(out, ref)
    assert st["solve_ctas_masses"] == (st["solve_ctas"] if masses else 0)


def test_box_batch():
    """more workers of boxes than SMs: two CTAs per SM, full rows staged, the bits of one CTA per SM"""
    from paper_2403_17261_gb300 import scenes as S
    parts = [S.box_building(seed=7 + k, storeys=1, cells=1 + k % 3, n_sets=2, iters=8) for k in range(90)]
    sc = S.concat_scenes("boxes", parts, iters=8)
    sc.half_extents = np.concatenate([p.half_extents for p in parts]).astype(np.float32)
    ref, st = _run(sc, {}, 3)
    assert st["solve_ctas_masses"] == st["solve_ctas"] >= 180
    for par in (dict(smem_slot_limit=5000), dict(pgs_cluster=2), dict(pgs_threads=32), dict(pgs_cluster=1, pgs_threads=512)):
        out, _ = _run(sc, par, 3)
        assert np.array_equal(out, ref), par


def _with_boxes(sc, share, seed=5):
    """turns a share of a pile's spheres into cubes of their width (the radius then bounds the cube)"""
    from paper_2403_17261_gb300 import scenes as S
    rng = S.SplitMix64(seed)
    pick = rng.uniform(sc.n_bodies) < share
    sc.half_extents = np.where(pick[:, None], 0.9 * sc.radius[:, None], 0.0).repeat(3, 1).astype(np.float32)
    sc.radius = np.where(pick, 1.6 * sc.radius, sc.radius).astype(np.float32)
    return sc


@pytest.mark.parametrize("n_scenes", [1, 60])
def test_workers_with_no_few_and_many_boxes(n_scenes):
    """one context with all kinds of workers, on one CTA per SM and on two, in clusters and without the masses"""
    from paper_2403_17261_gb300 import scenes as S
    rng = S.SplitMix64(7)
    parts = [_with_boxes(_pile(side, rng), share, 5 + j) for share in (0.0, 0.02, 0.3, 1.0) for j in range(n_scenes)
             for side in ((4, 5) if n_scenes > 1 else (9, 22))]
    he = np.concatenate([p.half_extents for p in parts])
    sc = S.concat_scenes("kinds", parts, iters=8)
    sc.half_extents = he
    sc.state[:, 7:13] = rng.uniform(6 * sc.n_bodies, -0.3, 0.3).reshape(-1, 6).astype(np.float32)
    ref, st = _run(sc, {}, 3)
    assert st["solve_ctas_masses"] == st["solve_ctas"]
    for par in (dict(smem_slot_limit=5000), dict(pgs_cluster=2), dict(pgs_cluster=1, pgs_threads=64), dict(pgs_cluster=4, smem_slot_limit=10)):
        out, _ = _run(sc, par, 3)
        assert np.array_equal(out, ref), par


def test_stats_name_the_launch():
    """threads and rows at once as the kernels ran them, not as the plan's shape table has them"""
    from paper_2403_17261_gb300 import scenes as S
    seen = lambda sc, par: tuple(_run(sc, par, 1)[1][k] for k in ("solve_threads", "solve_rows_per_thread"))
    pile, building = S.pile_small(), S.box_building(storeys=2, cells=3, n_sets=3, iters=4)
    assert seen(pile, {}) == (512, 1)
    assert seen(pile, dict(pgs_threads=1024)) == (512, 1)
    assert seen(pile, dict(pgs_threads=96)) == (96, 1)
    assert seen(pile, dict(smem_slot_limit=5000)) == (512, 2)
    assert seen(building, {}) == (256, 1)
    assert seen(building, dict(pgs_cluster=1)) == (128, 1)
    assert seen(building, dict(smem_slot_limit=5000)) == (512, 2)
    assert seen(_batch(350), {}) == (128, 1)


@pytest.mark.parametrize("boxes,most", [(False, 11), (True, 15)])
def test_autotuner_times_a_launch_once(boxes, most):
    """four cluster sizes, two thread counts and two row counts come to the same launches where the masses are kept: one row at
    a time, room enough with one CTA per SM or two; for boxes 128 threads where two share an SM, 256 and 512 the same otherwise.
    A candidate is three kernels (row order, row build, solve); three plans are timed too."""
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    sc = S.box_building(storeys=2, cells=3, n_sets=3, iters=4) if boxes else S.pile_small()
    sim = ovl.Simulation(sc, dict(flags=ovl.OVL_FLAG_AUTOTUNE))
    state = sim.state()
    n = []
    for _ in range(2):
        sim.set_state(state)
        sim.set_step_index(0)
        sim.step()
        n.append(sim.stats()["n_launches"])
    sim.close()
    assert n[0] - n[1] <= 3 * most + 3


@pytest.mark.parametrize("share", [0.0, 0.01])
def test_impulses_in_global_memory(share):
    """the masses in shared memory, the impulses not: two CTAs of some 5000 bodies and 10,000 rows each, spheres alone or with a
    few boxes.  One slot per body and 12 B per row are more than the 229,888 B a CTA may use."""
    from paper_2403_17261_gb300 import scenes as S
    rng = S.SplitMix64(11)
    pos = S._lattice_pile(22, 22, 21, 1.0, 0.5, 0.02, rng)
    n = pos.shape[0]
    sc = S._single("pile", pos, rng.uniform(n, 0.45, 0.52), rng.uniform(n, 0.5, 2.0), [[0, 0, 1, 0]], mu=0.5, dt=1 / 60, flags=1,
                   gamma=1, beta=4, n_sets=1, set_of_body=np.zeros(n, int), iters=12)
    sc.state[:, 7:13] = rng.uniform(6 * n, -0.3, 0.3).reshape(n, 6).astype(np.float32)
    if share:
        sc = _with_boxes(sc, share)
    out, st = _run(sc, dict(pgs_cluster=2))
    assert st["solve_ctas_masses"] == st["solve_ctas"] == 2
    assert 32 * (n // 2 + 1) + 12 * (st["n_pairs"] // 2) > 229888
    for par in ({}, dict(pgs_cluster=8), dict(pgs_cluster=4, smem_slot_limit=6000)):
        other, st = _run(sc, par)
        assert np.array_equal(other, out), par
