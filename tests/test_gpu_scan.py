"""The one-launch scan and the grouping by worker at the sizes where their
tiles and digits change (2048 items; 256 workers), through the step's records."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _apart(sizes):
    """scenes of spheres 3 m apart over a plane each lies on: body b has the one contact (b, plane)"""
    from paper_2403_17261_gb300 import scenes as S
    parts = []
    for n, k in sizes:
        pos = np.stack([3.0 * np.arange(n), np.zeros(n), np.full(n, 0.5)], axis=1)
        parts.append(S._single("row", pos, np.full(n, 0.5), np.ones(n), [[0, 0, 1, 0]], mu=0.5, dt=1 / 60, flags=1, gamma=1,
                               beta=2, n_sets=k, set_of_body=np.arange(n) % k, iters=2))
    return S.concat_scenes("rows", parts, iters=2)


@pytest.mark.parametrize("sizes", [
    [(1, 1)], [(7, 3)], [(2047, 1)], [(2048, 2)], [(2049, 64)], [(16384, 5)], [(16385, 64), (3, 1)],
    [(300, 64)] * 4,              # 256 workers
    [(300, 64)] * 4 + [(5, 1)],   # 257: two digits
    [(40, 20)] * 150 + [(70001, 64)],
])
def test_records(sizes):
    from paper_2403_17261_gb300 import ovl
    sc = _apart(sizes)
    sim = ovl.Simulation(sc, dict(lb_activate=0, lb_deact_every=0))
    base = np.cumsum([0] + [k for _, k in sizes])
    part = np.concatenate([base[i] + sc.set_of_body[sc.scene_of_body == i] for i in range(len(sizes))])
    for _ in range(2):                # the second step's scans run in the next epoch
        sim.step()
        st = sim.stats()
        n = sc.n_bodies
        assert (st["n_contacts"], st["n_entries"], st["n_pairs"], st["n_adjacency"]) == (n, n, n, 0)
        ab = sim.contacts()[0]
        assert np.array_equal(ab[:, 0], np.arange(n)) and np.array_equal(ab[:, 1], n + sc.scene_of_body)
        e = sim.entries()
        assert np.array_equal(e["entry_ptr"], np.arange(n + 1)) and np.array_equal(e["part"], part)
        order = np.argsort(part, kind="stable")
        p = sim.pairs()
        assert np.array_equal(p["part"], part[order])
        assert np.array_equal(p["key"] >> np.uint64(32), order.astype(np.uint64))
    sim.close()
