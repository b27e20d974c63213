"""The solve's row paths agree: impulses in shared memory or in global memory,
rows local to a CTA or reaching another one of its cluster, colour buckets
around multiples of a warp and of the CTA, joints in clusters."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pile(nx, ny, nz, n_sets):
    from paper_2403_17261_gb300 import scenes as S
    rng = S.SplitMix64(11)
    pos = S._lattice_pile(nx, ny, nz, 1.0, 0.5, 0.02, rng)
    n = pos.shape[0]
    sets = (np.argsort(np.argsort(pos[:, 0], kind="stable")) * n_sets) // n
    sc = S._single("pile", pos, rng.uniform(n, 0.45, 0.52), rng.uniform(n, 0.5, 2.0), [[0, 0, 1, 0]], mu=0.5, dt=1 / 60,
                   flags=1, gamma=1, beta=4, n_sets=n_sets, set_of_body=sets, iters=12)
    sc.state[:, 7:13] = rng.uniform(6 * n, -0.3, 0.3).reshape(n, 6).astype(np.float32)
    return sc


@pytest.mark.parametrize("shape,n_sets", [
    ((2, 1, 1), 1),       # one contact
    ((4, 4, 4), 1),       # buckets of a few rows
    ((8, 8, 8), 3),
    ((11, 11, 13), 1),    # buckets around one and two passes of a CTA
    ((19, 19, 19), 1),    # 6859 bodies in one CTA: the impulses do not fit beside them
])
def test_paths_agree(shape, n_sets):
    from oracle import oracle as O
    from paper_2403_17261_gb300 import ovl
    sc = _pile(*shape, n_sets)
    out = {}
    for name, par in (("plan", {}), ("c1", dict(pgs_cluster=1)), ("c2", dict(pgs_cluster=2)), ("c8", dict(pgs_cluster=8)),
                      ("t96", dict(pgs_cluster=4, pgs_threads=96)), ("plain", dict(pgs_cluster=4, smem_slot_limit=6000))):
        sim = ovl.Simulation(sc, par)
        sim.step()
        sim.step()                      # warm-started rows
        out[name] = sim.state()
        sim.close()
    for name, st in out.items():
        assert np.array_equal(st.view(np.uint32), out["plan"].view(np.uint32)), name
    orc = O.OracleSim(sc)
    orc.step()
    state, warm, masks = orc.state().astype(np.float32), orc.warmstart(), orc.masks()
    sim = ovl.Simulation(sc)
    sim.set_state(state)
    sim.set_membership(masks)
    sim.set_warmstart(warm[0], warm[1], np.asarray(warm[2], np.float32))
    sim.set_step_index(1)
    sim.step()
    orc.set_state(state.astype(np.float64))
    orc.set_warmstart(warm[0], warm[1], np.asarray(warm[2], np.float32).astype(np.float64))
    orc.step()
    assert np.abs(sim.state()[:, 7:13] - orc.state()[:, 7:13]).max() <= 1e-4
    sim.close()


@pytest.mark.parametrize("links,n_sets", [(3, 1), (257, 2), (2500, 1)])
def test_joint_rows_agree(links, n_sets):
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    sc = S.chain(n=links, n_sets=n_sets, iters=15)
    out = []
    for par in ({}, dict(pgs_cluster=1), dict(pgs_cluster=2), dict(pgs_cluster=8), dict(smem_slot_limit=4000)):
        sim = ovl.Simulation(sc, par)
        for _ in range(3):
            sim.step()
        out.append(sim.state())
        sim.close()
    for st in out[1:]:
        assert np.array_equal(st.view(np.uint32), out[0].view(np.uint32))


@pytest.mark.parametrize("scene", ["building", "bridge", "wide"])
def test_box_rows_agree(scene):
    """full rows staged a colour ahead, straight from memory (buckets beyond a CTA's threads), in clusters, and with the
    masses in the rows"""
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    sc = {"building": lambda: S.box_building(storeys=2, cells=3, n_sets=3, iters=10),
          "bridge": lambda: S.plank_bridge(planks=40, n_sets=2, iters=10),
          "wide": lambda: S.box_building(storeys=1, cells=24, n_sets=1, iters=6)}[scene]()
    out = []
    for par in ({}, dict(pgs_cluster=1), dict(pgs_cluster=4), dict(pgs_cluster=2, pgs_threads=32), dict(smem_slot_limit=5000)):
        sim = ovl.Simulation(sc, par)
        for _ in range(3):
            sim.step()
        out.append(sim.state())
        sim.close()
    for st in out[1:]:
        assert np.array_equal(st.view(np.uint32), out[0].view(np.uint32))
