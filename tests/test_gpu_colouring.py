"""The colouring where its paths change: lists with their queues in shared or
in global memory, rounds in clusters and in global memory, joints, priorities
that tie in their high word."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _mix(z):
    with np.errstate(over="ignore"):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _greedy(keys, ends):
    """first-fit colours in descending priority; ends: dynamic bodies of every constraint"""
    colour, used = np.zeros(len(keys), int), {}
    for i in np.argsort(_mix(keys))[::-1]:
        taken = set().union(*(used.setdefault(b, set()) for b in ends[i]))
        c = next(c for c in range(1000) if c not in taken)
        colour[i] = c
        for b in ends[i]:
            used[b].add(c)
    return colour


@pytest.mark.parametrize("cluster", [0, 1, 2, 3])
def test_tied_high_words(cluster):
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    n = 300000
    top = (_mix(np.arange(1, n, dtype=np.uint64) << np.uint64(2)) >> np.uint64(32)).astype(np.uint32)
    order = np.argsort(top, kind="stable")
    same = np.nonzero(top[order][1:] == top[order][:-1])[0]
    b1, b2 = sorted(int(order[same[0] + k]) + 1 for k in (0, 1))   # contacts (0, b1), (0, b2) tie
    pos = np.stack([5.0 * (np.arange(n) % 600), 5.0 * (np.arange(n) // 600), np.full(n, 50.0)], axis=1)
    pos[0] = (0, 0, 0)
    pos[b1], pos[b2] = (-1, 0, 0), (1, 0, 0)
    im = np.zeros(n)
    im[[0, b1, b2]] = 1.0
    sc = S._single("tie", pos, np.full(n, 0.5), im, np.zeros((0, 4)), mu=0.5, dt=1 / 60, flags=1, gamma=0, beta=2, n_sets=1,
                   set_of_body=np.zeros(n), iters=3)
    sim = ovl.Simulation(sc, dict(pgs_cluster=cluster) if cluster else {})
    sim.step()
    p = sim.pairs()
    want = np.array([b1, b2], np.uint64) << np.uint64(2)
    assert np.array_equal(p["key"], want)
    assert np.array_equal(p["colour"], _greedy(want, [(0, b1), (0, b2)]))
    sim.close()


@pytest.mark.parametrize("side,cluster,limit", [(1, 0, 0), (5, 0, 0), (13, 0, 0), (13, 1, 0), (13, 2, 0), (13, 8, 0), (20, 0, 0),
                                                (23, 0, 0), (24, 0, 0), (24, 4, 0), (13, 1, 64)])
def test_greedy(side, cluster, limit):
    """up to 13,824 bodies (about 33,000 constraints) in one worker: lists below 8,900 bodies with the queues in shared memory,
    below 13,000 in global memory; a fixed cluster size or a limit takes the rounds"""
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    rng = S.SplitMix64(3)
    pos = S._lattice_pile(side, side, side, 1.0, 0.5, 0.02, rng)
    n = pos.shape[0]
    first = np.arange(0, max(n - 40, 0), 7)
    j = np.stack([first, first + 40], axis=1)[: n // 9]
    sc = S._single("lattice", pos, rng.uniform(n, 0.46, 0.52), np.ones(n), [[0, 0, 1, 0]], mu=0.5, dt=1 / 60, flags=1, gamma=0,
                   beta=2, n_sets=1, set_of_body=np.zeros(n), joints=j, anchors=np.zeros((len(j), 6)), iters=1)
    par = dict(lb_activate=0, lb_deact_every=0)
    if cluster:
        par["pgs_cluster"] = cluster
    if limit:
        par["smem_slot_limit"] = limit
    sim = ovl.Simulation(sc, par)
    sim.step()
    p = sim.pairs()
    ends = []
    for k in p["key"]:
        if k >> np.uint64(62):
            ends.append(tuple(int(b) for b in j[int(k & np.uint64(0xffffffff))]))
        else:
            a, b = int(k >> np.uint64(32)), int(k & np.uint64(0xffffffff)) >> 2
            ends.append((a,) if b >= n else (a, b))
    assert np.array_equal(p["colour"], _greedy(p["key"], ends))
    sim.close()


def test_lists_beside_rounds():
    """workers of both kernels in one step: two of about 14,000 bodies, six small ones"""
    from paper_2403_17261_gb300 import ovl
    from paper_2403_17261_gb300 import scenes as S
    rng = S.SplitMix64(4)
    pos = S._lattice_pile(32, 32, 32, 1.0, 0.5, 0.02, rng)
    n = pos.shape[0]
    sets = np.where(np.arange(n) < 14500, 0, np.where(np.arange(n) < 29000, 1, 2 + (np.arange(n) - 29000) * 6 // (n - 29000)))
    sc = S._single("lattice", pos, rng.uniform(n, 0.46, 0.52), np.ones(n), [[0, 0, 1, 0]], mu=0.5, dt=1 / 60, flags=1, gamma=0,
                   beta=2, n_sets=8, set_of_body=sets, iters=1)
    sim = ovl.Simulation(sc, dict(lb_activate=0, lb_deact_every=0))
    for _ in range(3):
        sim.step()
        p = sim.pairs()
        for w in range(8):
            i = np.nonzero(p["part"] == w)[0]
            ends = []
            for k in p["key"][i]:
                a, b = int(k >> np.uint64(32)), int(k & np.uint64(0xffffffff)) >> 2
                ends.append((a,) if b >= n else (a, b))
            assert np.array_equal(p["colour"][i], _greedy(p["key"][i], ends)), w
    sim.close()
