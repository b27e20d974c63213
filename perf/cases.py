"""The work that users of this framework have it do, as timed cases.

A case is a dict of plain values; ``kind`` names the work:

* ``step``   one timestep of the method on one scene, from a state the caller
  holds on the device to a state the caller reads on the device (the call of a
  control loop or a renderer);
* ``period`` one load-balance period, ten timesteps of the large pile with the
  removal branches in the first of them;
* ``train``  training the learned warm start's network from given parameters
  on the rows of its log;
* ``infer``  the network alone on rows in host memory.

Piles are generated close to rest: staggered layers of jittered spheres of
radius U(0.4, 0.6) on the floor of a box, about three contacts per body, small
random velocities, workers in a grid of uneven blocks that overlap by
``reach`` metres.  Chains, the building and the bridge are the package's own
scenes with seeded masses and velocities.
"""
import math

import numpy as np
import torch

from paper_2403_17261_gb300 import ovl
from paper_2403_17261_gb300 import scenes as S

DT, GRAVITY, MARGIN, ERP, SLOP = 1.0 / 60.0, 9.81, 0.05, 0.2, 0.001


def _pile(name, nx, ny, nz, workers, **kw):
    """workers: 'wx,wy,wz' blocks of the initial partition"""
    c = dict(name=name, kind="step", scene="pile", nx=nx, ny=ny, nz=nz, workers=workers, reach=1.0, gamma=2, beta=6,
             iters=30, removals=False, learned=False, lb_contacts=False, uniform=False, big=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the 256-sphere, two-worker pile of the tests, where launches and waits are the time
        _pile("pile_256", 8, 8, 4, "2,1,1", gamma=1, beta=4, iters=20, removals=True),
        # ball joints only: the 4096-link hanging chain, 8 workers, 50 sweeps
        dict(name="chain_4096", kind="step", scene="chain", n=4096, workers=8, iters=50),
        # boxes: the building (2654 bodies, manifolds, up to 65 colours) and the jointed plank bridge
        dict(name="building", kind="step", scene="building", storeys=12, cells=10, workers=16, iters=30),
        dict(name="bridge", kind="step", scene="bridge", planks=1589, workers=8, iters=50),
        # an ordinary pile of ragged size, with the learned warm start (features and network) in the step
        _pile("pile_30k_learned", 31, 29, 33, "3,2,2", learned=True),
        # unequal contact counts under the contact load, removal branches in the step (two layers of big spheres)
        _pile("pile_mixed_removal", 64, 64, 8, "4,4,1", removals=True, lb_contacts=True, big=2),
        # the large pile of the benchmark, 262,144 bodies on 64 workers: most of its steps
        _pile("pile_large", 64, 64, 64, "4,4,4", reach=2.0),
        # the same late in its run, when the overlap has grown to nearly every body (about 5 M constraint pairs)
        _pile("pile_large_late", 64, 64, 64, "4,4,4", reach=9.0),
        # ten of its steps, removals in the first: what a second of simulation is made of
        dict(_pile("pile_large_period", 64, 64, 64, "4,4,4", reach=2.0), kind="period"),
        # 512 independent scenes (piles and chains of 64 to 16,384 bodies, 1 to 16 uneven workers each)
        dict(name="batch_512", kind="step", scene="batch", scenes=512, lo=64, hi=16384, iters=30),
        # training the learned warm start: 200 Adam steps of 4096 rows
        dict(name="train_4096x200", kind="train", rows=1 << 18, batch=4096, steps=200),
        # the network alone on host rows, as a program that evaluates it offline calls it
        dict(name="infer_host_300k", kind="infer", rows=300007),
    ]


def draw(rng):
    def loguniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    pick = rng.choice(["pile", "pile", "pile", "chain", "building", "bridge", "batch", "train", "infer"])
    if pick == "pile":
        n = loguniform(100, 262144)
        nz = max(2, min(64, int(round(n ** (1 / 3) * rng.uniform(0.5, 1.5)))))
        nx = max(2, int(round(math.sqrt(n / nz) * rng.uniform(0.8, 1.25))))
        ny = max(2, int(round(n / (nx * nz))))
        w = [rng.randint(1, max(1, min(4, d // 4))) for d in (nx, ny, nz)]
        big = rng.choice([0, 0, 0, 1]) if nx >= 16 and ny >= 16 else 0
        c = _pile("", nx, ny, nz, ",".join(map(str, w)), reach=round(rng.uniform(0.5, 5.0), 2), gamma=rng.randint(0, 2),
                  iters=rng.choice([10, 20, 30, 50]), removals=n < 60000 and rng.random() < 0.5,
                  learned=rng.random() < 0.25, lb_contacts=rng.random() < 0.25, uniform=rng.random() < 0.2, big=big)
        c["beta"] = 2 * c["gamma"] + 2
    elif pick == "chain":
        n = loguniform(64, 20000)
        c = dict(kind="step", scene="chain", n=n, workers=rng.randint(1, max(1, min(64, n // 16))), iters=rng.choice([20, 30, 50]))
    elif pick == "building":
        c = dict(kind="step", scene="building", storeys=rng.randint(1, 12), cells=rng.randint(2, 10), workers=rng.randint(1, 16),
                 iters=rng.choice([20, 30]))
    elif pick == "bridge":
        c = dict(kind="step", scene="bridge", planks=loguniform(16, 1589), workers=rng.randint(1, 8), iters=rng.choice([20, 50]))
    elif pick == "batch":
        c = dict(kind="step", scene="batch", scenes=loguniform(2, 256), lo=loguniform(16, 256), hi=loguniform(512, 16384), iters=30)
    elif pick == "train":
        c = dict(kind="train", rows=loguniform(5000, 1 << 18), batch=loguniform(100, 8192), steps=rng.randint(20, 200))
    else:
        c = dict(kind="infer", rows=loguniform(1, 1 << 20))
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------

def _scene(state, radius, inv_mass, planes, mu, dt, flags, gamma, beta, n_sets, sets, iters, joints=None, anchors=None,
           assign=False, name=""):
    n = state.shape[0]
    f, i = np.float32, np.int32
    pl = np.asarray(planes, np.float64).reshape(-1, 4).astype(f)
    return S.Scene(
        name=name, state=state.astype(f), radius=radius.astype(f), inv_mass=inv_mass.astype(f), planes=pl,
        plane_scene=np.zeros(len(pl), i), joints=np.zeros((0, 2), i) if joints is None else joints,
        anchors=np.zeros((0, 6), f) if anchors is None else anchors.astype(f), scene_of_body=np.zeros(n, i),
        scene_mu=np.array([mu], f), scene_dt=np.array([dt], f), scene_flags=np.array([flags], i),
        scene_gamma=np.array([gamma], i), scene_beta=np.array([beta], i), n_sets=np.array([n_sets], i),
        set_of_body=sets.astype(i), iters=iters, assign_overlap=assign)


def _at_rest(pos, rng, speed, spin):
    n = pos.shape[0]
    st = np.zeros((n, 13))
    st[:, 0:3] = pos
    q = rng.normal(size=(n, 4))
    st[:, 3:7] = q / np.linalg.norm(q, axis=1, keepdims=True)
    st[:, 7:10] = rng.normal(0.0, speed, (n, 3))
    st[:, 10:13] = rng.normal(0.0, spin, (n, 3))
    return st


def _layers(nx, ny, nz, sp, z0, rng):
    """staggered layers, spacing 1.04 sp in a layer and 0.76 sp between layers, jittered"""
    k, j, i = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    odd = 0.5 * (k % 2)
    pos = np.stack([(i - (nx - 1) / 2 + odd) * 1.04 * sp, (j - (ny - 1) / 2 + odd) * 1.04 * sp, z0 + 0.76 * sp * k], -1)
    pos = pos.reshape(-1, 3)
    return pos + rng.uniform(-0.03 * sp, 0.03 * sp, pos.shape)


def _pile_scene(c, seed):
    """the scene and its membership masks: a worker holds its block and what lies within `reach` of it"""
    rng = np.random.default_rng(seed)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    pos = _layers(nx, ny, nz, 1.0, 0.55, rng)
    r = rng.uniform(0.4, 0.6, len(pos))
    if c["big"]:
        bx, by = max(1, int(nx * 1.04 / 2.75)), max(1, int(ny * 1.04 / 2.75))
        big = _layers(bx, by, c["big"], 2.55, 1.27, rng)
        pos[:, 2] += big[:, 2].max() + 1.3
        pos, r = np.concatenate([big, pos]), np.concatenate([np.full(len(big), 1.25), r])
    m = (4.0 / 3.0) * math.pi * r ** 3
    half = np.abs(pos[:, :2]).max() + 1.5
    w = [int(x) for x in c["workers"].split(",")]
    axes, cell = [], []
    for k in range(3):
        lo, hi = pos[:, k].min() - 0.1, pos[:, k].max() + 0.1
        cut = lo + (hi - lo) * (np.arange(1, w[k]) + rng.uniform(-0.15, 0.15, w[k] - 1)) / w[k]
        edge = np.concatenate([[lo], cut, [hi]])
        axes.append([(pos[:, k] >= edge[i] - c["reach"]) & (pos[:, k] <= edge[i + 1] + c["reach"]) for i in range(w[k])])
        cell.append(np.clip(np.searchsorted(edge, pos[:, k], side="right") - 1, 0, w[k] - 1))
    masks = np.zeros(len(pos), np.uint64)
    for i in range(w[0]):
        for j in range(w[1]):
            xy = axes[0][i] & axes[1][j]
            for k in range(w[2]):
                masks |= (xy & axes[2][k]).astype(np.uint64) << np.uint64((i * w[1] + j) * w[2] + k)
    sets = (cell[0] * w[1] + cell[1]) * w[2] + cell[2]
    sc = _scene(_at_rest(pos, rng, 0.2, 0.5), r, 1.0 / m, S.box_planes(half), 0.6, DT, 1, c["gamma"], c["beta"],
                w[0] * w[1] * w[2], sets, c["iters"])
    return sc, masks


def _links(n, span, drop, ground_z, radius):
    """centres, joints and anchors of a U-shaped chain between two world anchors"""
    knots = np.array([[-span / 2, 0, 0], [-span / 2, 0, ground_z + radius], [span / 2, 0, ground_z + radius], [span / 2, 0, 0]])
    at = np.concatenate([[0.0], np.cumsum(np.linalg.norm(np.diff(knots, axis=0), axis=1))])
    s = (np.arange(n) + 1) * at[-1] / (n + 1)
    pos = np.stack([np.interp(s, at, knots[:, k]) for k in range(3)], 1)
    full = np.concatenate([knots[:1], pos, knots[3:]])
    piv = 0.5 * (full[:-1] + full[1:])
    joints = np.stack([np.arange(-1, n), np.append(np.arange(n), -1)], 1).astype(np.int32)
    anchors = np.concatenate([np.concatenate([piv[:1], piv[1:] - pos]), np.concatenate([piv[:-1] - pos, piv[-1:]])], 1)
    return pos, joints, anchors


def _chain_scene(n, workers, iters, rng, scale=1.0, gamma=2, sets=None):
    pos, joints, anchors = _links(n, 300.0 * scale, 50.0 * scale, -50.0 * scale, 0.1)
    st = _at_rest(pos, rng, 0.02, 0.02)
    st[:, 3:7] = (1, 0, 0, 0)
    sets = np.arange(n) * workers // n if sets is None else sets
    return _scene(st, np.full(n, 0.1), 1.0 / rng.uniform(0.5, 2.0, n), [[0, 0, 1, -50.0 * scale]], 0.5, 1.0 / 120.0, 0, gamma,
                  2 * gamma + 2, workers, sets, iters, joints, anchors, True)


def _cuts(rng, n, k):
    """n bodies in k uneven runs"""
    return np.searchsorted(np.sort(rng.uniform(0, n, k - 1)), np.arange(n), side="right")


def _batch_scene(c, seed):
    rng, sizes = np.random.default_rng(seed), np.random.default_rng(c["scenes"])   # the sizes belong to the case
    parts = []
    for s in range(c["scenes"]):
        n = int(round(math.exp(sizes.uniform(math.log(c["lo"]), math.log(c["hi"])))))
        k = min(int(sizes.integers(1, 17)), n)
        if s % 2:
            parts.append(_chain_scene(n, k, c["iters"], rng, scale=n / 4096.0, sets=_cuts(rng, n, k)))
            continue
        side = int(math.ceil(math.sqrt(n / 4.0)))
        kk, j, i = np.unravel_index(np.arange(n), (4, side, side))
        pos = np.stack([i - (side - 1) / 2, j - (side - 1) / 2, 0.5 + kk], 1) + rng.uniform(-0.01, 0.01, (n, 3))
        sets = np.empty(n, np.int64)
        sets[np.argsort(pos[:, 0], kind="stable")] = _cuts(rng, n, k)
        parts.append(_scene(_at_rest(pos, rng, 0.05, 0.05), np.full(n, 0.5), np.ones(n), [[0, 0, 1, 0]], 0.5, DT, 1, 1, 4, k, sets,
                            c["iters"]))
    return S.concat_scenes("batch", parts, iters=c["iters"], assign_overlap=True)


def _make(c, seed):
    """(scene, masks or None)"""
    rng = np.random.default_rng(seed)
    if c["scene"] == "pile":
        return _pile_scene(c, seed)
    if c["scene"] == "chain":
        return _chain_scene(c["n"], c["workers"], c["iters"], rng), None
    if c["scene"] == "batch":
        return _batch_scene(c, seed), None
    if c["scene"] == "building":
        sc = S.box_building(storeys=c["storeys"], cells=c["cells"], n_sets=c["workers"], iters=c["iters"])
    else:
        sc = S.plank_bridge(planks=c["planks"], n_sets=c["workers"], iters=c["iters"])
    sc.state[:, 7:13] += rng.normal(0.0, 0.02, (sc.n_bodies, 6)).astype(np.float32)
    return sc, None


# ---------------------------------------------------------------------------
# the passes
# ---------------------------------------------------------------------------

def _network(seed):
    """parameters as training leaves them: a small correction to the previous impulses"""
    th = S.mlp_init_params(seed=seed % 1000 + 5, bias_scale=0.1)
    th[4992:5184] *= 0.05
    return th


def _rows(n, seed):
    """features and targets in the ranges that steps log"""
    rng = np.random.default_rng(seed)
    f = np.zeros((n, 12), np.float32)
    f[:, 0:3] = rng.uniform(-3, 3, (n, 3))
    f[:, 3] = rng.uniform(0, 2, n)
    f[:, 4] = rng.uniform(0, 2, n)
    f[:, 5:7] = rng.uniform(-0.5, 0.5, (n, 2))
    f[:, 7:9] = rng.uniform(0, 4, (n, 2))
    f[:, 9:11] = rng.uniform(0, 1.5, (n, 2))
    f[:, 11] = rng.integers(0, 9, n) / 8.0
    t = f[:, 4:7] + 0.1 * f[:, 0:3] + rng.uniform(-0.3, 0.3, (n, 3)).astype(np.float32)
    return f, t.astype(np.float32)


def prepare(case, seed):
    if case["kind"] in ("train", "infer"):
        sim = ovl.Simulation(S.resting_sphere())
        theta = S.mlp_init_params(seed=seed % 1000 + 5) if case["kind"] == "train" else _network(seed)
        sim.mlp_set_params(theta)
        f, t = _rows(case["rows"], seed)
        if case["kind"] == "train":
            sim.log_reserve(case["rows"])
            sim.log_append(f, t)
        return dict(case=case, sim=sim, theta=theta, feat=f, seed=seed)
    sc, masks = _make(case, seed)
    stream = torch.cuda.Stream()
    params = {}
    if case["scene"] == "pile":
        params = dict(lb_deact_every=10 if case["kind"] == "period" else int(case["removals"]),
                      lb_load=ovl.OVL_LB_CONTACTS if case["lb_contacts"] else ovl.OVL_LB_BODIES,
                      weights=ovl.OVL_WEIGHTS_UNIFORM if case["uniform"] else ovl.OVL_WEIGHTS_GEODESIC)
    sim = ovl.Simulation(sc, params, stream=stream.cuda_stream, partition=masks is None)
    if masks is not None:
        sim.set_membership(masks)
    if case.get("learned"):
        sim.mlp_set_params(_network(seed))
        sim.set_warmstart_mode(ovl.OVL_WS_MLP)
    state = torch.from_numpy(sc.state).cuda()
    return dict(case=case, sim=sim, stream=stream, masks=masks, iters=sc.iters, state=state, out=torch.empty_like(state))


def run(state):
    sim, case = state["sim"], state["case"]
    if case["kind"] == "train":
        sim.mlp_set_params(state["theta"])
        loss = sim.mlp_train(0, case["rows"], case["batch"], case["steps"], seed=state["seed"])
        return dict(theta=sim.mlp_params(), loss=loss)
    if case["kind"] == "infer":
        return sim.mlp_forward(state["feat"])
    sim.set_state(state["state"])
    if case["kind"] == "period":
        sim.set_membership(state["masks"])
        sim.set_step_index(0)
        sim.step_n(10)
    else:
        sim.step()
    out = sim.state(out=state["out"])
    return dict(x=out[:, 0:3], q=out[:, 3:7], v=out[:, 7:10], w=out[:, 10:13])


def _size(c):
    """bodies, contacts and joints per body, workers per body, sweeps (estimates from the generators)"""
    if c["scene"] == "pile":
        n = c["nx"] * c["ny"] * c["nz"] * (1.03 if c["big"] else 1.0)
        copies = 1.0
        for d, w, pitch in zip((c["nx"], c["ny"], c["nz"]), c["workers"].split(","), (1.04, 1.04, 0.76)):
            copies *= min(int(w), 1.0 + 2.0 * c["reach"] * (int(w) - 1) / (d * pitch))
        return n, 2.9, copies, c["iters"]
    if c["scene"] == "chain":
        return c["n"], 1.2, 1.0 + 4.0 * c["workers"] / c["n"], c["iters"]
    if c["scene"] == "batch":
        return c["scenes"] * (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"] + 1e-9), 2.0, 1.1, c["iters"]
    if c["scene"] == "building":
        return c["storeys"] * ((c["cells"] + 1) ** 2 + c["cells"] ** 2) + 2, 14.0, 1.2, c["iters"]
    return c["planks"] + 2, 6.0, 1.2, c["iters"]


def work(case):
    """A step cannot do without: every body's state in and out (104 B) and its scene parameters (12 B), a mask in and out
    (16 B), and per (worker, constraint) pair the warm-start impulses in and out (24 B); per pair and sweep three rows
    of about 50 operations.  A training row is read once and costs three passes of 10,112 operations."""
    if case["kind"] == "train":
        rows = float(case["batch"]) * case["steps"]
        return dict(bytes=60.0 * rows + 8.0 * 5187, flops=3 * 10112.0 * rows)
    if case["kind"] == "infer":
        return dict(bytes=60.0 * case["rows"] + 4.0 * 5187, flops=10112.0 * case["rows"])
    n, per_body, copies, iters = _size(case)
    pairs = n * per_body * copies
    steps = 10 if case["kind"] == "period" else 1
    return dict(bytes=steps * (132.0 * n + 24.0 * pairs), flops=steps * 150.0 * pairs * iters)


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    """Spheres, joints and the network in 64 bits.  None for the ten-step period (a pile's step amplifies rounding), boxes
    and the learned start inside a step, and for batches and large removals, whose sequential load balance takes minutes here."""
    if case["kind"] == "infer":
        return _exact_infer(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "period" or case["scene"] in ("building", "bridge", "batch") or case.get("learned"):
        return None
    if case["scene"] == "pile" and case["removals"] and case["nx"] * case["ny"] * case["nz"] > 40000:
        return None
    sc, masks = _make(case, seed)
    return _exact_step(sc, masks, case)


def _layers64(theta):
    t = torch.as_tensor(theta).double()
    return [t[0:768].view(12, 64), t[768:832], t[832:4928].view(64, 64), t[4928:4992], t[4992:5184].view(64, 3), t[5184:5187]]


def _forward64(p, x):
    h1 = torch.relu(x @ p[0] + p[1])
    h2 = torch.relu(h1 @ p[2] + p[3])
    return x[:, 4:7] + h2 @ p[4] + p[5]


def _exact_infer(case, seed):
    f, _ = _rows(case["rows"], seed)
    return _forward64(_layers64(_network(seed)), torch.from_numpy(f).double()).numpy()


def _mix(z):
    """SplitMix64's finaliser on int64 tensors (logical shifts, wrapping products)"""
    def shr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)
    z = (z ^ shr(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ shr(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ shr(z, 31)


def _exact_train(case, seed):
    """Adam on the mean squared error; batches drawn with replacement by SplitMix64 of the sample's index"""
    f, t = _rows(case["rows"], seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f, t = torch.from_numpy(f).double().to(dev), torch.from_numpy(t).double().to(dev)
    th = torch.from_numpy(S.mlp_init_params(seed=seed % 1000 + 5)).double().to(dev).requires_grad_()
    m, v, losses = torch.zeros_like(th), torch.zeros_like(th), []
    B = case["batch"]
    for k in range(case["steps"]):
        idx = np.arange(k * B + 1, (k + 1) * B + 1, dtype=np.uint64)
        with np.errstate(over="ignore"):
            z = np.uint64(seed) + np.uint64(0x9E3779B97F4A7C15) * idx
        z = _mix(torch.from_numpy(z.view(np.int64))).numpy().view(np.uint64)
        rows = torch.from_numpy((z % np.uint64(case["rows"])).astype(np.int64)).to(dev)
        loss = ((_forward64(_layers64(th), f[rows]) - t[rows]) ** 2).mean()
        g, = torch.autograd.grad(loss, th)
        losses.append(loss.detach())
        with torch.no_grad():
            m.mul_(0.9).add_(0.1 * g)
            v.mul_(0.999).add_(0.001 * g * g)
            th -= 1e-3 * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return dict(theta=th.detach().cpu().numpy(), loss=torch.stack(losses).cpu().numpy())


def _near(x32, r32, rmax):
    """pairs a < b whose spheres pass the method's FP32 test d2 <= (ra + rb + margin)^2, in (a, b) order"""
    n, dev = len(r32), x32.device
    cs = 2.02 * float(rmax) + 1.02 * MARGIN
    cell = torch.floor((x32.double() - x32.double().min(0).values) / cs).long() + 1
    dim = cell.max(0).values + 2
    key = (cell[:, 0] * dim[1] + cell[:, 1]) * dim[2] + cell[:, 2]
    order = torch.argsort(key)
    ks = key[order]
    found = []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                want = key + (dx * dim[1] + dy) * dim[2] + dz
                lo, hi = torch.searchsorted(ks, want), torch.searchsorted(ks, want, right=True)
                for j in range(int((hi - lo).max())):
                    a = torch.nonzero(lo + j < hi)[:, 0]
                    b = order[(lo + j)[a]]
                    a, b = a[b > a], b[b > a]
                    d = x32[b] - x32[a]
                    d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
                    rs = (r32[a] + r32[b]) + np.float32(MARGIN)
                    hit = d2 <= rs * rs
                    found.append(a[hit] * n + b[hit])
    code = torch.sort(torch.cat(found)).values
    return code // n, code % n


def _balance(mask, ab, nbr, gamma, weight, workers, removals):
    """the method's sequential load balance (activation by the lighter side, gamma-balls; removals of bodies that bridge nothing)"""
    load = [0] * workers
    def bits(m):
        while m:
            yield (m & -m).bit_length() - 1
            m &= m - 1
    for b, m in enumerate(mask):
        for w in bits(m):
            load[w] += weight[b]
    def put(m, b, s):
        for w in bits(m):
            load[w] += s * weight[b]
        mask[b] = mask[b] | m if s > 0 else mask[b] & ~m
    def bridge(b):
        u = 0
        for v in nbr(b):
            u |= mask[v]
        return u & (u - 1) != 0
    for a, b in ab:
        wa, wb = mask[a], mask[b]
        if not wa & wb:
            if sum(load[w] for w in bits(wa)) <= sum(load[w] for w in bits(wb)):
                put(wa, b, 1)
                root = b
            else:
                put(wb, a, 1)
                root = a
            ball, edge = {root}, [root]
            for _ in range(gamma):
                edge = list({v for u in edge for v in nbr(u)} - ball)
                ball.update(edge)
            for u in ball:
                put((wa | wb) & ~mask[u], u, 1)
        elif removals:
            many_a, many_b = wa & (wa - 1), wb & (wb - 1)
            if many_a and not many_b and not bridge(a):
                put(wa & ~wb, a, -1)
            elif many_b and not many_a and not bridge(b):
                put(wb & ~wa, b, -1)
            elif wa == wb:
                keep = 1 << min(bits(wa), key=lambda w: (load[w], w))
                put(wa & ~keep, a, -1)
                put(wb & ~keep, b, -1)


def _chain_overlap(mask, joints, gamma):
    """articulated overlap of a chain: joints across workers activate both ends in both, then grow by gamma links"""
    n = len(mask)
    for a, b in joints:
        wa, wb = (mask[a], mask[b]) if a >= 0 and b >= 0 else (0, 0)
        if not wa or wa & (wa - 1) or wb & (wb - 1) or wa == wb:
            continue
        for end, other in ((a, b), (b, a)):
            mask[end] |= mask[other]
            both = mask[a] | mask[b]
            for u in range(max(0, end - gamma), min(n, end + gamma + 1)):
                if mask[u] & (mask[u] - 1) == 0:
                    mask[u] |= both


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _rotate(q, v):
    t = 2 * _cross(q[:, 1:], v)
    return v + q[:, :1] * t + _cross(q[:, 1:], t)


def _exact_step(sc, masks, case):
    """One timestep of the method: contacts, load balance, every worker's projected Gauss-Seidel sweeps colour by colour,
    integration, geodesic weights, blend."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    n, h, mu, nj = sc.n_bodies, float(sc.scene_dt[0]), float(sc.scene_mu[0]), len(sc.joints)
    W = int(sc.n_sets[0])
    s32 = torch.from_numpy(sc.state).to(dev)
    st, rad = s32.double(), torch.from_numpy(sc.radius).to(dev).double()
    im = torch.from_numpy(sc.inv_mass).to(dev).double()
    ii = im / (0.4 * rad * rad)
    x = st[:, 0:3]
    # contacts: sphere pairs, then each sphere's planes
    ca = cb = torch.zeros(0, dtype=torch.long, device=dev)
    if sc.scene_flags[0] & 1:
        ca, cb = _near(s32[:, 0:3].contiguous(), torch.from_numpy(sc.radius).to(dev), sc.radius.max())
    d = x[cb] - x[ca]
    L = d.norm(dim=1)
    nrm, phi = d / L[:, None], L - rad[ca] - rad[cb]
    balls = torch.stack([ca, cb], 1)
    for k, pl in enumerate(sc.planes):
        p32 = torch.from_numpy(pl).to(dev)
        g32 = (((p32[0] * s32[:, 0] + p32[1] * s32[:, 1]) + p32[2] * s32[:, 2]) - p32[3]) - torch.from_numpy(sc.radius).to(dev)
        hit = torch.nonzero(g32 <= np.float32(MARGIN))[:, 0]
        p = p32.double()
        ca, cb = torch.cat([ca, hit]), torch.cat([cb, torch.full_like(hit, n + k)])
        nrm = torch.cat([nrm, (-p[:3]).expand(len(hit), 3)])
        phi = torch.cat([phi, x[hit] @ p[:3] - p[3] - rad[hit]])
    order = torch.argsort(ca * (n + len(sc.planes)) + cb)
    ca, cb, nrm, phi = ca[order], cb[order], nrm[order], phi[order]
    nc = len(ca)
    # the constraint graph and the membership
    joints = torch.from_numpy(sc.joints.astype(np.int64)).to(dev)
    both = joints[(joints >= 0).all(1)]
    e = torch.cat([balls, both])
    e = torch.unique(torch.cat([e, e.flip(1)]), dim=0)
    m = [1 << int(w) for w in sc.set_of_body] if masks is None else [int(v) for v in masks]
    if masks is None and sc.assign_overlap:
        _chain_overlap(m, sc.joints.tolist(), int(sc.scene_gamma[0]))
    mt = torch.tensor([v - (1 << 64) if v >> 63 else v for v in m], device=dev)
    cand = balls if case.get("removals") else balls[(mt[balls[:, 0]] & mt[balls[:, 1]]) == 0]
    ptr, col = torch.searchsorted(e[:, 0].contiguous(), torch.arange(n + 1, device=dev)).tolist(), e[:, 1].tolist()
    weight = [1] * n
    if case.get("lb_contacts"):
        real = torch.cat([ca, cb[cb < n]])
        weight = (1 + torch.bincount(real, minlength=n)).tolist()
    _balance(m, cand.tolist(), lambda b: col[ptr[b]:ptr[b + 1]], int(sc.scene_gamma[0]), weight, W, case.get("removals"))
    member = torch.from_numpy(((np.array(m, dtype=np.uint64)[:, None] >> np.arange(W, dtype=np.uint64)) & np.uint64(1)).astype(bool)).to(dev)
    entry = torch.full((n, W), -1, dtype=torch.long, device=dev)
    eb, ew = torch.nonzero(member, as_tuple=True)
    E = len(eb)
    entry[eb, ew] = torch.arange(E, device=dev)
    # (worker, constraint) pairs; a plane or the world is the extra entry E
    A = torch.cat([ca, joints[:, 0]])
    B = torch.cat([torch.where(cb < n, cb, -1), joints[:, 1]])
    all_in = torch.cat([member, torch.ones(1, W, dtype=torch.bool, device=dev)])
    pc, pw = torch.nonzero(all_in[A] & all_in[B], as_tuple=True)
    side = torch.cat([entry, torch.full((1, W), E, dtype=torch.long, device=dev)])
    sa, sb = side[A[pc], pw], side[B[pc], pw]
    key = torch.cat([(ca << 32) | (cb << 2), (1 << 62) | torch.arange(nj, device=dev)])[pc]
    # greedy colours in descending order of the mixed key, by rounds of local maxima
    low = -(1 << 63)
    pr = _mix(key) ^ low
    colour = torch.full_like(pc, -1)
    used = torch.zeros(E + 1, dtype=torch.long, device=dev)
    live = torch.arange(len(pc), device=dev)
    while len(live):
        top = torch.full((E + 1,), low, dtype=torch.long, device=dev)
        top.scatter_reduce_(0, sa[live], pr[live], "amax")
        top.scatter_reduce_(0, sb[live], pr[live], "amax")
        ok = ((top[sa[live]] == pr[live]) | (sa[live] == E)) & ((top[sb[live]] == pr[live]) | (sb[live] == E))
        k = live[ok]
        free = ~(used[sa[k]] | used[sb[k]])
        c = torch.log2((free & -free).double()).round().long()
        colour[k] = c
        used[sa[k]] |= 1 << c
        used[sb[k]] |= 1 << c
        used[E] = 0
        live = live[~ok]
    # rows: directions and lever arms of the three rows of every pair, targets, 1 / (J M^-1 J^T)
    isc = pc < nc
    P = len(pc)
    zero3 = torch.zeros(1, 3, dtype=torch.float64, device=dev)
    eye = torch.eye(3, dtype=torch.float64, device=dev)
    an = nrm.abs()
    ax = torch.zeros(nc, dtype=torch.long, device=dev)
    best = an[:, 0].clone()
    for k in (1, 2):
        less = an[:, k] < best - 1e-4
        ax[less] = k
        best = torch.where(less, an[:, k], best)
    t1 = eye[ax] - nrm.gather(1, ax[:, None]) * nrm
    t1 = t1 / t1.norm(dim=1, keepdim=True)
    dirs = torch.cat([torch.stack([nrm, t1, _cross(nrm, t1)], 1), eye.expand(nj, 3, 3)])
    q = st[:, 3:7]
    anc = torch.from_numpy(sc.anchors).to(dev).double()
    def pivot(b, a):
        r = torch.where((b >= 0)[:, None], _rotate(q[b.clamp(min=0)], a), zero3)
        return r, torch.where((b >= 0)[:, None], x[b.clamp(min=0)], a)
    jra, jxa = pivot(joints[:, 0], anc[:, 0:3])
    jrb, jxb = pivot(joints[:, 1], anc[:, 3:6])
    rb_c = torch.where(cb < n, rad[cb.clamp(max=n - 1)], 0.0)
    ra = torch.cat([rad[ca][:, None] * nrm, jra])
    rb = torch.cat([-rb_c[:, None] * nrm, jrb])
    tn = torch.where(phi > 0, -phi / h, ERP * (-phi - SLOP).clamp(min=0) / h)
    target = torch.cat([torch.stack([tn, torch.zeros_like(tn), torch.zeros_like(tn)], 1), -ERP / h * ((jxb - jxa) + (jrb - jra))])
    ime, iie = torch.cat([im[eb], im.new_zeros(1)]), torch.cat([ii[eb], ii.new_zeros(1)])
    v = torch.cat([st[eb, 7:10] + torch.tensor([0.0, 0.0, -GRAVITY], device=dev, dtype=torch.float64) * h, zero3])
    w = torch.cat([st[eb, 10:13], zero3])
    lam = torch.zeros(P, 3, dtype=torch.float64, device=dev)
    groups = []
    for c in range(int(colour.max()) + 1 if P else 0):
        k = torch.nonzero(colour == c)[:, 0]
        i, a, b = pc[k], sa[k], sb[k]
        D = dirs[i]
        ja, jb = _cross(ra[i][:, None].expand(-1, 3, -1), D), _cross(rb[i][:, None].expand(-1, 3, -1), D)
        s = (ime[a] + ime[b])[:, None] + iie[a][:, None] * (ja * ja).sum(2) + iie[b][:, None] * (jb * jb).sum(2)
        groups.append((k, a, b, D, ja, jb, 1.0 / s, target[i], isc[k], ime[a][:, None], ime[b][:, None], iie[a][:, None], iie[b][:, None]))
    for _ in range(case["iters"]):
        for k, a, b, D, ja, jb, kk, tg, con, ma, mb, ia, ib in groups:
            va, vb, wa, wb, l = v[a], v[b], w[a], w[b], lam[k]
            for r in range(3):
                rel = (D[:, r] * (vb - va)).sum(1) + (jb[:, r] * wb).sum(1) - (ja[:, r] * wa).sum(1)
                new = l[:, r] + kk[:, r] * (tg[:, r] - rel)
                lim = mu * l[:, 0]
                box = new.clamp(min=0) if r == 0 else torch.minimum(torch.maximum(new, -lim), lim)
                new = torch.where(con, box, new)
                dl = (new - l[:, r])[:, None]
                l[:, r] = new
                va, vb = va - ma * dl * D[:, r], vb + mb * dl * D[:, r]
                wa, wb = wa - ia * dl * ja[:, r], wb + ib * dl * jb[:, r]
            lam[k] = l
            v[a], w[a], v[b], w[b] = va, wa, vb, wb
            v[E], w[E] = 0.0, 0.0
    v, w = v[:E], w[:E]
    qe = q[eb]
    dq = torch.cat([-(w * qe[:, 1:]).sum(1, keepdim=True), qe[:, :1] * w + _cross(w, qe[:, 1:])], 1)
    qe = qe + 0.5 * h * dq
    qe = qe / qe.norm(dim=1, keepdim=True)
    # D(o, i): levels of a search from the bodies of one worker only
    count = member.sum(1)
    seen = member & (count == 1)[:, None]
    dist = torch.full((n, W), 255, dtype=torch.uint8, device=dev)
    for level in range(1, int(sc.scene_beta[0]) + 1):
        new = torch.zeros(n, W, dtype=torch.int16, device=dev)
        for part in e.split(1 << 20):
            new.index_add_(0, part[:, 0], seen[part[:, 1]].to(torch.int16))
        new = new.bool() & ~seen
        dist[new] = level
        seen |= new
    de = dist[eb, ew].double()
    inv = torch.where((de < 255) & (count[eb] > 1), 1.0 / de, 0.0)
    total = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, eb, inv)[eb]
    wt = torch.where((total > 0) & (not case.get("uniform")), inv / total.clamp(min=1e-300), 1.0 / count[eb])
    first = torch.zeros(n, dtype=torch.long, device=dev)
    first[eb.flip(0)] = torch.arange(E - 1, -1, -1, device=dev)
    flip = torch.where((qe * qe[first[eb]]).sum(1) < 0, -1.0, 1.0)
    def mix(t):
        return torch.zeros(n, t.shape[1], dtype=torch.float64, device=dev).index_add_(0, eb, wt[:, None] * t)
    vn, wn, qn = mix(v), mix(w), mix(flip[:, None] * qe)
    return dict(x=x + h * vn, q=qn / qn.norm(dim=1, keepdim=True), v=vn, w=wn)
