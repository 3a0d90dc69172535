"""Performance cases of the library: what a user's program has it do, through its public entry points.

Four kinds of case:

* ``lattice``: a uniform lid-driven lattice.  ``after`` says what follows the steps of a pass:
  ``none`` (a run of steps), ``flags`` (the refinement flags and block maxima of the sensor) or
  ``learned`` (a dynamic-refinement interval: sensor, block features, predictor, predicted flags).
* ``mesh``: cycles of the multi-level block mesh and the block maxima of the sensor.
* ``train``: an epoch of the sensor predictor's training.
* ``regrid``: the regrid of a level (tags, buffer, clustering) and its level map.

``exact`` evaluates the same formulas in plain 64-bit torch.
"""
import numpy as np
import torch
import torch.nn.functional as F

import paper_1507_06767_gb300 as L
from paper_1507_06767_gb300 import learned as LN

DEV = "cuda"
TORCH_TYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
LBM_TYPE = {"f64": L.LBM_F64, "f32": L.LBM_F32, "f16": L.LBM_F16S, "bf16": L.LBM_BF16S}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
FLOPS = {9: 110, 19: 260}  # arithmetic of one cell update with the sensor
REGRID_EFFICIENCY, REGRID_MIN_WIDTH, MAX_BOXES = 0.8, 2, 8192

# The velocity sets in the order of the populations (rest, axes, diagonals) and 36 w_i.
C = {
    9: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)],
    19: [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
         (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
         (0, -1, 1)],
}
W36 = {9: [16, 4, 4, 4, 4, 1, 1, 1, 1], 19: [12] + [2] * 6 + [1] * 12}


def lattice(name, q, nx, ny, nz, dtype, re, steps, calls=1, every=0, after="none", frac=0.0, block=16, periodic=0):
    """`calls` lbm_step calls of `steps` steps each, the sensor every `every` steps (0: on a call's last step)."""
    return {"name": name, "kind": "lattice", "q": q, "nx": nx, "ny": ny, "nz": nz, "dtype": dtype, "re": re,
            "steps": steps, "calls": calls, "every": every, "after": after, "frac": frac, "block": block,
            "periodic": periodic}


def mesh(name, bx, by, bz, edge, lmax, re, warm, cycles):
    return {"name": name, "kind": "mesh", "bx": bx, "by": by, "bz": bz, "edge": edge, "lmax": lmax, "re": re,
            "warm": warm, "cycles": cycles}


def train(name, cin, hidden, batch, h, w, batches):
    return {"name": name, "kind": "train", "cin": cin, "hidden": hidden, "batch": batch, "h": h, "w": w,
            "batches": batches}


def regrid(name, q, nx, ny, nz, dtype, coarsen):
    return {"name": name, "kind": "regrid", "q": q, "nx": nx, "ny": ny, "nz": nz, "dtype": dtype, "re": 4.0 * nx,
            "coarsen": coarsen}


def listed():
    return [
        # a small 2-D run in the paper's own precision between two looks at its flags: launches and latency
        lattice("d2q9_128_f64", 9, 128, 128, 1, "f64", 100.0, 100, after="flags"),
        # a 2-D mesh that regrids at every step (Sec. 5.2), odd sides: the smallest call there is
        lattice("d2q9_301x203_f32_each_step", 9, 301, 203, 1, "f32", 400.0, 1, after="flags"),
        # the dynamic-refinement loop with the learned predictor: 200 steps, then a predicted regrid
        lattice("d2q9_1024_f32_learned", 9, 1024, 1024, 1, "f32", 1000.0, 200, after="learned"),
        # the headline: a 3-D cavity, sensor and top-10 % flags at every step
        lattice("d3q19_256_f32_each_step", 19, 256, 256, 256, "f32", 1000.0, 1, after="flags", frac=0.1),
        # a run of steps on odd, ragged sides
        lattice("d3q19_195x129x97_f32", 19, 195, 129, 97, "f32", 500.0, 16),
        # the large 3-D run in 16-bit storage
        lattice("d3q19_512_f16", 19, 512, 512, 512, "f16", 1000.0, 8),
        # ragged 3-D run in the other 16-bit type, sensor at every step, one periodic axis
        lattice("d3q19_250x182x130_bf16", 19, 250, 182, 130, "bf16", 800.0, 8, every=1, periodic=4),
        # the 64-bit run that the others are judged against
        lattice("d3q19_128_f64", 19, 128, 128, 128, "f64", 1000.0, 10, after="flags", frac=0.1),
        # the paper's refined mesh: three levels, 512^3 finest cells
        mesh("mesh_3level_512", 16, 16, 16, 32, 2, 1000.0, 4, 2),
        # a small refined mesh of small blocks
        mesh("mesh_3level_small", 8, 6, 4, 16, 2, 200.0, 16, 8),
        # an epoch of the predictor's training on 64 x 64 block grids
        train("train_16x64x64", 4, 16, 16, 64, 64, 8),
        # the regrid of the 3-D cavity
        regrid("regrid_256_f32", 19, 256, 256, 256, "f32", 4),
    ]


def _log_int(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng):
    kind = rng.choice(["lattice2", "lattice2", "lattice3", "lattice3", "mesh", "train", "regrid"])
    if kind == "lattice2":
        nx, ny = _log_int(rng, 40, 1600), _log_int(rng, 40, 1600)
        dtype = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        after = rng.choice(["flags", "none"] if dtype in ("f64", "f32") else ["none"])
        c = lattice("", 9, nx, ny, 1, dtype, nx * rng.uniform(0.5, 5.0), rng.choice([1, 7, 33, 64, 100]), after=after,
                    every=rng.choice([0, 0, 1]), block=rng.choice([8, 16]), periodic=rng.choice([0, 0, 1, 2]))
    elif kind == "lattice3":
        dtype = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        top = {"f64": 110, "f32": 280, "f16": 360, "bf16": 360}[dtype]
        nx, ny, nz = (_log_int(rng, 24, top) for _ in range(3))
        after = rng.choice(["flags", "none"] if dtype in ("f64", "f32") else ["none"])
        c = lattice("", 19, nx, ny, nz, dtype, nx * rng.uniform(0.8, 5.0), rng.choice([1, 2, 5, 8, 16]), after=after,
                    every=rng.choice([0, 0, 1]), frac=rng.choice([0.0, 0.1]), block=rng.choice([8, 16, 32]),
                    periodic=rng.choice([0, 0, 1, 4]))
    elif kind == "mesh":
        edge = rng.choice([8, 16, 32])
        most = {8: 12, 16: 10, 32: 8}[edge]
        bx, by, bz = (rng.randint(3, most) for _ in range(3))
        c = mesh("", bx, by, bz, edge, rng.choice([1, 2]), bx * edge * rng.uniform(0.8, 2.0), 4, rng.choice([1, 3, 6]))
    elif kind == "train":
        c = train("", rng.choice([3, 4]), rng.choice([8, 16]), rng.randint(2, 24), rng.randint(12, 80),
                  rng.randint(12, 80), rng.randint(2, 8))
    else:
        q = rng.choice([9, 19])
        if q == 9:
            c = regrid("", 9, _log_int(rng, 100, 2000), _log_int(rng, 100, 2000), 1, rng.choice(["f32", "f64"]),
                       rng.choice([1, 2, 4]))
        else:
            dtype = rng.choice(["f32", "f64"])
            nx, ny, nz = (_log_int(rng, 40, 256 if dtype == "f32" else 128) for _ in range(3))
            c = regrid("", 19, nx, ny, nz, dtype, rng.choice([2, 3, 4]))
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------ inputs
def _generator(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _lid(seed):
    """The lid velocity of a run: near 0.1, as everywhere in the tests and the benchmark."""
    return 0.09 + 0.02 * float(np.random.default_rng([int(seed), 77]).random())


def _tau(case, u):
    return 3.0 * u * case["nx"] / case["re"] + 0.5


def _smooth(g, shape, points=7):
    """A smooth random field in (-1, 1) over `shape` = (nz, ny, nx)."""
    if shape[0] == 1:
        r = torch.rand((1, 1, points, points), generator=g, device=DEV) * 2 - 1
        return F.interpolate(r, size=shape[1:], mode="bilinear", align_corners=True)[0]
    r = torch.rand((1, 1, points, points, points), generator=g, device=DEV) * 2 - 1
    return F.interpolate(r, size=shape, mode="trilinear", align_corners=True)[0, 0]


def _populations(case, seed):
    """A cavity in motion: the equilibrium of a smooth random flow below the lid's speed, with a
    per-mille of noise, in the storage convention of the type (16-bit types hold f - w)."""
    q, shape = case["q"], (case["nz"], case["ny"], case["nx"])
    g = _generator(seed)
    rho = 1 + 2e-3 * _smooth(g, shape)
    u = [0.05 * _smooth(g, shape) for _ in range(2 if q == 9 else 3)]
    usq = sum(v * v for v in u)
    f = torch.empty((q,) + shape, dtype=TORCH_TYPE[case["dtype"]], device=DEV)
    for i, c in enumerate(C[q]):
        w = W36[q][i] / 36.0
        cu = sum(c[a] * u[a] for a in range(len(u)) if c[a]) if any(c) else torch.zeros_like(rho)
        feq = w * (rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq) - 1)  # f_eq - w
        feq += w * 1e-3 * (torch.rand(shape, generator=g, device=DEV) - 0.5)
        f[i] = feq if case["dtype"] in ("f16", "bf16") else feq.to(f.dtype) + w
    return f


class _Run:
    """A lattice handle with the caller's two population buffers."""

    def __init__(self, case, seed):
        u = _lid(seed)
        self.case, self.u = case, u
        self.lat = L.Lattice(case["q"], case["nx"], case["ny"], case["nz"], _tau(case, u),
                             dtype=LBM_TYPE[case["dtype"]], lid=(u, 0.0), periodic=case.get("periodic", 0))
        self.bufs = [_populations(case, seed), None]
        self.bufs[1] = torch.empty_like(self.bufs[0])
        self.h = self.lat.h
        L.lbm_attach(self.h, self.bufs[0], self.bufs[1], L.lbm_population_bytes(self.h))

    def current(self):
        return self.bufs[L.lbm_steps_done(self.h) % 2]


def _threshold(case, u):
    return LN.threshold(_tau(case, u), u, case["nx"])


def _leaf_levels(case):
    """Leaf levels of a lid-driven cavity's blocks: finest under the lid and at its downstream
    corner, 2:1 balanced."""
    bx, by, bz, lmax = case["bx"], case["by"], case["bz"], case["lmax"]
    z, y, x = np.meshgrid(np.arange(bz), np.arange(by), np.arange(bx), indexing="ij")
    top = (by - 1 - y) / by
    corner = np.hypot(top, (bx - 1 - x) / bx)
    s = np.minimum(2.2 * top + 0.35 * np.abs(2 * (z + 0.5) / bz - 1), 1.6 * corner)
    leaf = np.where(s < 0.24, lmax, np.where(s < 0.55, lmax - 1, 0)).astype(np.int8)
    while True:
        pad = np.pad(leaf, 1, mode="edge")
        near = np.max([pad[a:a + bz, b:b + by, c:c + bx] for a in range(3) for b in range(3) for c in range(3)], axis=0)
        new = np.maximum(leaf, near - 1).astype(np.int8)
        if np.array_equal(new, leaf):
            return leaf
        leaf = new


def _mesh_tau(case, u):
    return 3.0 * u * case["bx"] * case["edge"] / case["re"] + 0.5


def _net_theta(cin, hidden, seed):
    """He-uniform parameters in the order W1, b1, W2, b2, W3, b3."""
    r = np.random.default_rng([int(seed), 5])
    parts = []
    for o, c in ((hidden, cin), (hidden, hidden), (1, hidden)):
        parts += [r.uniform(-1, 1, o * c * 9) * np.sqrt(6.0 / (c * 9)), r.uniform(-0.05, 0.05, o)]
    return np.concatenate(parts).astype(np.float32)


def _samples(case, seed):
    """Block features of cavities (density, velocity, log sensor) and the change of the log sensor."""
    g = _generator(seed, 3)
    n, shape = case["batch"] * case["batches"], (case["h"], case["w"])
    r = torch.rand((n, 4, 7, 7), generator=g, device=DEV) * 2 - 1
    s = F.interpolate(r, size=shape, mode="bicubic", align_corners=True)
    x = torch.stack([1 + 5e-3 * s[:, 0], 0.08 * s[:, 1], 0.05 * s[:, 2], s[:, 3]], dim=1)[:, :case["cin"]].contiguous()
    t = 0.3 * (s[:, 1] * s[:, 2] + s[:, 0:1].mean(dim=1)) + 0.02 * torch.randn((n,) + shape, generator=g, device=DEV)
    return x, t[:, None].contiguous()


def prepare(case, seed):
    if case["kind"] == "mesh":
        u = _lid(seed)
        m = L.BlockMesh(_leaf_levels(case), case["edge"], case["lmax"], _mesh_tau(case, u), lid=(u, 0.0))
        m.step(case["warm"])
        return {"case": case, "mesh": m}
    if case["kind"] == "train":
        net = L.Net(case["cin"], case["hidden"])
        net.set_normalisation(*LN.normalisation(0.1, case["cin"] == 4))
        net.set_params(_net_theta(case["cin"], case["hidden"], seed))
        x, t = _samples(case, seed)
        return {"case": case, "net": net, "x": x, "t": t, "seed": int(seed)}
    r = _Run(case, seed)
    if case["kind"] == "regrid":
        L.lbm_set_sensor_field(r.h, 1)
        r.lat.step(60)  # the start's noise has decayed
        maxima = np.sort(r.lat.sensor(16))
        return {"case": case, "run": r, "threshold": float(np.float32(0.93 * maxima[int(0.9 * (maxima.size - 1))]))}
    L.lbm_set_sensor_every(r.h, case["every"])
    L.lbm_set_block(r.h, case["block"])
    s = {"case": case, "run": r}
    if case["after"] != "none":
        nb = L.lbm_nblocks(r.h, case["block"])
        s |= {"nb": nb, "maxima": torch.empty(nb, dtype=torch.float64, device=DEV),
              "flags": torch.empty(nb, dtype=torch.int8, device=DEV), "threshold": _threshold(case, r.u)}
    if case["after"] == "learned":
        side = (-(-case["ny"] // case["block"]), -(-case["nx"] // case["block"]))
        net = L.Net(4, 16)
        net.set_normalisation(*LN.normalisation(r.u, True))
        net.set_params(_net_theta(4, 16, seed))
        s |= {"net": net, "features": torch.empty((1, 4) + side, device=DEV), "y": torch.empty((1, 1) + side, device=DEV),
              "predicted": torch.empty(nb, dtype=torch.float64, device=DEV)}
    return s


# ------------------------------------------------------------------------------------------ a pass
def run(state):
    case = state["case"]
    if case["kind"] == "mesh":
        # the maxima come from 32-bit arithmetic
        return {"maxima": state["mesh"].step(case["cycles"], block_max=True).astype(np.float32)}
    if case["kind"] == "train":
        losses = LN.train(state["net"], state["x"], state["t"], 1, case["batch"], 2e-3, state["seed"])
        return {"params": state["net"].params(), "loss": np.array(losses, dtype=np.float32)}
    r = state["run"]
    if case["kind"] == "regrid":
        boxes, tags = r.lat.regrid(state["threshold"], coarsen=case["coarsen"], efficiency=REGRID_EFFICIENCY,
                                   min_width=REGRID_MIN_WIDTH, max_boxes=MAX_BOXES)
        boxes = np.concatenate([boxes, np.zeros((MAX_BOXES - len(boxes), 6), dtype=boxes.dtype)])
        return {"boxes": boxes, "tags": tags.astype(np.uint8), "levels": r.lat.levels_fit(16, 0, 2)}
    for _ in range(case["calls"]):
        r.lat.step(case["steps"])
    if case["after"] == "none":
        return {"f": r.current()}
    stream = torch.cuda.current_stream().cuda_stream
    L.lbm_sensor_dev(r.h, case["block"], state["maxima"])
    # where the arithmetic is 32-bit, so are the maxima
    maxima = state["maxima"] if case["dtype"] == "f64" else state["maxima"].float()
    if case["after"] == "flags":
        if case["frac"]:
            L.lbm_flag_top_dev(r.h, case["frac"], state["flags"])
        else:
            L.lbm_flag_dev(r.h, state["threshold"], state["flags"])
        return {"f": r.current(), "flags": state["flags"], "maxima": maxima}
    nb, x, y, out = state["nb"], state["features"], state["y"], state["predicted"]
    L.lbm_block_features(r.h, case["block"], x)
    L.lbm_net_log_targets(state["maxima"], nb, LN.LOG_OFFSET, LN.FLOOR_K, x[0, 3], stream)
    state["net"].forward(x, y)
    L.lbm_net_to_maxima_residual(y, state["maxima"], nb, LN.FLOOR_K, out, stream)
    L.lbm_flags_from_maxima(out, L.LBM_F64, nb, L.LBM_FLAG_THRESHOLD, state["threshold"], state["flags"], stream)
    return {"f": r.current(), "flags": state["flags"], "maxima": maxima, "predicted": out.float()}


def _mesh_cells(case):
    leaf = _leaf_levels(case)
    return [int((leaf >= l).sum()) * (case["edge"] >> (case["lmax"] - l)) ** 3 for l in range(case["lmax"] + 1)]


def work(case):
    if case["kind"] == "mesh":
        cells = _mesh_cells(case)
        updates = case["cycles"] * sum(n << l for l, n in enumerate(cells))
        return {"bytes": 2 * 76 * sum(cells) + 8 * case["bx"] * case["by"] * case["bz"], "flops": FLOPS[19] * updates}
    if case["kind"] == "train":
        cin, hid, pos = case["cin"], case["hidden"], case["batch"] * case["h"] * case["w"]
        params = hid * cin * 9 + hid * hid * 9 + hid * 9
        # forward, weight gradients, and the input gradients of the second and third layer
        flops = 2 * pos * (3 * params - hid * cin * 9)
        return {"bytes": case["batches"] * pos * 4 * (cin + 1) + 8 * params, "flops": case["batches"] * flops}
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "regrid":
        return {"bytes": cells * BYTES[case["dtype"]] + cells // case["coarsen"] ** (2 if case["q"] == 9 else 3),
                "flops": cells}
    steps = case["steps"] * case["calls"]
    return {"bytes": 2 * case["q"] * cells * BYTES[case["dtype"]], "flops": steps * cells * FLOPS[case["q"]]}


# ------------------------------------------------------------------------------------------ 64 bits
def _moments64(q, f, shift):
    """rho - 1 and u of populations f (less the weights where `shift`)."""
    drho = sum(f[i] - (0.0 if shift else W36[q][i] / 36.0) for i in range(q))
    u = []
    for a in range(3 if q == 19 else 2):
        j = 0.0
        for i, c in enumerate(C[q]):
            if c[a]:
                j = j + c[a] * f[i]
        u.append(j / (1 + drho))
    return drho, u


def _feq64(q, i, drho, u, usq):
    """f_eq - w of direction i."""
    w = W36[q][i] / 36.0
    cu = 0.0
    for a, v in enumerate(u):
        if C[q][i][a]:
            cu = cu + C[q][i][a] * v
    if i == 0:
        cu = torch.zeros_like(drho)
    return w * (drho + (1 + drho) * (3 * cu + 4.5 * cu * cu - 1.5 * usq))


def _step64(q, f, omega, lid, periodic, sensor):
    """One pull step of the deviations f - w in 64 bits; returns the new ones and the sensor K."""
    nz, ny, nx = f.shape[1:]
    n = (nx, ny, nz)
    g = torch.empty_like(f)
    for i, c in enumerate(C[q]):
        o = C[q].index((-c[0], -c[1], -c[2]))
        g[i] = torch.roll(f[i], shifts=(c[2], c[1], c[0]), dims=(0, 1, 2))
        for a, dim in ((0, 2), (1, 1), (2, 0)):
            if c[a] and not periodic & (1 << a):
                at = 0 if c[a] == 1 else n[a] - 1
                g[i].select(dim, at).copy_(f[o].select(dim, at))
        if c[1] == -1 and not periodic & 2:
            g[i][:, ny - 1, :] += 6 * W36[q][i] / 36.0 * c[0] * lid
    drho, u = _moments64(q, g, True)
    usq = sum(v * v for v in u)
    k = torch.zeros_like(drho) if sensor else None
    for i in range(q):
        e = _feq64(q, i, drho, u, usq)
        d = g[i] - e
        if sensor:
            k += (d / (e + W36[q][i] / 36.0)).abs_()
        g[i] -= omega * d
    return g, (k / q if sensor else None)


def _block_max64(k, block, flat):
    bz = 1 if flat else block
    nz, ny, nx = k.shape
    k = F.pad(k, (0, -nx % block, 0, -ny % block, 0, -nz % bz))
    z, y, x = k.shape
    return k.view(z // bz, bz, y // block, block, x // block, block).amax(dim=(1, 3, 5)).reshape(-1)


def _conv64(x, theta, cin, hidden):
    at = 0
    for k, (o, c) in enumerate(((hidden, cin), (hidden, hidden), (1, hidden))):
        w, b = theta[at:at + o * c * 9].view(o, c, 3, 3), theta[at + o * c * 9:at + o * c * 9 + o]
        at += o * c * 9 + o
        x = F.conv2d(x, w, b, padding=1)
        x = F.relu(x) if k < 2 else x
    return x


def _normalised(x, u, with_sensor):
    shift, scale = LN.normalisation(u, with_sensor)
    s = [torch.tensor(v, dtype=torch.float64, device=DEV).view(1, -1, 1, 1) for v in (shift, scale)]
    return (x - s[0]) * s[1]


def _exact_mesh(case, seed):
    u, lmax, edge = _lid(seed), case["lmax"], case["edge"]
    tau_f, leaf = _mesh_tau(case, u), torch.from_numpy(_leaf_levels(case)).to(DEV)
    n = [edge >> (lmax - l) for l in range(lmax + 1)]
    tau = [3.0 * (tau_f - 0.5) / 3.0 / (1 << (lmax - l)) + 0.5 for l in range(lmax + 1)]

    def wide(b, m):
        return b.repeat_interleave(m, 0).repeat_interleave(m, 1).repeat_interleave(m, 2)

    mask = [wide(leaf >= l, n[l]) for l in range(lmax + 1)]
    f = [torch.zeros((19,) + tuple(m.shape), dtype=torch.float64, device=DEV) for m in mask]
    k = [None] * (lmax + 1)

    def finer(a, dim):
        """Linear interpolation to twice the cells along an axis, extrapolated at the walls."""
        m = a.shape[dim]
        lo = torch.cat([1.25 * a.narrow(dim, 0, 1) - 0.25 * a.narrow(dim, 1, 1),
                        0.75 * a.narrow(dim, 1, m - 1) + 0.25 * a.narrow(dim, 0, m - 1)], dim)
        hi = torch.cat([0.75 * a.narrow(dim, 0, m - 1) + 0.25 * a.narrow(dim, 1, m - 1),
                        1.25 * a.narrow(dim, m - 1, 1) - 0.25 * a.narrow(dim, m - 2, 1)], dim)
        return torch.stack([lo, hi], dim + 1).flatten(dim, dim + 1)

    def rescale(g, scale):
        """g with its non-equilibrium part times `scale`, in place."""
        drho, v = _moments64(19, g, True)
        usq = sum(x * x for x in v)
        for i in range(19):
            e = _feq64(19, i, drho, v, usq)
            g[i] = e + scale * (g[i] - e)
        return g

    def advance(l, theta, before):
        src = f[l]
        if l:
            ghost = torch.empty_like(src)
            for i in range(19):
                a = (1 - theta) * before[i] + theta * f[l - 1][i]
                for dim in range(3):
                    a = finer(a, dim)
                ghost[i] = a
            rescale(ghost, (tau[l] - 1) / (2 * (tau[l - 1] - 1)))
            for i in range(19):
                ghost[i][mask[l]] = src[i][mask[l]]
            src = ghost
        new, k[l] = _step64(19, src, 1 / tau[l], u, 0, True)
        del src
        old, f[l] = f[l], new
        f[l] *= mask[l]
        if l < lmax:
            advance(l + 1, 0.0, old)
            advance(l + 1, 0.5, old)
            mean = torch.stack([F.avg_pool3d(f[l + 1][i][None, None], 2)[0, 0] for i in range(19)])
            rescale(mean, 2 * (tau[l] - 1) / (tau[l + 1] - 1))
            under = wide(leaf >= l + 1, n[l])
            for i in range(19):
                f[l][i][under] = mean[i][under]

    for _ in range(case["warm"] + case["cycles"]):
        advance(0, 0.0, None)
    out = torch.zeros(leaf.numel(), dtype=torch.float64, device=DEV)
    for l in range(lmax + 1):
        m = _block_max64(k[l], n[l], False)
        at = leaf.reshape(-1) == l
        out[at] = m[at]
    return {"maxima": out}


def _exact_train(case, seed):
    x, t = (v.double() for v in _samples(case, seed))
    x = _normalised(x, 0.1, case["cin"] == 4)
    theta = torch.from_numpy(_net_theta(case["cin"], case["hidden"], seed)).to(DEV).double().requires_grad_(True)
    m, v, losses = torch.zeros_like(theta), torch.zeros_like(theta), []
    order = torch.from_numpy(np.random.default_rng(np.random.SeedSequence(int(seed))).permutation(x.shape[0])).to(DEV)
    for b in range(case["batches"]):
        at = order[b * case["batch"]:(b + 1) * case["batch"]]
        loss = ((_conv64(x[at], theta, case["cin"], case["hidden"]) - t[at]) ** 2).mean()
        g, = torch.autograd.grad(loss, theta)
        losses.append(float(loss))
        with torch.no_grad():
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            theta -= 2e-3 * (m / (1 - 0.9 ** (b + 1))) / ((v / (1 - 0.999 ** (b + 1))).sqrt() + 1e-8)
    return {"params": theta.detach(), "loss": np.array([np.mean(losses)])}


def exact(case, seed):
    if case["kind"] == "mesh":
        return _exact_mesh(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "regrid":
        return None  # whole numbers only
    q, u, shift = case["q"], _lid(seed), case["dtype"] in ("f16", "bf16")
    stored = _populations(case, seed)
    f = torch.empty(stored.shape, dtype=torch.float64, device=DEV)
    for i in range(q):
        f[i] = stored[i]
        if not shift:
            f[i] -= W36[q][i] / 36.0
    del stored
    steps, omega, k = case["steps"] * case["calls"], 1 / _tau(case, u), None
    for s in range(steps):
        f, k = _step64(q, f, omega, u, case["periodic"], s == steps - 1 and case["after"] != "none")
    drho, v = _moments64(q, f, True) if case["after"] == "learned" else (None, None)
    if not shift:
        for i in range(q):
            f[i] += W36[q][i] / 36.0
    if case["after"] == "none":
        return {"f": f}
    maxima = _block_max64(k, case["block"], q == 9)
    out = {"f": f, "flags": None, "maxima": maxima}
    if case["after"] == "learned":
        b = case["block"]
        x = torch.stack([F.avg_pool2d(a[None], b, ceil_mode=True)[0, 0] for a in (1 + drho, v[0], v[1])])
        now = torch.log10(maxima.clamp(min=LN.FLOOR_K))
        x = torch.cat([x, (now - LN.LOG_OFFSET).view((1,) + x.shape[1:])])[None]
        y = _conv64(_normalised(x, u, True), torch.from_numpy(_net_theta(4, 16, seed)).to(DEV).double(), 4, 16)
        out["predicted"] = 10 ** (y.reshape(-1) + now)
    return out
