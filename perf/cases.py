"""Workloads of the TensorMD library as its users run them.

A case is one call, or one short run of calls, through the public binding
(`paper_2310_08439_gb300.tmd`): a single evaluation on a kept neighbour table,
a single point (table and evaluation), the descriptors with dE/dG, the
allocation-free call, MD on one resident system (device-resident or from host
buffers), and a batch of uneven systems evaluated or advanced together.  Sizes
and models are those of the package's workloads (`inputs.py`), its tests and
its benchmark, and others of the same ranges.

Outputs are handed on in the precision of the arithmetic that forms them:
energies, virials and velocities come back from the library in FP64 but are
sums of FP32 terms (or moved by FP32 forces), so they are returned as float32,
as trajectory and log files keep them; forces, dE/dG and virials of the BF16
network form (about three significant digits) are returned as bfloat16.
Positions stay float64.
"""
import math

import numpy as np
import torch

from paper_2310_08439_gb300 import inputs as I
from paper_2310_08439_gb300 import tmd

MASSES = [55.845, 63.546, 26.982, 183.84, 107.868]
ACC = 103.6427          # amu A^2/fs^2 per eV


def _case(name, kind, lattice="fcc", a=4.05, nx=4, ny=4, nz=4, S=1, K=16, rc=6.0, skin=1.0, net="64-64", act="tanh",
          precision="fp32", sigma=0.1, table=0, vacuum=0.0, systems=0, active=0, n_max=0, steps=0):
    return {"name": name, "kind": kind, "lattice": lattice, "a": a, "nx": nx, "ny": ny, "nz": nz, "S": S, "K": K,
            "rc": rc, "skin": skin, "net": net, "act": act, "precision": precision, "sigma": sigma, "table": table,
            "vacuum": vacuum, "systems": systems, "active": active, "n_max": n_max, "steps": steps}


def listed():
    return [
        # the smallest call: one 32-atom cell (the `tiny` workload), table and evaluation, as a
        # calculator does for every new configuration of a small cell; launches and latency
        _case("single_point_32", "single", a=3.61, nx=2, ny=2, nz=2, K=8, rc=5.0, skin=0.0, net="32-32", sigma=0.05),
        # a host MD code that owns the table and all device memory: the allocation-free call,
        # a few thousand atoms, odd repeats
        _case("noalloc_bcc_8k", "noalloc", lattice="bcc", a=2.9, nx=15, ny=17, nz=16, sigma=0.08),
        # single point of a two-species film (open along z, ragged): table and evaluation, as for
        # each new structure of a screening run
        _case("single_point_film_19k", "single", a=3.61, nx=23, ny=21, nz=10, S=2, vacuum=12.0, skin=0.0),
        # descriptors and dE/dG of a two-species cell: what fitting and uncertainty tools read
        _case("descriptors_37k", "descriptors", a=3.61, nx=21, ny=21, nz=21, S=2, skin=0.0),
        # MD of the `medium` workload (16,384 atoms, two species): 10 steps of 1 fs, table every
        # 5 steps, then a frame for the trajectory
        _case("md_16k", "md", a=3.61, nx=16, ny=16, nz=16, S=2, steps=10),
        # MD driven from host buffers (the benchmark's end-to-end path) on a ragged quarter-million-atom
        # cell: 5 steps a call, the state up and down through pinned memory
        _case("md_host_262k", "md_host", nx=41, ny=40, nz=40, steps=5),
        # the largest call: force evaluation of the `large` workload (1,048,576 atoms) on a kept table
        _case("eval_1m", "eval", nx=64, ny=64, nz=64),
        # the same potential with the BF16 network form on 131k atoms
        _case("eval_bf16_131k", "eval", nx=32, ny=32, nz=32, precision="bf16"),
        # the paper's k = 32 potential (128-128-128, SquarePlus) on bcc W, FP32
        _case("eval_k32_148k", "eval", lattice="bcc", a=3.1887, nx=42, ny=42, nz=42, K=32, net="128-128-128",
              act="squareplus", skin=0.0),
        # the paper's k = 128 potential on the dense bcc W lattice (a = 2.8 A), BF16 network
        _case("eval_k128_bf16_39k", "eval", lattice="bcc", a=2.8, nx=27, ny=27, nz=27, K=128, net="128-128-128-128",
              act="squareplus", skin=0.0, precision="bf16"),
        # uneven systems evaluated together (the `batch` workload's recipe: 32 to 8,192 atoms each,
        # three species, 128-128 network), tables kept
        _case("batch_128_systems", "batch", S=3, net="128-128", systems=128, active=128, n_max=8192),
        # one tick of the serving loop: the systems with an open request advance one MD step
        # (the `serve` workload's recipe, 64 to 16,384 atoms each, two species)
        _case("serve_tick_24_of_48", "serve", S=2, net="128-128", systems=48, active=24, n_max=16384, steps=1),
    ]


def draw(rng):
    """One more case: a kind, then sizes over the ranges above (log-uniform)."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["eval", "eval", "eval", "single", "descriptors", "noalloc", "md", "md_host", "batch", "serve"])
    precision = "fp32" if kind in ("md", "md_host", "serve") else rng.choice(["fp32", "fp32", "fp32", "bf16"])
    if kind in ("batch", "serve"):
        S = rng.choice([1, 2, 3])
        systems = logint(4, 128)
        active = systems if kind == "batch" else max(1, int(systems * rng.uniform(0.2, 1.0)))
        return _drawn(kind, S=S, K=16, net="128-128", precision=precision, systems=systems, active=active,
                      n_max=logint(256, 8192), steps=1 if kind == "serve" else 0)
    K = rng.choice([8, 16, 16, 16, 32, 64, 128])
    S = 1 if K == 128 else rng.choice([1, 1, 2] if K == 64 else [1, 1, 2, 3, 5])
    net = rng.choice(["64-64", "64-64", "32-32", "128-128", "128-128-128", "64"])
    lattice, per = rng.choice([("fcc", 4), ("bcc", 2), ("hcp", 4)])
    a = rng.uniform(3.5, 4.1) if lattice == "fcc" else rng.uniform(2.8, 3.3) if lattice == "bcc" else rng.uniform(2.9, 3.2)
    # atoms: the evaluation of the largest costs less than that of `eval_1m`
    top = {8: 700000, 16: 600000, 32: 150000, 64: 60000, 128: 30000}[K] / S
    if kind == "noalloc":
        top = min(top, (40 << 20) / (4 * S * K * 28 + 120))
    if kind in ("md", "md_host"):
        top = min(top / 8, 60000)
    n = logint(100, max(200, int(top)))
    r = (n / per) ** (1.0 / 3.0)
    if lattice == "hcp":
        r /= 1.4
    nx, ny = max(2, int(round(r * rng.uniform(0.8, 1.25)))), max(2, int(round(r * rng.uniform(0.8, 1.25))))
    nz = max(2, int(round(n / per / nx / ny)))
    vacuum = rng.choice([0.0, 0.0, 15.0]) if kind in ("eval", "single") else 0.0
    table = rng.choice([0, 0, 64, 256]) if kind in ("eval", "single") and K <= 32 else 0
    return _drawn(kind, lattice=lattice, a=round(a, 3), nx=nx, ny=ny, nz=nz, S=S, K=K, net=net, precision=precision,
                  act=rng.choice(["tanh", "tanh", "squareplus"]), sigma=round(rng.uniform(0.05, 0.15), 3), table=table,
                  skin=0.0 if kind == "single" else rng.choice([0.0, 1.0]) if kind in ("eval", "noalloc", "descriptors") else 1.0,
                  vacuum=vacuum, steps={"md": 10, "md_host": 5}.get(kind, 0))


def _drawn(kind, **kw):
    c = _case("", kind, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _crystal(case, seed):
    pos, box = I.lattice(case["lattice"], (case["nx"], case["ny"], case["nz"]), case["a"])
    rng = np.random.default_rng(seed)
    pbc = np.ones(3, dtype=np.int32)
    if case["vacuum"] > 0.0:      # a film: open along z, vacuum on both sides
        pbc[2] = 0
        box = box + np.array([0.0, 0.0, case["vacuum"]])
        pos = pos + np.array([0.0, 0.0, 0.5 * case["vacuum"]])
    pos = I.jitter_and_wrap(pos, box, case["sigma"], rng)
    types = rng.integers(0, case["S"], size=len(pos)).astype(np.int32)
    masses = np.asarray(MASSES)[types]
    return I.System(pos, types, box, pbc, vel=I.maxwell_velocities(masses, 300.0, rng), masses=masses)


def _uneven(case, seed):
    """Systems of the `batch` / `serve` workloads' recipe; the sizes are the
    case's own, positions and species the seed's."""
    size, rng = np.random.default_rng(61), np.random.default_rng(seed)
    lo, out = (32 if case["kind"] == "batch" else 64), []
    for _ in range(case["systems"]):
        n = math.exp(size.uniform(math.log(lo), math.log(case["n_max"])))
        kind = ["fcc", "bcc", "hcp"][int(size.integers(0, 3 if case["kind"] == "batch" else 2))]
        a, ns = size.uniform(2.9, 4.1), int(size.integers(1, case["S"] + 1))
        basis, cell = I._BASIS[kind]
        reps = I._best_reps(n, basis.shape[0], cell)
        sigma = rng.uniform(0.05, 0.15) if case["kind"] == "batch" else 0.1
        pos, box = I.lattice(kind, reps, a)
        pos = I.jitter_and_wrap(pos, box, sigma, rng)
        types = rng.integers(0, ns, size=len(pos)).astype(np.int32)
        masses = np.asarray(MASSES)[types]
        out.append(I.System(pos, types, box, np.ones(3, dtype=np.int32),
                            vel=I.maxwell_velocities(masses, 300.0, rng), masses=masses))
    return out


def _params(case):
    """The potential: random weights whose first layer is normalised by the
    descriptor RMS of a small cell of the same lattice (stored with a trained
    potential; formed here in FP64)."""
    widths = [int(w) for w in case["net"].split("-")]
    args = (case["S"], case["K"], case["rc"], widths)
    p = I.random_model(*args, seed=17, activation=case["act"], masses=MASSES[:case["S"]])
    if case["systems"]:
        cell = dict(case, lattice="fcc", a=3.6, nx=4, ny=4, nz=4, vacuum=0.0)
    else:
        reps = 6 if case["lattice"] == "bcc" else 4
        cell = dict(case, nx=reps, ny=reps, nz=reps, vacuum=0.0)
    s = _crystal(cell, 3)
    G = _evaluate64(p, case, s.pos, s.types, s.box, s.pbc, descriptors=True)
    scale = [np.sqrt((G[s.types == t] ** 2).mean(axis=0)) for t in range(case["S"])]
    return I.random_model(*args, seed=17, activation=case["act"], masses=MASSES[:case["S"]], feature_scale=scale)


def prepare(case, seed):
    st = {"case": case}
    p = _params(case)
    model = tmd.Model(p, precision=case["precision"])
    if case["table"]:
        model.set_radial_table_values(case["table"], *_table_values(case))
    st["model"] = model
    kind = case["kind"]
    if kind in ("batch", "serve"):
        systems = _uneven(case, seed)
        b = tmd.Batch(systems, skin=case["skin"], rebuild_every=0 if kind == "batch" else 5)
        ids = np.sort(np.random.default_rng(62).permutation(case["systems"])[:case["active"]]).astype(np.int32)
        b.compute(model, ids)                       # resident tables and forces
        st.update(batch=b, ids=ids)
        return st
    s = _crystal(case, seed)
    st.update(box=s.box, pbc=s.pbc)
    if kind == "md":
        g = tmd.System(s.n, s.box, s.pbc, skin=case["skin"])
        g.set_state(s.pos, s.vel, s.types, s.masses)
        g.step(model, 1.0, 0, thermo=False)         # table and forces at the start
        st["system"] = g
        return st
    if kind == "md_host":
        g = tmd.System(s.n, s.box, s.pbc, skin=case["skin"])
        g.set_state(s.pos, s.vel, s.types, s.masses)
        g.step(model, 1.0, 0, thermo=False)
        pos, vel, f = g.get_state()
        st.update(system=g, pos=torch.from_numpy(pos).pin_memory(), vel=torch.from_numpy(vel).pin_memory(),
                  forces=torch.from_numpy(f).pin_memory())
        return st
    pos = torch.as_tensor(s.pos, dtype=torch.float64, device="cuda")
    types = torch.as_tensor(s.types, dtype=torch.int32, device="cuda")
    nl = tmd.NeighborList()
    st.update(pos=pos, types=types, nl=nl)
    if kind != "single":
        nl.build(pos, types, s.box, s.pbc, case["rc"] + case["skin"])
    if kind == "noalloc":                           # the caller's own table, on the device
        off, nbr, sh = nl.export()
        sh4 = np.concatenate([sh, s.types[nbr].astype(np.int8)[:, None]], axis=1)
        st.update(off=torch.as_tensor(off, device="cuda"), nbr=torch.as_tensor(nbr, device="cuda"),
                  shift4=torch.as_tensor(np.ascontiguousarray(sh4), device="cuda"))
        del st["nl"]
    if kind != "descriptors":
        red = torch.zeros(10, dtype=torch.float64, device="cuda")
        st.update(red=red, energy=red[:1], virial=red[1:], e_atom=torch.zeros(s.n, dtype=torch.float32, device="cuda"),
                  forces=torch.zeros((s.n, 3), dtype=torch.float32, device="cuda"))
    return st


def run(st):
    case, model = st["case"], st["model"]
    kind = case["kind"]
    if kind == "batch":
        e, w = st["batch"].compute(model, st["ids"])
        f = [st["batch"].get_system(int(k))[2] for k in st["ids"][:4]]     # structures still being relaxed
        return {"energy": e.astype(np.float32), "virial": _kept(w.astype(np.float32), case),
                "forces": [_kept(x, case) for x in f]}
    if kind == "serve":
        th = st["batch"].step(model, st["ids"], 1.0, case["steps"])
        pos, vel, f = st["batch"].get_system(int(st["ids"][0]))     # the state of a finished request
        return {"energy": np.array([t["e_pot"] for t in th], dtype=np.float32),
                "virial": _kept(np.array([t["virial"] for t in th], dtype=np.float32), case),
                "pos": pos, "vel": vel.astype(np.float32), "forces": _kept(f, case)}
    if kind == "md":
        st["system"].step(model, 1.0, case["steps"], rebuild_every=5, thermo=False)
        pos, vel, f = st["system"].get_state()
        return {"pos": pos, "vel": vel.astype(np.float32), "forces": _kept(f, case)}
    if kind == "md_host":
        st["system"].step_host(model, st["pos"], st["vel"], st["forces"], 1.0, case["steps"], rebuild_every=5)
        return {"pos": st["pos"], "vel": st["vel"].float(), "forces": _kept(st["forces"], case)}
    if kind == "descriptors":
        G, dG = tmd.descriptors(model, st["nl"], st["pos"], st["types"], st["box"], with_grad=True)
        return {"G": G, "dG": _kept(dG, case)}
    out = (st["energy"], st["e_atom"], st["forces"], st["virial"])
    if kind == "noalloc":
        tmd.compute_noalloc(model, st["off"], st["nbr"], st["shift4"], st["pos"], st["types"], st["box"], *out)
    else:
        if kind == "single":
            st["nl"].build(st["pos"], st["types"], st["box"], st["pbc"], case["rc"])
        tmd.compute(model, st["nl"], st["pos"], st["types"], st["box"], *out)
    red = st["red"].float()
    return {"energy": red[:1], "virial": _kept(red[1:], case), "e_atom": st["e_atom"],
            "forces": _kept(st["forces"], case)}


def _kept(x, case):
    """Forces, dE/dG or virials as the program keeps them: bfloat16 for the BF16 form."""
    if case["precision"] != "bf16":
        return x
    return (torch.from_numpy(x) if isinstance(x, np.ndarray) else x).to(torch.bfloat16)


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Bytes in and out once (positions, species, the table where it is an
    input, outputs, weights) and the multiply-adds of the method: 16
    independent moment components (1 + 3 + 5 + 7) per channel and pair, once
    forward and twice backward, the radial functions, and the network forward
    and for its input gradient."""
    K, S = case["K"], case["S"]
    dims = [4 * K * S] + [int(w) for w in case["net"].split("-")] + [1]
    mac = sum(a * b for a, b in zip(dims, dims[1:]))
    if case["systems"]:
        sizes = _uneven_sizes(case)
        n, pairs, listed_pairs = sum(x[0] for x in sizes), sum(x[1] for x in sizes), 0.0
    else:
        per = {"fcc": (4, 1.0), "bcc": (2, 1.0), "hcp": (4, math.sqrt(8.0))}[case["lattice"]]
        n = per[0] * case["nx"] * case["ny"] * case["nz"]
        density = per[0] / (per[1] * case["a"] ** 3)
        pairs = n * density * 4.0 / 3.0 * math.pi * case["rc"] ** 3
        listed_pairs = n * density * 4.0 / 3.0 * math.pi * (case["rc"] + case["skin"]) ** 3
    weights = 4 * S * mac
    fwd, bwd = 2 * 16 * K + 8 * K + 50, 4 * 16 * K + 10 * K + 165
    evals = max(1, case["steps"])
    flops = evals * (pairs * (fwd + bwd) + 4 * n * mac)
    kind = case["kind"]
    if kind == "descriptors":
        return {"bytes": n * (28 + 8 * dims[0]) + 8 * listed_pairs + weights, "flops": pairs * fwd + 4 * n * mac}
    if kind in ("eval", "noalloc"):
        return {"bytes": n * (28 + 16) + 8 * listed_pairs + weights, "flops": flops}
    if kind == "single":
        return {"bytes": n * (28 + 16) + weights, "flops": flops}
    if kind == "batch":
        return {"bytes": n * (28 + 12) + 80 * case["active"] + weights, "flops": flops}
    return {"bytes": evals * n * 120 + weights, "flops": flops}     # state read and written every step


def _uneven_sizes(case):
    size = np.random.default_rng(61)
    lo, out = (32 if case["kind"] == "batch" else 64), []
    for _ in range(case["systems"]):
        n = math.exp(size.uniform(math.log(lo), math.log(case["n_max"])))
        kind = ["fcc", "bcc", "hcp"][int(size.integers(0, 3 if case["kind"] == "batch" else 2))]
        a = size.uniform(2.9, 4.1)
        size.integers(1, case["S"] + 1)
        basis, cell = I._BASIS[kind]
        reps = I._best_reps(n, basis.shape[0], cell)
        m = basis.shape[0] * reps[0] * reps[1] * reps[2]
        vol = float(np.prod(np.asarray(cell) * a * np.asarray(reps)))
        out.append((m, m * m / vol * 4.0 / 3.0 * math.pi * case["rc"] ** 3))
    ids = np.sort(np.random.default_rng(62).permutation(case["systems"])[:case["active"]])
    return [out[i] for i in ids]


# ---------------------------------------------------------------------------
# the method in 64 bits, plain torch
# ---------------------------------------------------------------------------
def exact(case, seed):
    p = _params(case)
    if case["systems"]:
        systems = _uneven(case, seed)
        ids = np.sort(np.random.default_rng(62).permutation(case["systems"])[:case["active"]])
        if case["kind"] == "batch":
            r = [_evaluate64(p, case, s.pos, s.types, s.box, s.pbc) for s in (systems[i] for i in ids)]
            return {"energy": np.array([x["energy"] for x in r]), "virial": np.array([x["virial"] for x in r]),
                    "forces": [x["forces"] for x in r[:4]]}
        r = [_dynamics64(p, case, systems[i]) for i in ids]
        return {"energy": np.array([x["energy"] for x in r]), "virial": np.array([x["virial"] for x in r]),
                "pos": r[0]["pos"], "vel": r[0]["vel"], "forces": r[0]["forces"]}
    s = _crystal(case, seed)
    if case["kind"] in ("md", "md_host"):
        r = _dynamics64(p, case, s)
        return {k: r[k] for k in ("pos", "vel", "forces")}
    r = _evaluate64(p, case, s.pos, s.types, s.box, s.pbc, gradients=case["kind"] == "descriptors")
    if case["kind"] == "descriptors":
        return {"G": r["G"], "dG": r["dG"]}
    return {"energy": np.array([r["energy"]]), "virial": r["virial"].ravel(), "e_atom": r["e_atom"],
            "forces": r["forces"]}


def _dynamics64(p, case, s):
    """Velocity-Verlet of 1 fs; the table is rebuilt, and positions wrapped
    with it, on every fifth step (systems of a batch also on their last step
    where that is one)."""
    x, v, m = s.pos.copy(), s.vel.copy(), s.masses[:, None]
    f = _evaluate64(p, case, x, s.types, s.box, s.pbc)["forces"]
    for it in range(1, case["steps"] + 1):
        v = v + 0.5 * f / (m * ACC)
        x = x + v
        if it % 5 == 0:
            x = x - np.floor(x / s.box) * s.box
        r = _evaluate64(p, case, x - np.floor(x / s.box) * s.box, s.types, s.box, s.pbc)
        f = r["forces"]
        v = v + 0.5 * f / (m * ACC)
    return {"pos": x, "vel": v, **{k: r[k] for k in ("forces", "energy", "virial")}}


def _table_values(case):
    return I.embedding_radial_table(case["S"], case["K"], case["rc"], case["table"], seed=5)


def _pairs64(pos, box, pbc, rc):
    """For chunks of atoms: (atoms, neighbour ids [m, w], displacement [m, w, 3]);
    unused places have id -1."""
    dev = pos.device
    reach = [int(math.ceil(rc / float(L))) if b else 0 for L, b in zip(box, pbc)]
    xs, ids = [], []
    L = torch.as_tensor(np.asarray(box, dtype=np.float64), device=dev)
    for sx in range(-reach[0], reach[0] + 1):
        for sy in range(-reach[1], reach[1] + 1):
            for sz in range(-reach[2], reach[2] + 1):
                y = pos + torch.tensor([sx, sy, sz], dtype=torch.float64, device=dev) * L
                ok = ((y >= -rc) & (y <= L + rc)).all(1).nonzero()[:, 0]
                xs.append(y[ok])
                ids.append(ok)
    xs, ids = torch.cat(xs), torch.cat(ids)
    nc = [max(1, int((float(b) + 2 * rc) / rc)) for b in box]
    side = torch.tensor([(float(b) + 2 * rc) / c for b, c in zip(box, nc)], dtype=torch.float64, device=dev)
    top = torch.tensor(nc, device=dev) - 1

    def cell(y):
        c = ((y + rc) / side).long()
        return torch.minimum(torch.clamp(c, min=0), top)

    def flat(c):
        return (c[..., 0] * nc[1] + c[..., 1]) * nc[2] + c[..., 2]

    where = flat(cell(xs))
    order = torch.argsort(where, stable=True)
    where = where[order]
    total = nc[0] * nc[1] * nc[2]
    start = torch.searchsorted(where, torch.arange(total, device=dev))
    count = torch.bincount(where, minlength=total)
    occ = int(count.max())
    tab = torch.full((total + 1, occ), -1, dtype=torch.long, device=dev)
    tab[where, torch.arange(len(where), device=dev) - start[where]] = order
    steps = torch.tensor([(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)], device=dev)
    m = max(256, int(6e6 / (27 * occ)))
    mine = torch.argsort(flat(cell(pos)))
    for at in mine.split(m):
        c = cell(pos[at])[:, None, :] + steps
        inside = ((c >= 0) & (c <= top)).all(-1)
        cand = tab[torch.where(inside, flat(c), total)].reshape(len(at), -1)
        D = xs[cand.clamp(min=0)] - pos[at][:, None, :]
        r2 = (D * D).sum(-1)
        keep = (cand >= 0) & (r2 < rc * rc) & (r2 > 0)
        w = max(1, int(keep.sum(1).max()))
        first = torch.argsort((~keep).to(torch.uint8), dim=1, stable=True)[:, :w]
        ok = keep.gather(1, first)
        j = torch.where(ok, ids[cand.clamp(min=0)].gather(1, first), -1)
        yield at, j, D.gather(1, first[..., None].expand(-1, -1, 3))


def _moments64(u):
    x, y, z = u.unbind(-1)
    one = [torch.ones_like(x)]
    first = [x, y, z]
    second = [x * x, x * y, x * z, y * y, y * z, z * z]
    third = [x * x * x, x * x * y, x * x * z, x * y * y, x * y * z, x * z * z, y * y * y, y * y * z, y * z * z, z * z * z]
    return torch.stack(one + first + second + third, dim=-1)


TIMES = [1, 1, 1, 1, 1, 2, 2, 1, 2, 1, 1, 3, 3, 3, 6, 3, 1, 3, 3, 1]
RANK = [0] + [1] * 3 + [2] * 6 + [3] * 10


def _evaluate64(p, case, pos, types, box, pbc, descriptors=False, gradients=False):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f64 = dict(dtype=torch.float64, device=dev)
    S, K, rc, n = p.n_species, p.n_radial, p.rc, len(pos)
    x = torch.as_tensor(np.asarray(pos), **f64)
    t = torch.as_tensor(np.asarray(types), device=dev).long()
    mu, eta = torch.as_tensor(p.mu, **f64), torch.as_tensor(p.eta, **f64)
    T, rank = torch.tensor(TIMES, **f64), torch.tensor(RANK, device=dev)
    layers = [[(torch.as_tensor(W, **f64), torch.as_tensor(b, **f64)) for W, b in p.unpack(s)] for s in range(S)]
    grid = None
    if case["table"] and not descriptors:      # cubic Hermite through H and H' on the grid, zero from rc on
        H, dH = _table_values(case)
        pad = ((0, 0), (0, 0), (0, 3), (0, 0))
        r_g = np.arange(H.shape[2] + 3) / case["table"]
        live = (r_g < rc)[None, None, :, None]
        grid = [torch.as_tensor(np.pad(a, pad) * live, **f64) for a in (H, dH)]
    e_atom = torch.zeros(n, **f64)
    forces, virial = torch.zeros((n, 3), **f64), torch.zeros((3, 3), **f64)
    Gs = torch.zeros((n, 4 * K * S), **f64) if descriptors or gradients else None
    dGs = torch.zeros_like(Gs) if gradients else None
    for atoms, near, disp in _pairs64(x, box, pbc, rc):
        for part in torch.arange(len(atoms), device=dev).split(max(64, int(3e7 / (near.shape[1] * (K + 24))))):
            at, j = atoms[part], near[part]
            ok = j >= 0
            D = torch.where(ok[..., None], disp[part], torch.full_like(disp[part], rc))
            D.requires_grad_(not descriptors)
            r = D.norm(dim=-1)
            ti, tj = t[at][:, None].expand_as(j), t[j.clamp(min=0)]
            if grid is None:
                H = torch.exp(-eta[ti, tj] * (r[..., None] - mu[ti, tj]) ** 2)
                H = H * (0.5 * (torch.cos(math.pi * r / rc) + 1.0))[..., None]
            else:
                h = 1.0 / case["table"]
                cell = torch.clamp((r.detach() / h).long(), max=grid[0].shape[2] - 2)
                s = (r / h - cell)[..., None]
                y0, y1 = grid[0][ti, tj, cell], grid[0][ti, tj, cell + 1]
                d0, d1 = grid[1][ti, tj, cell] * h, grid[1][ti, tj, cell + 1] * h
                H = y0 + s * (d0 + s * ((3 * (y1 - y0) - 2 * d0 - d1) + s * (2 * (y0 - y1) + d0 + d1)))
            H = torch.where(ok[..., None], H, torch.zeros_like(H))
            M = _moments64(D / r[..., None])
            G = []
            for b in range(S):
                Hb = H if S == 1 else torch.where((tj == b)[..., None], H, torch.zeros_like(H))
                P = Hb.transpose(1, 2) @ M                          # [m, K, 20]
                sq = P * P * T
                G.append(torch.stack([P[..., 0].abs()] + [sq[..., rank == q].sum(-1) for q in (1, 2, 3)], dim=-1))
            G = torch.stack(G, dim=1).reshape(len(at), -1)
            if Gs is not None:
                Gs[at] = G.detach()
            if descriptors:
                continue
            if gradients:
                G.retain_grad()
            e = torch.zeros(len(at), **f64)
            for q in range(S):
                a = G
                for W, b in layers[q][:-1]:
                    z = a @ W.T + b
                    a = torch.tanh(z) if p.activation == "tanh" else 0.5 * (z + torch.sqrt(z * z + p.squareplus_b))
                W, b = layers[q][-1]
                e = torch.where(t[at] == q, (a @ W.T + b)[:, 0], e)
            e.sum().backward()
            e_atom[at] = e.detach()
            if gradients:
                dGs[at] = G.grad
            g = torch.where(ok[..., None], D.grad, torch.zeros_like(D))
            forces.index_add_(0, at, g.sum(1))
            forces.index_add_(0, j[ok], -g[ok])
            virial -= torch.einsum("pwa,pwb->ab", torch.where(ok[..., None], D.detach(), torch.zeros_like(g)), g)
    if descriptors:
        return Gs.cpu().numpy()
    out = {"energy": float(e_atom.sum()), "e_atom": e_atom.cpu().numpy(), "forces": forces.cpu().numpy(),
           "virial": virial.cpu().numpy()}
    if gradients:
        out.update(G=Gs.cpu().numpy(), dG=dGs.cpu().numpy())
    return out
