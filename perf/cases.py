"""The calls this library is timed on, from the smallest box to the million-atom one.

Each case is one pass a user's program makes: a neighbour list and the energy,
forces and virial on it (an MD engine's step), a packed batch of molecules, an
energy alone (Monte Carlo), a short molecular-dynamics run, or the autograd
function in both directions.  The models are the architectures this repository
is configured, tested and benchmarked with; their weights are drawn once from a
fixed seed, as a program loads one model, and every structure is drawn from the
case's seed.  `exact` evaluates the same model in float64 with plain torch.
"""
import math
import struct

import numpy as np
import torch

from paper_2304_10061_gb300 import Allegro, AllegroEnergy

RC, BESSEL, P_ENV, AVG_NEIGH = 4.0, 8, 6, 27.0
WATER = (0.63, 0.30, 0.05, 0.015, 0.005)          # H, O, C, N, S
MASSES = (1.008, 15.999, 12.011, 14.007, 32.06)
CHARGES = (1, 8, 6, 7, 16)
DENSITY = 0.1                                      # atoms per cubic Angstrom (liquid water)
# ordered pairs with a cutoff of their own (row = centre): H-H 3.0, H-C 1.25, H-O 1.25, O-H 3.0
PAIR_RC = np.full((5, 5), RC)
PAIR_RC[0, 0], PAIR_RC[0, 2], PAIR_RC[0, 1], PAIR_RC[1, 0] = 3.0, 1.25, 1.25, 3.0

MODELS = {
    # one layer, the smallest model
    "small": dict(ns=2, lmax=1, nl=1, C=8, tb=(32,), lat=(32,), edge=()),
    # the two-layer model of the solvated-protein, molecule and million-atom workloads
    "two_layer": dict(ns=5, lmax=2, nl=2, C=64, tb=(64, 128, 256), lat=(256, 256), edge=(128,)),
    # the paper's production model, 1024 wide
    "production": dict(ns=5, lmax=2, nl=2, C=64, tb=(128, 256, 512, 1024), lat=(1024, 1024, 1024), edge=(128,)),
    # three layers, l_max 3, 128 channels (the four-million-atom model)
    "three_layer": dict(ns=5, lmax=3, nl=3, C=128, tb=(64, 128, 512), lat=(512, 512), edge=(128,)),
}


def listed():
    box = dict(kind="box", triclinic=False, pair_cutoffs=False, zbl=False, forces=True)
    return [
        # the smallest call: a 64-atom periodic box, where launches and waits are the time
        dict(box, name="box_64_fp32", model="small", precision="fp32", n=64),
        # a geometry optimiser or a trainer in torch: the energy's autograd function, forward and backward
        dict(name="autograd_997_fp32", kind="autograd", model="two_layer", precision="fp32", n=997),
        # the production precision of the paper (float32 with TF32 products) on its 3,072-atom water box
        dict(box, name="box_3072_tf32", model="two_layer", precision="tf32", n=3072),
        # molecular dynamics of a mid-sized box: 10 steps of 1 fs, the neighbour list reused within a skin
        dict(name="md_4096_bf16", kind="md", model="two_layer", precision="bf16", n=4096, steps=10, skin=0.4),
        # batched inference: 2,048 molecules of 8 to 64 atoms in one packed list, replayed as a CUDA graph
        dict(name="molecules_2048_bf16", kind="molecules", model="two_layer", precision="bf16", n_mol=2048, graphs=True),
        # Monte Carlo: energies alone, an odd number of atoms in a triclinic cell
        dict(box, name="energy_12345_bf16", model="two_layer", precision="bf16", n=12345, triclinic=True, forces=False),
        # the solvated-protein-like box in all float32
        dict(box, name="box_23552_fp32", model="two_layer", precision="fp32", n=23552),
        # the production model with its per-pair cutoffs and ZBL repulsion, a ragged size
        dict(box, name="production_16411_bf16", model="production", precision="bf16", n=16411, pair_cutoffs=True, zbl=True),
        # the three-layer model under FP8 MLPs
        dict(box, name="three_layer_16384_fp8", model="three_layer", precision="fp8", n=16384),
        # the three-layer model at a size that fills the GPU
        dict(box, name="three_layer_65536_bf16", model="three_layer", precision="bf16", n=65536),
        # the largest: the million-atom box
        dict(box, name="box_1048576_bf16", model="two_layer", precision="bf16", n=1048576),
    ]


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n | 1 if rng.random() < 0.5 else n

    kind = rng.choice(("box", "box", "box", "energy", "production", "three_layer", "md", "molecules", "autograd"))
    if kind == "autograd":
        return dict(kind="autograd", model="two_layer", precision=rng.choice(("fp32", "tf32", "bf16")), n=size(200, 8000))
    if kind == "md":
        return dict(kind="md", model="two_layer", precision=rng.choice(("fp32", "bf16")), n=size(800, 8000),
                    steps=rng.randint(2, 10), skin=rng.choice((0.0, 0.4)))
    if kind == "molecules":
        return dict(kind="molecules", model="two_layer", precision=rng.choice(("bf16", "fp32")),
                    n_mol=size(8, 2048), graphs=rng.random() < 0.5)
    case = dict(kind="box", triclinic=rng.random() < 0.25, pair_cutoffs=False, zbl=False, forces=kind != "energy")
    if kind == "production":
        return dict(case, model="production", precision=rng.choice(("bf16", "tf32")), n=size(512, 16411),
                    pair_cutoffs=True, zbl=True)
    if kind == "three_layer":
        precision = rng.choice(("bf16", "bf16", "fp8"))
        return dict(case, model="three_layer", precision=precision, n=size(512, 16384 if precision == "fp8" else 65536))
    if rng.random() < 0.15:
        return dict(case, model="small", precision=rng.choice(("fp32", "bf16")), n=size(64, 20000), triclinic=False)
    precision = rng.choice(("fp32", "tf32", "bf16", "bf16"))
    return dict(case, model="two_layer", precision=precision, pair_cutoffs=rng.random() < 0.25,
                n=size(1000, {"fp32": 40000, "tf32": 100000, "bf16": 400000}[precision]))


# ---------------------------------------------------------------------------
# models
# ---------------------------------------------------------------------------
def _shapes(a):
    """(name, shape) of the float32 arrays in file order; sigma and mu (float64) follow."""
    lm, out, fan = a["lmax"] + 1, [], 2 * a["ns"] + BESSEL
    nw = a["C"] * lm
    for k, w in enumerate(a["tb"]):
        out.append((("tb", k), (w, fan)))
        fan = w
    out.append((("embed",), (nw, fan)))
    kin = fan
    for L in range(1, a["nl"] + 1):
        out.append((("env", L), (nw, kin)))
        out.append((("tp", L), (lm, 2, lm, 2, lm)))
        fan = kin + a["C"]
        for k, w in enumerate(a["lat"]):
            out.append((("lat", L, k), (w, fan)))
            fan = w
        kin = fan
    for k, w in enumerate(a["edge"] + (1,)):
        out.append((("edge", k), (w, fan)))
        fan = w
    return out


def _weights(name):
    """Matrices N(0, 1 / fan_in), path weights N(0, 1), scale 1 + 0.1 N(0, 1), shift 10 N(0, 1)."""
    a, rng, w = MODELS[name], np.random.default_rng(1), {}
    for key, shape in _shapes(a):
        x = rng.standard_normal(shape)
        w[key] = (x if key[0] == "tp" else x * math.sqrt(1.0 / shape[1])).astype(np.float32)
    w["sigma"] = 1.0 + 0.1 * rng.standard_normal(a["ns"])
    w["mu"] = 10.0 * rng.standard_normal(a["ns"])
    return w


def _blob(name):
    """The library's weights image ("ALGW" version 1)."""
    a, w = MODELS[name], _weights(name)
    parts = [b"ALGW", struct.pack("<Idd", 1, RC, AVG_NEIGH),
             struct.pack("<9i", a["ns"], BESSEL, P_ENV, a["lmax"], a["nl"], a["C"], len(a["tb"]), len(a["lat"]), len(a["edge"]))]
    widths = a["tb"] + a["lat"] + a["edge"]
    parts.append(struct.pack("<%di" % len(widths), *widths))
    parts += [w[key].tobytes() for key, _ in _shapes(a)]
    return b"".join(parts) + w["sigma"].tobytes() + w["mu"].tobytes()


# ---------------------------------------------------------------------------
# structures
# ---------------------------------------------------------------------------
def _species(a, n, gen, dev):
    mix = WATER if a["ns"] == 5 else (43 / 64, 21 / 64)
    edges = torch.tensor(np.cumsum(mix)[:-1], device=dev)
    return torch.bucketize(torch.rand(n, generator=gen, device=dev, dtype=torch.float64), edges).to(torch.int32)


def _box(case, seed, dev="cuda"):
    """Jittered lattice at the density of water: n of the smallest cube of sites, each displaced by
    up to a quarter of the spacing (any two atoms at least half a spacing apart)."""
    gen = torch.Generator(device=dev).manual_seed(seed)
    n, m = case["n"], 1
    while m ** 3 < n:
        m += 1
    side = (n / DENSITY) ** (1.0 / 3.0)
    site = torch.sort(torch.randperm(m ** 3, generator=gen, device=dev)[:n])[0]
    grid = torch.stack([site // (m * m), (site // m) % m, site % m], 1).to(torch.float64)
    frac = (grid + 0.5 + 0.5 * (torch.rand(n, 3, generator=gen, device=dev, dtype=torch.float64) - 0.5)) / m
    cell = np.eye(3) * side
    if case.get("triclinic"):
        cell[1, 0], cell[2, 0], cell[2, 1] = 0.20 * side, -0.10 * side, 0.15 * side
    pos = (frac @ torch.tensor(cell, device=dev)).contiguous()
    return pos, _species(MODELS[case["model"]], n, gen, dev), cell


def _molecules(n_mol, seed):
    """Gas-phase molecules of 8 to 64 atoms: random walks of bonds 1.0 to 1.5 Angstrom with no two
    atoms of a molecule nearer than 0.9; all walks step together, a failed step is drawn again."""
    rng = np.random.default_rng(seed)
    sizes = np.random.default_rng(n_mol).integers(8, 65, n_mol)   # the batch's sizes are the case's, the geometries the seed's
    pos = np.full((n_mol, 64, 3), 1e6)
    pos[:, 0] = 0.0
    done, at, fails = np.ones(n_mol, int), np.zeros(n_mol, int), np.zeros(n_mol, int)
    while True:
        act = np.nonzero(done < sizes)[0]
        if not act.size:
            break
        v = rng.normal(size=(act.size, 3))
        v *= rng.uniform(1.0, 1.5, (act.size, 1)) / np.linalg.norm(v, axis=1, keepdims=True)
        new = pos[act, at[act]] + v
        good = ((pos[act] - new[:, None]) ** 2).sum(-1).min(1) >= 0.81
        g, b = act[good], act[~good]
        pos[g, done[g]] = new[good]
        at[g] = done[g]
        done[g] += 1
        fails[g] = 0
        fails[b] += 1
        stuck = b[fails[b] > 200]
        at[stuck] = rng.integers(0, done[stuck])
        fails[stuck] = 0
    keep = np.arange(64)[None, :] < sizes[:, None]
    spec = np.searchsorted(np.cumsum(WATER)[:-1], rng.random(int(sizes.sum()))).astype(np.int32)
    return pos[keep], spec, np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def prepare(case, seed):
    model = Allegro(_blob(case["model"]), precision=case["precision"])
    state = dict(case=case, model=model)
    if case["kind"] == "molecules":
        pos, types, offsets = _molecules(case["n_mol"], seed)
        state.update(pos=torch.tensor(pos, device="cuda"), types=torch.tensor(types, device="cuda"), offsets=offsets)
        model.set_graphs(case["graphs"])
        return state
    pos, types, cell = _box(case, seed)
    state.update(pos=pos, types=types, cell=cell)
    if case["kind"] == "md":
        state["vel"] = _velocities(types, seed)
        model.set_md_skin(case["skin"])
    if case.get("pair_cutoffs"):
        model.set_pair_cutoffs(PAIR_RC)
    if case.get("zbl"):
        model.set_zbl(CHARGES)
    return state


def _velocities(types, seed):
    """Maxwell-Boltzmann at 300 K (Angstrom / fs)."""
    gen = torch.Generator(device=types.device).manual_seed(seed + 1)
    mass = torch.tensor(MASSES, dtype=torch.float64, device=types.device)[types.long()]
    kt = 8.617333e-5 * 300.0 * 9.648533212e-3
    return torch.randn(len(types), 3, generator=gen, device=types.device, dtype=torch.float64) * (kt / mass).sqrt()[:, None]


def run(state):
    case, m = state["case"], state["model"]
    if case["kind"] == "autograd":
        pos = state["pos"].detach().requires_grad_(True)
        energy = AllegroEnergy.apply(pos, m, state["types"], state["cell"], None)
        energy.backward()
        return dict(E=energy.detach(), grad=pos.grad)
    if case["kind"] == "md":
        pos, vel = state["pos"].clone(), state["vel"].clone()
        torch.cuda.current_stream().synchronize()    # the run works on a stream of the model's own
        e_pot, e_kin = m.md_verlet(pos, vel, state["types"], MASSES, 1.0, case["steps"], cell=state["cell"])
        return dict(pos=pos, vel=vel, E_pot=e_pot, E_kin=e_kin)
    if case["kind"] == "molecules":
        n_edges = m.neighbors_batched(state["offsets"], state["pos"], state["types"])
    else:
        n_edges = m.neighbors(state["pos"], state["types"], state["cell"])
    forces = case.get("forces", True)
    return dict(m.energy_forces(forces=forces, virial=forces), n_edges=n_edges)


def work(case):
    a = MODELS[case["model"]]
    macs = [s[0] * s[1] for key, s in _shapes(a) if key[0] in ("tb", "embed", "env", "lat")] + [a["lat"][-1]]
    if case["kind"] == "molecules":
        n, per_atom, n_struct = 36 * case["n_mol"], 15.9, case["n_mol"]
    else:
        n, per_atom, n_struct = case["n"], 11.25 if case.get("pair_cutoffs") else 25.1, 1
    evals = case["steps"] + 1 if case["kind"] == "md" else 1
    both = case["kind"] != "box" or case["forces"]
    flops = 2.0 * sum(macs) * n * per_atom * (2 if both else 1) * evals
    weights = sum(int(np.prod(s)) for _, s in _shapes(a)) * (4 if case["precision"] in ("fp32", "tf32") else 2)
    if case["kind"] == "md":
        return dict(bytes=weights + n * (24 + 24 + 4 + 24 + 24) + 16 * evals, flops=flops)
    return dict(bytes=weights + n * (24 + 4 + 8 + (24 if both else 0)) + n_struct * (8 + (72 if both else 0)), flops=flops)


# ---------------------------------------------------------------------------
# the same model in float64
# ---------------------------------------------------------------------------
def _harmonics(lmax, r):
    x, y, z = r.unbind(-1)
    s = math.sqrt
    Y = [torch.ones_like(x), s(3) * y, s(3) * z, s(3) * x]
    if lmax >= 2:
        Y += [s(15) * x * y, s(15) * y * z, s(5) / 2 * (3 * z * z - 1), s(15) * x * z, s(15) / 2 * (x * x - y * y)]
    if lmax >= 3:
        Y += [s(35 / 8) * y * (3 * x * x - y * y), s(105) * x * y * z, s(21 / 8) * y * (5 * z * z - 1),
              s(7) / 2 * z * (5 * z * z - 3), s(21 / 8) * x * (5 * z * z - 1), s(105) / 2 * z * (x * x - y * y),
              s(35 / 8) * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _couplings(lmax):
    """For l1, l2, l3 <= lmax the tensor of unit norm that every rotation leaves as it is, its first
    nonzero entry positive: the null vector of two rotations' D1 x D2 x D3 - 1."""
    rng = np.random.default_rng(0)
    pts = rng.normal(size=(64, 3))
    pts /= np.linalg.norm(pts, axis=1, keepdims=True)
    Y0 = _harmonics(3, torch.tensor(pts)).numpy()
    D = []
    for _ in range(2):
        q, _r = np.linalg.qr(rng.normal(size=(3, 3)))
        q *= np.sign(np.linalg.det(q))
        D.append([np.linalg.lstsq(Y0[:, l * l:(l + 1) ** 2], _harmonics(3, torch.tensor(pts @ q.T)).numpy()[:, l * l:(l + 1) ** 2],
                                  rcond=None)[0].T for l in range(lmax + 1)])
    out = {}
    for l1 in range(lmax + 1):
        for l2 in range(lmax + 1):
            for l3 in range(abs(l1 - l2), min(l1 + l2, lmax) + 1):
                rows = [np.kron(np.kron(d[l1], d[l2]), d[l3]) for d in D]
                t = np.linalg.svd(np.concatenate([k - np.eye(len(k)) for k in rows]))[2][-1]
                t = np.where(np.abs(t) < 1e-9, 0.0, t / np.linalg.norm(t))
                t *= np.sign(t[np.nonzero(t)[0][0]])
                out[l1, l2, l3] = t.reshape(2 * l1 + 1, 2 * l2 + 1, 2 * l3 + 1)
    return out


def _tensors(a, w):
    """Per layer W[a, b, c]: features before the layer x harmonics -> features after it, keeping the
    products that can still reach the scalar."""
    lmax, nl = a["lmax"], a["nl"]
    C = _couplings(lmax)

    def products(irreps):
        got = {(lo, p * (-1) ** l2) for l, p in irreps for l2 in range(lmax + 1)
               for lo in range(abs(l - l2), min(l + l2, lmax) + 1)}
        return sorted(got, key=lambda t: (t[0], -t[1]))

    def reaches(ir, steps):
        return ir == (0, 1) if steps == 0 else any(reaches(o, steps - 1) for o in products([ir]))

    sets = [[(l, (-1) ** l) for l in range(lmax + 1)]]
    for L in range(1, nl + 1):
        sets.append([ir for ir in products(sets[-1]) if reaches(ir, nl - L)])
    out = []
    for L in range(1, nl + 1):
        dim = [sum(2 * l + 1 for l, _ in s) for s in sets[L - 1:L + 1]]
        W, theta, c0 = np.zeros((dim[0], (lmax + 1) ** 2, dim[1])), w["tp", L].astype(np.float64), 0
        for lo, po in sets[L]:
            paths, a0 = [], 0
            for l1, p1 in sets[L - 1]:
                paths += [(l1, p1, l2, a0) for l2 in range(lmax + 1)
                          if abs(l1 - l2) <= lo <= l1 + l2 and po == p1 * (-1) ** l2]
                a0 += 2 * l1 + 1
            for l1, p1, l2, at in paths:
                t = theta[lo, (1 - po) // 2, l1, (1 - p1) // 2, l2] / math.sqrt(len(paths))
                W[at:at + 2 * l1 + 1, l2 * l2:(l2 + 1) ** 2, c0:c0 + 2 * lo + 1] += t * C[l1, l2, lo]
            c0 += 2 * lo + 1
        out.append(W)
    return out


class _Float64:
    """Energy, forces and virial of one model, differentiated by autograd, centres in blocks."""

    def __init__(self, name, pair_cutoffs=False, zbl=False, dev="cuda"):
        self.a, self.dev, self.zbl = MODELS[name], dev, zbl
        w = _weights(name)
        t = lambda x: torch.tensor(np.asarray(x, np.float64), device=dev)
        self.w = {k: t(v) for k, v in w.items()}
        self.W = [t(x) for x in _tensors(self.a, w)]
        self.rc = t(PAIR_RC if pair_cutoffs else np.full((self.a["ns"],) * 2, RC))
        self.Z = t(CHARGES)
        self.l_of = torch.tensor([l for l in range(self.a["lmax"] + 1) for _ in range(2 * l + 1)], device=dev)

    def edges(self, pos, types, cell, struct_of, a0, a1):
        """Edges of the centres [a0, a1): every image within one cell of the neighbour's own."""
        shifts = [(0, 0, 0)] if cell is None else [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)]
        c = torch.zeros(3, 3, dtype=torch.float64, device=self.dev) if cell is None else torch.tensor(cell, device=self.dev)
        rc2 = (self.rc ** 2)[types[a0:a1].long()][:, types.long()]
        own = torch.arange(a0, a1, device=self.dev)[:, None] == torch.arange(len(pos), device=self.dev)[None]
        found = []
        for s in shifts:
            off = torch.tensor(s, dtype=torch.float64, device=self.dev) @ c
            d2 = sum((pos[None, :, k] + off[k] - pos[a0:a1, None, k]) ** 2 for k in range(3))
            ok = d2 < rc2
            if s == (0, 0, 0):
                ok &= ~own
            if struct_of is not None:
                ok &= struct_of[a0:a1, None] == struct_of[None]
            i, j = ok.nonzero(as_tuple=True)
            found.append((i + a0, j, off.expand(len(i), 3)))
        return [torch.cat(x) for x in zip(*found)]

    def atoms(self, d, ti, tj, i, n):
        """Energies of n centres from their edge vectors; i: each edge's centre, from 0."""
        a, w = self.a, self.w
        C, lm = a["C"], a["lmax"] + 1
        r = d.norm(dim=1)
        rc = self.rc[ti, tj]
        x = r / rc
        u = (1 - 28 * x ** 6 + 48 * x ** 7 - 21 * x ** 8)[:, None]
        k = torch.arange(1, BESSEL + 1, dtype=torch.float64, device=self.dev)
        B = torch.sqrt(2 / rc)[:, None] * torch.sin(k * math.pi * x[:, None]) / r[:, None]
        Y = _harmonics(a["lmax"], d / r[:, None])
        one = torch.eye(a["ns"], dtype=torch.float64, device=self.dev)
        h = torch.cat([one[ti], one[tj], B], 1)
        for q in range(len(a["tb"])):
            h = torch.nn.functional.silu(h @ w["tb", q].T)
        h = u * h
        v0 = (h @ w["embed",].T).view(-1, C, lm)[:, :, self.l_of] * Y[:, None]
        gammas = []
        for L in range(1, a["nl"] + 1):
            env = (h @ w["env", L].T).view(-1, C, lm)[:, :, self.l_of] * Y[:, None]
            gammas.append(torch.zeros(n, C, Y.shape[1], dtype=torch.float64, device=self.dev).index_add(0, i, env) / math.sqrt(AVG_NEIGH))
            # the scalar of V^0 M^1 ... M^L with M^k = W^k . gamma^k, from its right end
            q = torch.einsum("iub,ab->iua", gammas[-1], self.W[L - 1][:, :, 0])
            for K in range(L - 1, 0, -1):
                q = torch.einsum("iub,iuc,abc->iua", gammas[K - 1], q, self.W[K - 1])
            h = torch.cat([h, (v0 * q[i]).sum(-1)], 1)
            for q in range(len(a["lat"])):
                h = torch.nn.functional.silu(h @ w["lat", L, q].T)
            h = u * h
        for q in range(len(a["edge"]) + 1):
            h = h @ w["edge", q].T
        e = torch.zeros(n, dtype=torch.float64, device=self.dev).index_add(0, i, h[:, 0])
        rep = 0.0
        if self.zbl:
            za, zb = self.Z[ti], self.Z[tj]
            s = r * (za ** 0.23 + zb ** 0.23) / (0.8854 * 0.529177)
            phi = sum(c * torch.exp(-b * s) for c, b in ((0.18175, 3.19980), (0.50986, 0.94229), (0.28022, 0.40290), (0.02817, 0.20162)))
            rep = torch.zeros(n, dtype=torch.float64, device=self.dev).index_add(0, i, 0.5 * 14.399645 * za * zb / r * phi * u[:, 0])
        return e, rep

    def evaluate(self, pos, types, cell=None, struct_of=None, n_struct=1, forces=True, block=2048):
        n = len(pos)
        E_atom, F, n_edges = torch.zeros(n, dtype=torch.float64, device=self.dev), torch.zeros_like(pos), 0
        W_atom = torch.zeros(n, 9, dtype=torch.float64, device=self.dev)
        for a0 in range(0, n, block):
            a1 = min(n, a0 + block)
            i, j, off = self.edges(pos, types, cell, struct_of, a0, a1)
            n_edges += len(i)
            d = ((pos[j] + off) - pos[i]).requires_grad_(forces)
            t = types[a0:a1].long()
            with torch.set_grad_enabled(forces):
                e, rep = self.atoms(d, types[i].long(), types[j].long(), i - a0, a1 - a0)
                e = self.w["sigma"][t] * e + self.w["mu"][t] + rep
            E_atom[a0:a1] = e.detach()
            if forces and len(i):
                (g,) = torch.autograd.grad(e.sum(), d)
                F.index_add_(0, i, g).index_add_(0, j, -g)
                W_atom.index_add_(0, i, -(d.detach()[:, :, None] * g[:, None, :]).reshape(-1, 9))
        s = torch.zeros(n, dtype=torch.long, device=self.dev) if struct_of is None else struct_of
        total = lambda v: torch.zeros((n_struct,) + v.shape[1:], dtype=torch.float64, device=self.dev).index_add(0, s, v)
        return dict(E=total(E_atom), E_atom=E_atom, F=F, virial=total(W_atom).view(-1, 3, 3), n_edges=n_edges)


def exact(case, seed):
    if work(case)["flops"] > 1.5e13 or case.get("n", 0) > 50000:   # float64 at about 1 TFLOP/s, all pairs of atoms
        return None
    ref = _Float64(case["model"], case.get("pair_cutoffs", False), case.get("zbl", False))
    if case["kind"] == "molecules":
        pos, types, offsets = _molecules(case["n_mol"], seed)
        pos, types = torch.tensor(pos, device="cuda"), torch.tensor(types, device="cuda")
        struct_of = torch.tensor(np.repeat(np.arange(case["n_mol"]), np.diff(offsets)), device="cuda")
        return ref.evaluate(pos, types, None, struct_of, case["n_mol"])
    pos, types, cell = _box(case, seed)
    if case["kind"] == "md":
        vel = _velocities(types, seed)
        mass = torch.tensor(MASSES, dtype=torch.float64, device="cuda")[types.long()][:, None]
        acc, e_pot, e_kin = 9.648533212e-3 / mass, [], []
        for k in range(case["steps"] + 1):
            if k:
                vel = vel + 0.5 * acc * F
                pos = pos + vel
            got = ref.evaluate(pos, types, cell)
            F = got["F"]
            if k:
                vel = vel + 0.5 * acc * F
            e_pot.append(got["E"].item())
            e_kin.append((0.5 * (mass / 9.648533212e-3) * vel ** 2).sum().item())
        return dict(pos=pos, vel=vel, E_pot=np.array(e_pot), E_kin=np.array(e_kin))
    got = ref.evaluate(pos, types, cell, forces=case.get("forces", True))
    if case["kind"] == "autograd":
        return dict(E=got["E"][0], grad=-got["F"])
    if not case["forces"]:
        return dict(E=got["E"], E_atom=got["E_atom"], n_edges=got["n_edges"])
    if case["precision"] == "fp8":   # three mantissa bits: forces carry an error of order 10 % by design
        got.update(F=None, virial=None)
    return got
