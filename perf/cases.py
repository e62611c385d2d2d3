"""Performance cases of the TensorNet library: what its users have it do, from
one 32-atom molecule to a 96,000-atom water box, through the public Python
binding (paper_2402_17660_gb300.tnet).

A case is a dict of plain values:
  kind    "step"   neighbor search + energies (+ forces): one energy call of a
                   simulation, an optimiser or a data-set evaluation
          "train"  energies of a batch through the autograd function, then the
                   backward pass to positions and to every weight
          "md"     velocity-Verlet steps on the captured graph
          "pairs"  the neighbor search alone
  system  "molecule" / "batch" (atoms at 0.148 per cubic Angstrom in vacuum),
          "walk" (self-avoiding random walk in vacuum), "water" (rigid waters,
          periodic cube), "tilted" (rigid waters, triclinic cell)
  F, K, L, cutoff, precision (0 FP32, 1 BF16, 2 3xTF32), table: the model
"""
import math

import numpy as np
import torch

from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import EnergyFn, TensorNet, pack_weights, unpack_weights

DEV = "cuda"
MAX_Z = 100
ACCEL = 9.64853321e-3      # 1 eV/(A amu) in A/fs^2
WATER_SITE = 3.104         # lattice constant of liquid water, A per molecule
MOL_DENSITY = 32 / 6.0 ** 3


def _case(name=None, kind="step", system="water", size=10, keep=0, F=128, K=32, L=2, cutoff=5.0, precision=2, table=0,
          forces=True, steps=0):
    c = dict(kind=kind, system=system, size=size, keep=keep, F=F, K=K, L=L, cutoff=cutoff, precision=precision,
             table=table, forces=forces, steps=steps)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small molecule, the paper's smallest use: launches and latency
        _case("molecule32_fp32", system="molecule", size=32, precision=0),
        # a protein-like molecule of the paper's speed table at its 4.5 A cutoff, one layer
        _case("walk2489_l1", system="walk", size=2489, L=1, cutoff=4.5),
        # a data set evaluated in one call: 512 molecules of 8..96 atoms
        _case("batch512", system="batch", size=512),
        # the plain FP32 form on a periodic box
        _case("water3000_fp32", size=10, precision=0),
        # energies alone (screening, Monte Carlo) in a triclinic cell of ragged size
        _case("tilted3993_energy", system="tilted", size=11, forces=False),
        # a narrow model (64 channels, one layer) on a box of a ragged atom count
        _case("water12k_f64", size=16, keep=4001, F=64, K=16, L=1),
        # one training step on a mini-batch of molecules: gradients of every weight
        _case("train_batch64", kind="train", system="batch", size=64),
        # mixed precision on a box of 24,000 atoms
        _case("water24k_bf16", size=20, precision=1),
        # tabulated radial functions, the inference mode of production runs
        _case("water14k_table", size=17, table=2048),
        # molecular dynamics: steps with a 1 A skin on the captured graph
        _case("md_water3000", kind="md", size=10, steps=10),
        # the neighbor search of a large box at cutoff plus skin
        _case("pairs_water176k", kind="pairs", size=39, keep=58611, cutoff=6.0),
        # the largest box of the benchmark
        _case("water96k", size=32, keep=32000),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def water(atoms_lo, atoms_hi):
        mol = log(atoms_lo / 3, atoms_hi / 3)
        side = 4
        while side ** 3 < mol:
            side += 1
        return dict(system=rng.choice(["water", "water", "tilted"]), size=side, keep=mol)

    kind = rng.choice(["step"] * 6 + ["train", "md", "pairs"])
    if kind == "pairs":
        return _case(kind=kind, **water(300, 200000), cutoff=rng.choice([5.0, 6.0]))
    if kind == "md":
        w = water(600, 6000)
        return _case(kind=kind, system="water", size=max(w["size"], 5), keep=w["keep"], precision=rng.choice([1, 2, 2]),
                     steps=rng.choice([4, 5, 10]))
    if kind == "train":
        return _case(kind=kind, system="batch", size=log(2, 128), F=rng.choice([64, 128, 128]), L=rng.choice([1, 2]),
                     precision=rng.choice([0, 2, 2]))
    F = rng.choice([64, 128, 128, 128, 128, 256])
    L = rng.choice([0, 1, 2, 2, 2, 3])
    precision = rng.choice([0, 1, 2, 2])
    table = rng.choice([0, 0, 0, 0, 1024, 2048])
    top = {0: 9000, 1: 60000, 2: 60000}[precision] * 128 // F * 2 // max(L, 2)
    pick = rng.choice(["molecule", "batch", "walk", "water", "water", "water"])
    if pick == "water":
        where = water(300, top)
    elif pick == "molecule":
        where = dict(system=pick, size=log(2, 200))
    elif pick == "walk":
        where = dict(system=pick, size=log(20, 6000))
    else:
        where = dict(system=pick, size=log(2, min(512, top // 60)))
    return _case(kind=kind, **where, F=F, K=rng.choice([16, 32, 32]), L=L, cutoff=4.5 if pick == "walk" else 5.0,
                 precision=precision, table=table, forces=rng.random() < 0.8)


# ------------------------------------------------------------------ inputs ---
def _waters(case, seed):
    """Rigid waters on a jittered lattice, random orientations; a triclinic
    cell has the cube's volume."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["size"]
    a = WATER_SITE
    B = torch.eye(3, dtype=torch.float64, device=DEV) * (n * a)
    if case["system"] == "tilted":
        B[1, 0], B[2, 0], B[2, 1] = 0.3 * n * a, 0.2 * n * a, -0.25 * n * a
    k = torch.arange(n, device=DEV, dtype=torch.float64)
    frac = (torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3) + 0.5) / n
    if case["keep"] and case["keep"] < len(frac):
        frac = frac[torch.randperm(len(frac), generator=g, device=DEV)[:case["keep"]].sort().values]
    m = len(frac)
    c = frac @ B + (torch.rand(m, 3, generator=g, device=DEV, dtype=torch.float64) - 0.5) * 0.6
    q = torch.nn.functional.normalize(torch.randn(m, 4, generator=g, device=DEV, dtype=torch.float64), dim=1)
    w, v = q[:, :1, None], q[:, None, 1:]
    t = math.radians(104.52) / 2
    frame = 0.9572 * torch.tensor([[0, 0, 0], [math.sin(t), math.cos(t), 0], [-math.sin(t), math.cos(t), 0]],
                                  dtype=torch.float64, device=DEV)
    f = frame.expand(m, 3, 3)
    cr = 2 * torch.linalg.cross(v.expand(m, 3, 3), f)
    rot = f + w * cr + torch.linalg.cross(v.expand(m, 3, 3), cr)
    pos = (c[:, None] + rot).reshape(-1, 3).float()
    z = torch.tensor([8, 1, 1], dtype=torch.int32, device=DEV).repeat(m)
    return z, pos, None, B.float()[None].contiguous(), 1


def _inputs(case, seed):
    """z, pos, batch (None: one system), box (None: vacuum), number of systems"""
    if case["system"] in ("water", "tilted"):
        return _waters(case, seed)
    if case["system"] == "batch":
        counts = np.random.default_rng(case["size"]).integers(8, 97, case["size"])
        mols = [synth.random_cluster(int(n), seed=1000 * seed + m) for m, n in enumerate(counts)]
        s = synth.System("batch", np.concatenate([m.z for m in mols]), np.concatenate([m.pos for m in mols]),
                         np.repeat(np.arange(len(mols), dtype=np.int32), counts), None, len(mols))
    elif case["system"] == "walk":
        s = synth.random_walk_molecule(case["size"], seed=seed)
    else:
        s = synth.random_cluster(case["size"], seed=seed)
    to = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
    return to(s.z), to(s.pos), to(s.batch) if s.n_systems > 1 else None, None, s.n_systems


def _weights(case, seed):
    shape = synth.ModelShape(F=case["F"], K=case["K"], L=case["L"], max_z=MAX_Z, cutoff_upper=case["cutoff"])
    make = synth.md_weights if case["kind"] == "md" else synth.init_weights
    w = make(shape, seed)
    # an atom's mean energy: of one sign and above its fluctuation, as in a
    # trained potential (random weights alone give totals near zero)
    w["head2_b"] = np.full(1, -10.0, np.float32)
    return w


SKIN = 1.0


def _capacity(case, z, batch):
    """Directed pairs to allow for: the user's estimate from the density."""
    n = len(z)
    if case["system"] in ("water", "tilted"):
        r = case["cutoff"] + (SKIN if case["kind"] == "md" else 0.0)
        return int(n * (3 / WATER_SITE ** 3 * 4.18879 * r ** 3 * 1.15 + 8))
    if case["system"] == "batch" and batch is not None:
        c = torch.bincount(batch.long())
        return int((c * (c - 1)).sum()) + 64
    return min(n * (n - 1), 200 * n) + 64


def prepare(case, seed):
    z, pos, batch, box, S = _inputs(case, seed)
    W = _weights(case, seed)
    n = len(z)
    cap = _capacity(case, z, batch)
    if case["kind"] == "pairs":  # the search uses no model: the context with the smallest workspace serves
        W, model_of = _weights({**case, "F": 64, "K": 8, "L": 0}, seed), dict(F=64, K=8, L=0, radial_table=256)
    else:
        model_of = dict(F=case["F"], K=case["K"], L=case["L"], precision=case["precision"], radial_table=case["table"])
    model = TensorNet(W, max_z=MAX_Z, cutoff_upper=case["cutoff"], max_atoms=n, max_systems=S, max_pairs=cap,
                      device=DEV, **model_of)
    st = dict(case=case, model=model, z=z, pos=pos, batch=batch, box=box, S=S)
    if case["kind"] == "md":
        mass = torch.where(z == 8, 15.999, 1.008).float()
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        vel = torch.randn(n, 3, generator=g, device=DEV) * (8.617333262e-5 * 300 * ACCEL / mass).sqrt()[:, None]
        st.update(inv_mass=1 / mass, pos0=pos.clone(), vel0=vel, vel=vel.clone(),
                  e=[torch.zeros(case["steps"], dtype=torch.float64, device=DEV) for _ in range(2)])
        return st
    st["nl"] = model.neighbors(pos, batch, box, S)  # the list's buffers are kept from call to call
    st["nl"].col.zero_()
    if case["kind"] == "train":
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        st["target"] = torch.randn(S, generator=g, device=DEV, dtype=torch.float64)
        st["w"] = model.weights.clone().requires_grad_()
    return st


def run(st):
    case, m = st["case"], st["model"]
    if case["kind"] == "md":
        st["pos"].copy_(st["pos0"])
        st["vel"].copy_(st["vel0"])
        ek, ep = m.md(st["z"], st["inv_mass"], st["pos"], st["vel"], st["box"], 0.5, SKIN, 5, case["steps"], *st["e"])
        return [st["pos"], st["vel"], ek.float(), ep.float()]
    nl = m.neighbors(st["pos"], st["batch"], st["box"], st["S"], out=st["nl"])
    if case["kind"] == "pairs":
        return [nl.row_ptr, nl.col, nl.n_pairs]
    if case["kind"] == "train":
        pos = st["pos"].detach().requires_grad_()
        st["w"].grad = None
        E = EnergyFn.apply(pos, st["w"], m, st["z"], nl, st["batch"], st["box"], st["S"])
        # d/dE of a mean squared error; FP32 like the model's other outputs
        E.backward((E.detach() - st["target"]) * (2.0 / st["S"]))
        return [E.detach().float(), pos.grad, st["w"].grad]
    E, Fo, _ = m.energy_forces(st["z"], st["pos"], nl, st["batch"], st["box"], st["S"], forces=case["forces"])
    # the energies' FP64 is the type of their sum over atoms, whose terms are
    # FP32: handed on in the terms' type, like the forces
    return [E.float(), Fo] if case["forces"] else [E.float()]


# -------------------------------------------------------------------- work ---
def _sizes(case):
    """Atoms and directed pairs of a case, from its densities."""
    if case["system"] in ("water", "tilted"):
        sites = case["size"] ** 3
        n = 3 * (case["keep"] if case["keep"] and case["keep"] < sites else sites)
        return n, n * (n / (sites * WATER_SITE ** 3)) * 4.18879 * case["cutoff"] ** 3
    if case["system"] == "batch":
        return 52 * case["size"], 52 * case["size"] * 33.0
    n = case["size"]
    return n, n * min(n - 1, 33.0)


def work(case):
    n, edges = _sizes(case)
    if case["kind"] == "pairs":
        return {"bytes": 12.0 * n + 4.0 * n + 4.0 * edges, "flops": 10.0 * edges}
    F, K, L = case["F"], case["K"], case["L"]
    u = edges / 2
    radial = 2 * 3 * F * K + L * 2 * (K * F + 2 * F * F + 6 * F * F)
    per_edge = 2 * 12 * F + L * 2 * 9 * F
    atom = (1 + 2 * L) * 2 * 9 * F * F + 2 * F * F * 11.5
    if case["table"]:
        radial = (1 + L) * 6 * 3 * F
    one = u * radial + edges * per_edge + n * atom
    passes = 3 if case["kind"] == "train" else 2 if case["forces"] or case["kind"] == "md" else 1
    weights = 4.0 * (MAX_Z * F + 2 * F * F + 3 * F * K + 8 * F * F + 3 * F * F + L * (K * F + 14 * F * F) + 3.5 * F * F)
    bytes_ = 16.0 * n + weights * (2 if case["kind"] == "train" else 1) + 12.0 * n
    times = case["steps"] + 1 if case["kind"] == "md" else 1
    return {"bytes": bytes_ * times, "flops": one * passes * times}


# ------------------------------------------------------------------- exact ---
def _nearest(r, box):
    if box is not None:
        for k in (2, 1, 0):
            r = r - torch.round(r[:, k] / box[k, k])[:, None] * box[k]
    return r


def _pairs(pos, batch, box, rc):
    """Undirected pairs (i < j) of one system within rc."""
    n, out = len(pos), []
    step = max(1, min(n, 40_000_000 // n))
    j = torch.arange(n, device=DEV)
    for a in range(0, n, step):
        i = torch.arange(a, min(n, a + step), device=DEV)
        r = _nearest((pos[i][:, None] - pos[None]).reshape(-1, 3), box)
        ok = ((r * r).sum(-1) < rc * rc).view(len(i), n) & (i[:, None] < j[None])
        if batch is not None:
            ok &= batch[i][:, None] == batch[None]
        p = ok.nonzero()
        out.append(torch.stack([p[:, 0] + a, p[:, 1]]))
    return torch.cat(out, 1)


def _split(X):
    I = X.diagonal(dim1=-2, dim2=-1).mean(-1)[..., None, None] * torch.eye(3, dtype=X.dtype, device=X.device)
    T = X.transpose(-1, -2)
    return I, (X - T) / 2, (X + T) / 2 - I


def _sq(X):
    return X.square().sum((-1, -2))


def _energy64(case, p, z, pos, batch, box, S):
    """Per-system TensorNet energies in 64 bits (differentiable)."""
    from torch.utils.checkpoint import checkpoint
    F, K, L, rc = case["F"], case["K"], case["L"], case["cutoff"]
    act, norm = torch.nn.functional.silu, torch.nn.functional.layer_norm
    n = len(z)
    i, j = _pairs(pos.detach(), batch, box, rc)
    mu0 = math.exp(-rc)
    mu = torch.linspace(mu0, 1, K, dtype=torch.float64, device=DEV)
    beta = (2 / K * (1 - mu0)) ** -2
    eye = torch.eye(3, dtype=torch.float64, device=DEV)

    def geometry(pos, a, b):
        r = _nearest(pos[a] - pos[b], box)
        d = r.norm(dim=1)
        phi = 0.5 * (torch.cos(math.pi * d / rc) + 1)
        e = phi[:, None] * torch.exp(-beta * (torch.exp(-5 / rc * d)[:, None] - mu) ** 2)
        return r / d[:, None], phi, e

    def embed(pos, a, b, emb, w, wb, dw, db):
        u, phi, e = geometry(pos, a, b)
        f = torch.einsum("ek,pck->epc", e, dw) + db
        o = torch.zeros_like(u[:, 0])
        A = torch.stack([o, -u[:, 2], u[:, 1], u[:, 2], o, -u[:, 0], -u[:, 1], u[:, 0], o], 1).view(-1, 1, 3, 3)
        Sm = (u[:, :, None] * u[:, None] - eye / 3)[:, None]
        even = f[:, 0, :, None, None] * eye + f[:, 2, :, None, None] * Sm
        odd = f[:, 1, :, None, None] * A
        zab = torch.cat([emb[z[a]], emb[z[b]]], 1) @ w.T + wb
        zba = torch.cat([emb[z[b]], emb[z[a]]], 1) @ w.T + wb
        return (phi[:, None] * zab)[..., None, None] * (even + odd), (phi[:, None] * zba)[..., None, None] * (even - odd)

    def message(pos, a, b, Y, w1, b1, w2, b2, w3, b3):
        _, phi, e = geometry(pos, a, b)
        g = phi[:, None] * act(act(act(e @ w1.T + b1) @ w2.T + b2) @ w3.T + b3)
        g = g.view(len(a), F, 3)[..., None, None]
        out = []
        for q in (b, a):
            I, A, Sm = _split(Y[q])
            out.append(g[:, :, 0] * I + g[:, :, 1] * A + g[:, :, 2] * Sm)
        return out

    def gathered(fn, *args):
        X = torch.zeros(n, F, 3, 3, dtype=torch.float64, device=DEV)
        for a, b in zip(i.split(32768), j.split(32768)):
            to_a, to_b = checkpoint(fn, pos, a, b, *args, use_reentrant=False)
            X = X.index_add(0, a, to_a).index_add(0, b, to_b)
        return X

    def mix(W, parts):
        return sum(torch.einsum("cd,ndab->ncab", W[q], parts[q]) for q in range(3))

    X = gathered(embed, p["emb"], p["emb2_w"], p["emb2_b"], p["dproj_w"], p["dproj_b"])
    h = norm(_sq(X), (F,), p["emb_ln_g"], p["emb_ln_b"])
    s = act(act(h @ p["emb_mlp1_w"].T + p["emb_mlp1_b"]) @ p["emb_mlp2_w"].T + p["emb_mlp2_b"]).view(n, F, 3)
    parts = _split(X)
    X = sum(s[:, :, q, None, None] * torch.einsum("cd,ndab->ncab", p["emb_mix_w"][q], parts[q]) for q in range(3))
    for l in range(L):
        X = X / (_sq(X) + 1)[..., None, None]
        Y = mix(p[f"l{l}_mix1_w"], _split(X))
        M = gathered(message, Y, *(p[f"l{l}_mlp{k}_{t}"] for k in (1, 2, 3) for t in "wb"))
        T = Y @ M + M @ Y
        D = mix(p[f"l{l}_mix2_w"], _split(T / (_sq(T) + 1)[..., None, None]))
        X = X + D + D @ D
    h = norm(torch.cat([_sq(q) for q in _split(X)], 1), (3 * F,), p["out_ln_g"], p["out_ln_b"])
    h = act(act(h @ p["out_w"].T + p["out_b"]) @ p["head1_w"].T + p["head1_b"])
    e = (h @ p["head2_w"].T)[:, 0] + p["head2_b"]
    at = torch.zeros(n, dtype=torch.long, device=DEV) if batch is None else batch.long()
    return torch.zeros(S, dtype=torch.float64, device=DEV).index_add(0, at, e)


def exact(case, seed):
    n, _ = _sizes(case)
    if case["kind"] == "pairs" or n * (case["steps"] + 1) * case["F"] * max(case["L"], 1) > 64000 * 256:
        return None
    z, pos, batch, box, S = _inputs(case, seed)
    z = z.long()
    shape = (case["F"], case["K"], case["L"], MAX_Z)
    blob = torch.from_numpy(pack_weights(_weights(case, seed), *shape)).to(DEV, torch.float64).requires_grad_()
    p, at = {}, 0
    for name, w in unpack_weights(np.zeros(blob.numel(), np.int8), *shape).items():  # names and shapes of the blob
        p[name] = blob[at:at + w.size].view(w.shape)
        at += w.size
    box = None if box is None else box[0].double()

    def value(x, wants):
        x = x.detach().requires_grad_()
        E = _energy64(case, p, z, x, batch, box, S)
        return E, x, wants(E, x)

    def force(E, x):
        return -torch.autograd.grad(E.sum(), x)[0]

    pos = pos.double()
    if case["kind"] == "md":
        inv = 1 / torch.where(z == 8, 15.999, 1.008).float().double()[:, None]
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        mass = torch.where(z == 8, 15.999, 1.008).float()
        v = (torch.randn(n, 3, generator=g, device=DEV) * (8.617333262e-5 * 300 * ACCEL / mass).sqrt()[:, None]).double()
        F = value(pos, force)[2]
        ek, ep = [], []
        for _ in range(case["steps"]):
            v = v + 0.25 * ACCEL * F * inv
            pos = pos + 0.5 * v
            E, _, F = value(pos, force)
            v = v + 0.25 * ACCEL * F * inv
            ek.append((0.5 * v * v / inv).sum() / ACCEL)
            ep.append(E.detach()[0])
        return [pos, v, torch.stack(ek), torch.stack(ep)]
    if case["kind"] == "train":
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        target = torch.randn(S, generator=g, device=DEV, dtype=torch.float64)
        E, _, (gx, gw) = value(pos, lambda E, x: torch.autograd.grad(
            (E * (E.detach() - target)).sum() * (2.0 / S), (x, blob)))
        return [E.detach(), gx, gw]
    if not case["forces"]:
        with torch.no_grad():
            return [_energy64(case, p, z, pos, batch, box, S)]
    E, _, F = value(pos, force)
    return [E.detach(), F]
