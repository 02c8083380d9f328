"""Workloads of the VESIS library, each through the calls a program makes.

A case is a dict of plain values; `kind` says which part of the library it
exercises:

  fields  energy density and Coulomb field of a solute on its grid
  forces  gradient of the free energy of every atom (fields included)
  sweep   interface relaxation by flips at fixed atoms
  relax   outer iterations of the full relaxation of one small solute
  batch   the same for several small solutes at once
  pmf     one point of a two-atom potential of mean force
  guess   the learned initialiser's labels of a whole grid
  train   training steps of the learned initialiser, weights read back

Inputs are seeded synthetic solutes (random-walk globules up to 2,000 atoms,
jittered close-packed balls of the same density above) with the parameter
distributions of the repository's workloads.  Energy densities that a case
takes as its input are made here with torch, pair by pair within a cutoff,
in integer sums that come out the same on every run.
"""
import math

import numpy as np
import torch

from paper_2208_05524_gb300 import pmf, synth, vesis

RHO, GAMMA_T, R_MIN = 0.0333, 298.0, 0.2
EPS_M, EPS_W = 1.0, 80.0
# e^2 / (4 pi eps0 kB T) in Angstrom (CODATA 2018)
L_B = 1.602176634e-19 ** 2 / (4.0 * math.pi * 8.8541878128e-12 * 1.380649e-23 * GAMMA_T) * 1e10
CFA = L_B / (8.0 * math.pi) * (1.0 / EPS_W - 1.0 / EPS_M)
DENSITY = 0.05                       # atoms per cubic Angstrom of a globule
SCALE = 0.01                         # kBT / A^3 inside the features' asinh
CHANNELS = (32, 64, 128, 128)
# (out, in, kernel edge) of the network's layers in the order of its
# parameter vector
LAYERS = ((32, 3, 3), (64, 32, 3), (128, 64, 3), (128, 128, 3), (64, 256, 3), (32, 128, 3),
          (32, 64, 3), (1, 32, 1))


def listed():
    return [
        # the smallest call: fields of one charged atom on the 64^3 box that
        # the closed-form sphere is checked on; launches and latency
        dict(name="fields_ion_64", kind="fields", atoms=1, nx=64, ny=64, nz=64, h=0.25),
        # the protein-like solute's fields, evaluated at every trial step
        dict(name="fields_protein_256", kind="fields", atoms=2000, nx=256, ny=256, nz=256, h=0.4),
        # gradient of a host-guest sized solute at that set's spacing on a
        # box cut to the solute (ragged, not a multiple of 8)
        dict(name="forces_host_ragged", kind="forces", atoms=1500, nx=203, ny=190, nz=197, h=0.3),
        # fields and gradient of the 20,000-atom two-domain complex
        dict(name="forces_complex_384", kind="forces", atoms=20000, nx=384, ny=384, nz=384, h=0.4),
        # interface relaxation from the tight start: the protein-like solute
        dict(name="sweep_protein_256", kind="sweep", atoms=2000, nx=256, ny=256, nz=256, h=0.4,
             surface="gauss"),
        # the same for the complex
        dict(name="sweep_complex_384", kind="sweep", atoms=20000, nx=384, ny=384, nz=384, h=0.4,
             surface="gauss"),
        # the paper's sin^2 surface kernel on a box cut to its solute
        dict(name="sweep_sin2_ragged", kind="sweep", atoms=500, nx=150, ny=141, nz=133, h=0.4,
             surface="sin2"),
        # full relaxation of a small solute, ten outer iterations of it
        dict(name="relax_small_112", kind="relax", atoms=276, nx=112, ny=112, nz=112, h=0.4,
             outer=10),
        # the many-solute service: eight small solutes at once
        dict(name="batch_small_8", kind="batch", count=8, least=60, most=400, h=0.4, outer=4),
        # one separation of the two-atom curve
        dict(name="pmf_two_atoms_128", kind="pmf", d=7.5, opposite=True, n=128, h=0.2),
        # the learned start of a protein-like solute's whole grid
        dict(name="guess_256", kind="guess", nx=256, ny=256, nz=256, h=0.4, atoms=2000),
        # training on 64^3 crops, one crop a step
        dict(name="train_64", kind="train", crop=64, steps=4, h=0.4, atoms=300),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(atoms, h, rng, margin=8.0):
    """Cells per axis of a box that holds the solute and a margin, the three
    axes drawn apart (ragged) or as one multiple of 16."""
    need = 2.0 * (_radius(atoms) + 4.0 + margin) / h
    if atoms > 2000:
        need = 2.0 * (_half_extent(atoms) + margin) / h
    if rng.random() < 0.5:
        n = 16 * int(math.ceil(need / 16.0))
        return n, n, n
    return tuple(int(math.ceil(need)) + rng.randrange(0, 24) for _ in range(3))


def draw(rng):
    kind = rng.choice(["fields", "fields", "forces", "forces", "sweep", "sweep", "relax", "batch",
                       "pmf", "guess", "train"])
    if kind in ("fields", "forces", "sweep"):
        atoms = int(round(_log(rng, 1 if kind != "forces" else 20, 20000)))
        h = 0.4 if atoms > 4000 else round(rng.uniform(0.3, 0.5), 3)
        nx, ny, nz = _side(atoms, h, rng)
        case = dict(kind=kind, atoms=atoms, nx=min(nx, 384), ny=min(ny, 384), nz=min(nz, 384), h=h)
        if kind == "sweep":
            case["surface"] = rng.choice(["gauss", "gauss", "sin2"])
        return case
    if kind == "relax":
        atoms = int(round(_log(rng, 60, 400)))
        nx, ny, nz = _side(atoms, 0.4, rng)
        return dict(kind=kind, atoms=atoms, nx=nx, ny=ny, nz=nz, h=0.4, outer=rng.randint(3, 12))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 12), least=60, most=rng.randint(120, 400),
                    h=0.4, outer=rng.randint(2, 5))
    if kind == "pmf":
        return dict(kind=kind, d=round(rng.uniform(4.0, 12.0), 2), opposite=rng.random() < 0.5,
                    n=rng.choice([96, 111, 128, 130]), h=round(rng.uniform(0.2, 0.25), 3))
    if kind == "guess":
        n = [8 * int(round(_log(rng, 64, 256) / 8.0)) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], h=round(rng.uniform(0.38, 0.42), 3),
                    atoms=300)
    return dict(kind=kind, crop=rng.choice([32, 48, 64, 80]), steps=rng.randint(2, 5),
                h=round(rng.uniform(0.38, 0.42), 3), atoms=300)


# ------------------------------------------------------------------ solutes
def _radius(atoms):
    return max((3.0 * atoms / (4.0 * math.pi * DENSITY)) ** (1.0 / 3.0), 2.0 * 3.8)


def _half_extent(atoms):
    """Half-width of the two packed balls along the body diagonal."""
    r = _radius(atoms // 2)
    return (r + 3.0) / math.sqrt(3.0) + r + 1.0


def _ball(n, rng, centre):
    """n beads at globule density: a jittered face-centred cubic lattice cut
    to a ball, and the bonds between consecutive beads that touch."""
    a = (4.0 / DENSITY) ** (1.0 / 3.0)
    m = int(math.ceil(_radius(n) / a)) + 2
    k = np.arange(-m, m + 1)
    cell = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 1, 3)
    base = np.array([[0, 0, 0], [0, 0.5, 0.5], [0.5, 0, 0.5], [0.5, 0.5, 0]])
    p = ((cell + base).reshape(-1, 3) + rng.uniform(0.0, 1.0, 3)) * a
    keep = np.sort(np.argsort(np.linalg.norm(p, axis=1), kind="stable")[:n])
    p = p[keep]
    d = np.linalg.norm(np.diff(p, axis=0), axis=1)
    i = np.nonzero(d < 1.1 * a / math.sqrt(2.0))[0]
    p = p + rng.uniform(-0.3, 0.3, p.shape) + centre
    return p, np.stack([i, i + 1], 1).astype(np.int32)


def _solute(case, seed, atoms=None):
    """One solute of the case in the form vesis.System takes."""
    n = int(case["atoms"] if atoms is None else atoms)
    rng = np.random.default_rng([int(seed), n])
    shape = [int(case[k]) for k in ("nx", "ny", "nz")]
    h = float(case["h"])
    if n == 1:
        s = synth.single_ion(n=64, h=h, q=float(rng.choice([-1.0, 1.0])),
                             center=tuple(rng.uniform(-0.5, 0.5, 3)))
        s["sigma_sw"] = rng.uniform(3.0, 4.0, 1)
    elif n <= 2000:
        s = synth.protein_like(n_atoms=n, n=16, h=h, seed=int(rng.integers(1 << 31)))
    else:
        off = (_radius(n // 2) + 3.0) / math.sqrt(3.0)
        a, ba = _ball(n - n // 2, rng, -off)
        b, bb = _ball(n // 2, rng, off)
        xyz = np.concatenate([a, b])
        bonds = np.concatenate([ba, bb + len(a)])
        r0 = np.linalg.norm(xyz[bonds[:, 0]] - xyz[bonds[:, 1]], axis=1)
        kbt = synth.kbt_kj_per_mol(GAMMA_T)
        sigma, eps = rng.uniform(3.0, 4.0, n), rng.uniform(0.1, 0.9, n) / kbt
        q = rng.normal(0.0, 0.35, n)
        q += (-3.0 - q.sum()) / n
        s = dict(xyz=xyz, sigma_sw=sigma, eps_sw=eps, q=q, sigma_ss=sigma, eps_ss=eps,
                 bonds=bonds, bond_k=np.full(len(bonds), 800.0), bond_r0=r0)
    s = dict(s, n=np.array(shape), h=h, origin=np.array([-0.5 * m * h for m in shape]))
    return s


# ----------------------------------------------------- inputs made with torch
def _patches(s, reach):
    """For groups of atoms: the linear indices of the grid cells within
    `reach` of each atom and d = cell centre - atom, on the GPU."""
    dev = torch.device("cuda", torch.cuda.current_device())
    nx, ny, nz = (int(v) for v in s["n"])
    h = float(s["h"])
    xyz = torch.as_tensor(np.asarray(s["xyz"]), dtype=torch.float64, device=dev)
    org = torch.as_tensor(np.asarray(s["origin"]), dtype=torch.float64, device=dev)
    m = int(math.ceil(reach / h))
    k = torch.arange(-m, m + 1, device=dev)
    off = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    off = off[(off.double().norm(dim=1) - 1.0) * h <= reach]
    lim = torch.tensor([nx, ny, nz], device=dev)
    per = max(1, (1 << 24) // len(off))
    for a in range(0, len(xyz), per):
        p = xyz[a:a + per]
        c = torch.floor((p - org) / h).long()[:, None, :] + off
        ok = ((c >= 0) & (c < lim)).all(-1)
        d = (org + (c.double() + 0.5) * h) - p[:, None, :]
        ok &= d.square().sum(-1) < reach * reach
        idx = (c[..., 0] * ny + c[..., 1]) * nz + c[..., 2]
        yield a, ok, idx, d


def _tight(s):
    """Labels of the tight start: 1 within sigma of an atom."""
    dev = torch.device("cuda", torch.cuda.current_device())
    chi = torch.zeros(int(np.prod(s["n"])), dtype=torch.uint8, device=dev)
    sig = torch.as_tensor(np.asarray(s["sigma_sw"]), device=dev)
    for a, ok, idx, d in _patches(s, float(np.max(s["sigma_sw"]))):
        r = d.square().sum(-1).sqrt()
        ok &= r < sig[a:a + len(r), None]
        chi[idx[ok]] = 1
    return chi


def _densities(s, cutoff=8.0):
    """Energy density parts (LJ, CFA) and field of the atoms within the
    cutoff of each cell, as float32 planes, summed in integers."""
    dev = torch.device("cuda", torch.cuda.current_device())
    G = int(np.prod(s["n"]))
    one = float(1 << 32)
    acc = [torch.zeros(G, dtype=torch.int64, device=dev) for _ in range(4)]
    sig, eps, q = (torch.as_tensor(np.asarray(s[k]), device=dev)
                   for k in ("sigma_sw", "eps_sw", "q"))
    for a, ok, idx, d in _patches(s, cutoff):
        m = len(ok)
        r2 = d.square().sum(-1).clamp_(min=R_MIN * R_MIN)
        s6 = (sig[a:a + m, None].square() / r2) ** 3
        lj = (4.0 * RHO * eps[a:a + m, None] * (s6 * s6 - s6)).clamp_(max=1e4)
        qr3 = q[a:a + m, None] * r2 ** -1.5
        idx = idx[ok]
        acc[0].index_add_(0, idx, (lj[ok] * one).round_().long())
        for c in range(3):
            acc[1 + c].index_add_(0, idx, ((qr3 * d[..., c])[ok] * one).round_().long())
    E = torch.stack([v.double() / one for v in acc[1:]])
    return (acc[0].double() / one).float(), (CFA * E.square().sum(0)).float(), E.float().reshape(-1)


def _features(s):
    lj, cfa, _ = _densities(s)
    return torch.stack([torch.asinh(lj / SCALE), torch.asinh(cfa / SCALE), _tight(s).float()])


# ------------------------------------------------------------------- a pass
def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda", torch.cuda.current_device())
    st = dict(case=case)
    if kind in ("fields", "forces"):
        s = _solute(case, seed)
        st["S"] = vesis.System(s)
        G = st["S"].G
        if kind == "fields":
            st["U"] = torch.empty(G, dtype=torch.float32, device=dev)
            st["E"] = torch.empty(3 * G, dtype=torch.float32, device=dev)
        else:
            st["chi"] = _tight(s)
    elif kind == "sweep":
        s = _solute(case, seed)
        st["S"] = vesis.System(s, kernel=case["surface"])
        lj, cfa, st["E"] = _densities(s)
        st["U"] = lj + cfa
        st["chi0"] = _tight(s)
        st["chi"] = st["chi0"].clone()
    elif kind == "relax":
        s = _solute(case, seed)
        st["S"] = vesis.System(s)
        st["xyz"] = s["xyz"].copy()
        st["chi0"] = _tight(s)
        st["chi"] = st["chi0"].clone()
    elif kind == "batch":
        ss = []
        for i in range(case["count"]):
            t = (i + 0.5) / case["count"]
            atoms = int(round(case["least"] * (case["most"] / case["least"]) ** t))
            n = 16 * int(math.ceil(2.0 * (_radius(atoms) + 12.0) / (16.0 * case["h"])))
            ss.append(_solute(dict(case, nx=n, ny=n, nz=n), seed * 100 + i, atoms))
        st["S"] = [vesis.System(s) for s in ss]
        st["xyz"] = [s["xyz"].copy() for s in ss]
        st["chi0"] = [_tight(s) for s in ss]
        st["chi"] = [c.clone() for c in st["chi0"]]
    elif kind == "pmf":
        s = _pair(case, seed)
        st["S"] = vesis.System(s)
        st["xyz"] = s["xyz"].copy()
        G = st["S"].G
        st["U"] = torch.empty(G, dtype=torch.float32, device=dev)
        st["E"] = torch.empty(3 * G, dtype=torch.float32, device=dev)
        st["chi"] = torch.empty(G, dtype=torch.uint8, device=dev)
    elif kind == "guess":
        s = _solute(case, seed)
        st["shape"] = tuple(int(v) for v in s["n"])
        st["x"] = _features(s).reshape(-1).contiguous()
        st["logits"] = torch.empty(int(np.prod(s["n"])), dtype=torch.float32, device=dev)
        st["chi"] = torch.empty(int(np.prod(s["n"])), dtype=torch.uint8, device=dev)
        st["net"] = vesis.Net(3)
        st["net"].set_params(_theta(seed))
    elif kind == "train":
        st["net"] = vesis.Net(3)
        st["net"].set_params(_theta(seed))
        st["x"], st["y"] = _crops(case, seed)
    else:
        raise ValueError(kind)
    return st


def _theta(seed):
    """He-normal weights, exact in bfloat16, and zero biases."""
    rng = np.random.default_rng(int(seed))
    parts = []
    for co, ci, k in LAYERS:
        w = rng.normal(0.0, math.sqrt(2.0 / (ci * k ** 3)), co * ci * k ** 3).astype(np.float32)
        parts += [torch.from_numpy(w).bfloat16().float().numpy(), np.zeros(co, np.float32)]
    return np.concatenate(parts)


def _pair(case, seed):
    rng = np.random.default_rng(int(seed))
    q = (1.0, -1.0) if case["opposite"] else (1.0, 1.0)
    s = synth.two_atom(case["d"], q, n=case["n"], h=case["h"], sigma=float(rng.uniform(3.4, 3.6)))
    s["eps_sw"] = s["eps_sw"] * rng.uniform(0.9, 1.1)
    return s


def _crops(case, seed):
    c = int(case["crop"])
    xs, ys = [], []
    for i in range(case["steps"]):
        s = _solute(dict(case, nx=c, ny=c, nz=c), seed * 100 + i)
        keep = (np.abs(s["xyz"]) < 0.5 * c * s["h"]).all(1)
        s = dict(s, **{k: np.asarray(s[k])[keep] for k in ("xyz", "sigma_sw", "eps_sw", "q")})
        x = _features(s)
        xs.append(x.reshape(-1).contiguous())
        # a smoother solute than the tight labels, as the sweep leaves it
        soft = torch.nn.functional.avg_pool3d(x[2].view(1, 1, c, c, c), 5, 1, 2)
        ys.append((soft.reshape(-1) > 0.4).to(torch.uint8).contiguous())
    return xs, ys


def run(st):
    case = st["case"]
    kind = case["kind"]
    S = st.get("S")
    if kind == "fields":
        S.energy_field(st["U"], st["E"])
        return dict(U=st["U"], E=st["E"])
    if kind == "forces":
        return dict(grad=S.atom_forces(st["chi"]))
    if kind == "sweep":
        st["chi"].copy_(st["chi0"])
        r = S.blsm_relax(st["chi"], st["U"], st["E"])
        return dict(chi=st["chi"], rounds=r["rounds"], flips=r["flips"], dE_sum=r["dE_sum"],
                    terms=r["terms"])
    if kind == "relax":
        st["chi"].copy_(st["chi0"])
        r = S.relax(st["chi"], st["xyz"], max_outer=case["outer"])
        return dict(chi=st["chi"], **_relaxed(r))
    if kind == "batch":
        for c, c0 in zip(st["chi"], st["chi0"]):
            c.copy_(c0)
        rs = vesis.relax_batch(S, st["chi"], st["xyz"], max_outer=case["outer"])
        # as one array each: a batch may hold many systems
        return dict(chi=torch.cat(st["chi"]), xyz=np.concatenate([r["xyz"] for r in rs]),
                    G=np.array([r["G"] for r in rs]),
                    terms=np.array([[r["terms"][t] for t in vesis.TERMS] for r in rs]),
                    counts=np.array([[r["flips"], r["flip_rounds"], r["gd_trials"]] for r in rs]))
    if kind == "pmf":
        p = pmf.relaxed_parts(S, st["chi"], st["U"], st["E"], st["xyz"], "tight")
        return dict(chi=st["chi"], **p)
    if kind == "guess":
        st["net"].forward(st["x"], st["shape"], logits=st["logits"], chi=st["chi"])
        return dict(logits=st["logits"], chi=st["chi"])
    net, c = st["net"], (case["crop"],) * 3
    losses = []
    for x, y in zip(st["x"], st["y"]):
        losses.append(net.loss_grad(x, y, c))
        net.adam_step(lr=1e-3)
    return dict(losses=np.array(losses), theta=net.get_params())


def _relaxed(r):
    return dict(xyz=r["xyz"], G=r["G"], terms=r["terms"], M=r["M"], max_grad=r["max_grad"],
                flips=r["flips"], flip_rounds=r["flip_rounds"], gd_trials=r["gd_trials"])


# --------------------------------------------------------------------- work
def _conv_flops(nx, ny, nz):
    """2 x 27 x Cin x Cout per cell of every convolution of the network."""
    v = float(nx) * ny * nz
    c = CHANNELS
    per = [(3 * c[0], 1), (c[0] * c[1], 8), (c[1] * c[2], 64), (c[2] * c[3], 512),
           ((c[2] + c[3]) * 64, 64), ((64 + 64) * 32, 8), ((32 + 32) * 32, 1)]
    return sum(54.0 * m * v / d for m, d in per) + 64.0 * v


def work(case):
    """Each input read once, each output written once; operations of the
    sums as they are defined (every atom with every cell)."""
    k = case["kind"]
    if k == "train":
        v = float(case["crop"]) ** 3
        return dict(bytes=case["steps"] * 13.0 * v + 4.0 * 1.33e6,
                    flops=case["steps"] * 3.0 * _conv_flops(*(case["crop"],) * 3))
    if k == "pmf":
        G, N = float(case["n"]) ** 3, 2.0
        return dict(bytes=17.0 * G, flops=22.0 * G * N)
    if k == "batch":
        b = f = 0.0
        for i in range(case["count"]):
            t = (i + 0.5) / case["count"]
            N = case["least"] * (case["most"] / case["least"]) ** t
            G = (2.0 * (_radius(N) + 12.0) / case["h"]) ** 3
            b += 2.0 * G
            f += (22.0 * (case["outer"] + 1) + 36.0 * case["outer"]) * G * N
        return dict(bytes=b, flops=f)
    G = float(case["nx"]) * case["ny"] * case["nz"]
    N = float(case["atoms"])
    if k == "fields":
        return dict(bytes=16.0 * G + 48.0 * N, flops=22.0 * G * N)
    if k == "forces":
        return dict(bytes=1.0 * G + 72.0 * N, flops=(22.0 + 36.0) * G * N)
    if k == "sweep":
        return dict(bytes=18.0 * G, flops=54.0 * G)
    if k == "relax":
        return dict(bytes=2.0 * G + 96.0 * N,
                    flops=(22.0 * (case["outer"] + 1) + 36.0 * case["outer"]) * G * N)
    return dict(bytes=17.0 * G, flops=_conv_flops(case["nx"], case["ny"], case["nz"]))


# -------------------------------------------------------------------- exact
def _cells64(s):
    dev = torch.device("cuda", torch.cuda.current_device())
    ax = [torch.as_tensor(float(o) + (np.arange(int(n)) + 0.5) * float(s["h"]), device=dev)
          for o, n in zip(s["origin"], s["n"])]
    return torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)


def _atoms64(s):
    dev = torch.device("cuda", torch.cuda.current_device())
    t = {k: torch.as_tensor(np.asarray(s[k]), dtype=torch.float64, device=dev)
         for k in ("xyz", "sigma_sw", "eps_sw", "q", "sigma_ss", "eps_ss", "bond_k", "bond_r0")}
    s6 = t["sigma_sw"] ** 6
    t["A"], t["B"] = 4.0 * t["eps_sw"] * s6 * s6, 4.0 * t["eps_sw"] * s6
    return t


def _field64(pts, t):
    """U and E at points, in 64 bits."""
    U = torch.empty(len(pts), dtype=torch.float64, device=pts.device)
    E = torch.empty((len(pts), 3), dtype=torch.float64, device=pts.device)
    per = max(1, (1 << 25) // len(t["q"]))
    for a in range(0, len(pts), per):
        d = [pts[a:a + per, None, c] - t["xyz"][None, :, c] for c in range(3)]
        r2 = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).clamp_(min=R_MIN * R_MIN)
        i2 = r2.reciprocal_()
        i6 = i2 * i2 * i2
        U[a:a + per] = RHO * torch.mv(i6 * i6, t["A"]) - RHO * torch.mv(i6, t["B"])
        w = i2 * i2.sqrt() * t["q"]
        for c in range(3):
            E[a:a + per, c] = (w * d[c]).sum(1)
    return U + CFA * E.square().sum(1), E


def _far64(s):
    """Quadrature of the space outside the box: six face pyramids about its
    centre, 16 x 16 Gauss points on a face and 8 along the rays."""
    xu, wu = np.polynomial.legendre.leggauss(16)
    xt, wt = np.polynomial.legendre.leggauss(8)
    L = 0.5 * np.asarray(s["n"], np.float64) * float(s["h"])
    c = np.asarray(s["origin"]) + L
    pts, w = [], []
    for axis in range(3):
        o = [d for d in range(3) if d != axis]
        for sg in (-1.0, 1.0):
            u, v, t = np.meshgrid(xu, xu, 0.5 * (xt + 1.0), indexing="ij")
            f = np.zeros(u.shape + (3,))
            f[..., axis], f[..., o[0]], f[..., o[1]] = sg * L[axis], u * L[o[0]], v * L[o[1]]
            ww = wu[:, None, None] * wu[None, :, None] * 0.5 * wt * L.prod() / t ** 4
            pts.append((f / t[..., None] + c).reshape(-1, 3))
            w.append(ww.reshape(-1))
    dev = torch.device("cuda", torch.cuda.current_device())
    return (torch.as_tensor(np.concatenate(pts), device=dev),
            torch.as_tensor(np.concatenate(w), device=dev))


def _solvation_grad64(pts, wts, E, t):
    """sum over points of w d/dr_n of the energy density, in 64 bits."""
    g = torch.zeros_like(t["xyz"])
    per = max(1, (1 << 24) // len(t["q"]))
    for a in range(0, len(pts), per):
        d = pts[a:a + per, None, :] - t["xyz"]
        r2 = d.square().sum(-1)
        free = r2 >= R_MIN * R_MIN
        i2 = r2.clamp(min=R_MIN * R_MIN).reciprocal_()
        i3 = i2 * i2.sqrt()
        Ep, w = E[a:a + per], wts[a:a + per, None]
        dE = (d * Ep[:, None, :]).sum(-1)
        k = RHO * i2 ** 4 * (12.0 * t["A"] * i2 ** 3 - 6.0 * t["B"]) + 6.0 * CFA * t["q"] * i3 * i2 * dE
        k = torch.where(free, k, torch.zeros_like(k)) * w
        g += torch.einsum("pn,pnc->nc", k, d)
        g += torch.einsum("pn,pc->nc", -2.0 * CFA * t["q"] * i3 * w, Ep)
    return g


def _ss64(s, t):
    """Solute-solute energies (bonds, LJ, Coulomb) and gradient."""
    x = t["xyz"]
    n = len(x)
    b = torch.as_tensor(np.asarray(s["bonds"]).reshape(-1, 2), device=x.device).long()
    keep = ~torch.eye(n, dtype=torch.bool, device=x.device)
    keep[b[:, 0], b[:, 1]] = keep[b[:, 1], b[:, 0]] = False
    d = x[:, None, :] - x
    r2 = torch.where(keep, d.square().sum(-1), torch.ones((), dtype=x.dtype, device=x.device))
    i2 = 1.0 / r2
    sg = 0.5 * (t["sigma_ss"][:, None] + t["sigma_ss"])
    ep = (t["eps_ss"][:, None] * t["eps_ss"]).sqrt()
    s6 = (sg * sg * i2) ** 3
    zero = torch.zeros_like(r2)
    lj = torch.where(keep, 4.0 * ep * (s6 * s6 - s6), zero)
    co = torch.where(keep, L_B / EPS_M * t["q"][:, None] * t["q"] * i2.sqrt(), zero)
    f = torch.where(keep, (4.0 * ep * (6.0 * s6 - 12.0 * s6 * s6) - co) * i2, zero)
    g = (f[..., None] * d).sum(1)
    e_b = 0.0
    if len(b):
        db = x[b[:, 0]] - x[b[:, 1]]
        r = db.norm(dim=1)
        dr = r - t["bond_r0"]
        e_b = float((0.5 * t["bond_k"] * dr * dr).sum())
        fb = (t["bond_k"] * dr / r)[:, None] * db
        g.index_add_(0, b[:, 0], fb)
        g.index_add_(0, b[:, 1], -fb)
    return e_b, 0.5 * float(lj.sum()), 0.5 * float(co.sum()), g


def _net64(theta, x):
    """The network in 64 bits: x [3][nx][ny][nz], theta the flat vector."""
    F = torch.nn.functional
    lay, o = [], 0
    for co, ci, k in LAYERS:
        w = theta[o:o + co * ci * k ** 3].view(co, ci, k, k, k)
        o += co * ci * k ** 3
        lay.append((w, theta[o:o + co]))
        o += co

    def cv(v, l):
        w, b = lay[l]
        return F.conv3d(v, w, b, padding=w.shape[-1] // 2)

    up = lambda v: F.interpolate(v, scale_factor=2, mode="nearest")  # noqa: E731
    e = [F.relu(cv(x[None], 0))]
    for l in (1, 2, 3):
        e.append(F.relu(cv(F.avg_pool3d(e[-1], 2), l)))
    v = e[3]
    for l, skip in ((4, e[2]), (5, e[1]), (6, e[0])):
        v = F.relu(cv(torch.cat([skip, up(v)], 1), l))
    return cv(v, 7).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda", torch.cuda.current_device())
    if kind == "fields":
        if float(case["nx"]) * case["ny"] * case["nz"] * case["atoms"] > 4e10:
            return None
        s = _solute(case, seed)
        U, E = _field64(_cells64(s), _atoms64(s))
        return dict(U=U, E=E.t().contiguous().reshape(-1))
    if kind == "forces":
        if float(case["nx"]) * case["ny"] * case["nz"] * case["atoms"] > 1.5e10:
            return None
        s = _solute(case, seed)
        t = _atoms64(s)
        pts = _cells64(s)[_tight(s) == 0]
        _, E = _field64(pts, t)
        w = torch.full((len(pts),), float(s["h"]) ** 3, dtype=torch.float64, device=dev)
        g = _solvation_grad64(pts, w, E, t)
        fp, fw = _far64(s)
        g += _solvation_grad64(fp, fw, _field64(fp, t)[1], t)
        return dict(grad=g + _ss64(s, t)[3])
    if kind in ("sweep", "pmf"):
        # labels come out of the flips; the parts that do not depend on them
        s = _solute(case, seed) if kind == "sweep" else _pair(case, seed)
        if len(s["xyz"]) > 4000:
            return None
        t = _atoms64(s)
        b, lj, co, _ = _ss64(s, t)
        fp, fw = _far64(s)
        far = float((_field64(fp, t)[0] * fw).sum())
        if kind == "sweep":
            return dict(terms=dict(far=far, ss=b + lj + co))
        return dict(far=far, lj=lj, coulomb=co)
    if kind == "guess":
        if case["nx"] * case["ny"] * case["nz"] > 1 << 21:
            return None
        s = _solute(case, seed)
        x = _features(s).double().view(3, case["nx"], case["ny"], case["nz"])
        theta = torch.as_tensor(_theta(seed), dtype=torch.float64, device=dev)
        with torch.no_grad():
            return dict(logits=_net64(theta, x))
    if kind == "train":
        th = torch.as_tensor(_theta(seed), dtype=torch.float64, device=dev)
        m, v = torch.zeros_like(th), torch.zeros_like(th)
        c, losses = case["crop"], []
        for k, (x, y) in enumerate(zip(*_crops(case, seed)), 1):
            th.requires_grad_(True)
            z = _net64(th, x.double().view(3, c, c, c))
            loss = torch.nn.functional.binary_cross_entropy_with_logits(z, y.double())
            g, = torch.autograd.grad(loss, th)
            th = th.detach()
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            th = th - 1e-3 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
            losses.append(float(loss.detach()))
        return dict(losses=np.array(losses), theta=th)
    return None
