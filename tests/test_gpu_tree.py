"""Hierarchical pair sums (systems of at least 256 atoms and 2e9 pairs, 4e9
for the gradient) against plain sums in 64 bits: atoms anywhere in the box (its faces and
tile borders included), ragged grids, tiles cut by the grid's end.

Tolerances follow from the arithmetic: coordinates are FP32 (each within
2^-24 of the box half-width L), a pair term depends on the distance with at
most the 14th power, a term takes some 32 roundings and n of them are summed
with random signs (8 sqrt(n) ulps), and the interpolation of far terms is
good to 5e-6 of their magnitudes at these spacings.
"""
import numpy as np
import pytest

import oracle as O
from paper_2208_05524_gb300 import synth, vesis

pytestmark = pytest.mark.gpu
ULP = 2.0 ** -24


def box_system(n_atoms, n, h, seed, parked=()):
    """Atoms spread over the whole box, some parked at given fractions of it."""
    rng = np.random.default_rng(seed)
    n = np.array(n)
    L = 0.5 * n * h
    xyz = rng.uniform(-0.98, 0.98, (n_atoms, 3)) * L
    for i, p in enumerate(parked):
        xyz[i] = np.asarray(p) * L
    sigma, eps, q = synth._params(rng, n_atoms, 298.0, -3.0)
    z = np.zeros(n_atoms)
    return dict(xyz=xyz, sigma_sw=sigma, eps_sw=eps, q=q, sigma_ss=z, eps_ss=z,
                bonds=np.zeros((0, 2), np.int32), bond_k=np.zeros(0), bond_r0=np.zeros(0), n=n,
                h=h, origin=-L)


def field64(s, cells, p):
    """U, E and the bounds on their FP32 errors at some cells."""
    pos = np.asarray(s["origin"]) + (cells + 0.5) * s["h"]
    d = pos[:, None, :] - s["xyz"][None]
    r = np.maximum(np.sqrt((d ** 2).sum(-1)), p["rmin"])
    A = 4 * s["eps_sw"] * s["sigma_sw"] ** 12
    B = 4 * s["eps_sw"] * s["sigma_sw"] ** 6
    C = O.cfa_prefactor(p)
    lj, w = p["rho_w"] * (A * r ** -12 - B * r ** -6), s["q"] * r ** -3
    E = (w[..., None] * d).sum(1)
    delta = 4 * ULP * np.abs(np.asarray(s["origin"])).max() / r
    rel = 14 * delta + ULP * (32 + 8 * np.sqrt(len(s["xyz"]))) + 5e-6
    bE = (np.abs(s["q"]) * r ** -2 * rel).sum(1)
    bL = (p["rho_w"] * (A * r ** -12 + B * r ** -6) * rel).sum(1)
    En = np.linalg.norm(E, axis=1)
    U = lj.sum(1) + C * En ** 2
    return U, E, bL + np.abs(C) * (2 * En * bE + bE ** 2) + 4 * ULP * np.abs(U), bE


CASES = [
    # tiles cut by the grid's end on every axis
    (1000, (150, 141, 133), 0.4, 1),
    # a thin box: one 64-cell tile across z, odd rows
    (1500, (257, 130, 65), 0.4, 2),
    # spacing at the edge of the rule (16 h = 1.2 sigma of the largest atom)
    (900, (145, 160, 128), 0.3, 3),
    # whole tiles
    (512, (192, 128, 192), 0.5, 4),
]


@pytest.mark.parametrize("n_atoms,n,h,seed", CASES)
def test_fields(n_atoms, n, h, seed):
    import torch
    # atoms on tile borders, in corners and at cell centres
    s = box_system(n_atoms, n, h, seed, [(0, 0, 0), (-0.999, -0.999, -0.999), (0.999, 0.999, 0.999),
                                         (0.999, -0.999, 0), (16 / n[0] - 1 + 16 / n[0], 0, 0)])
    s["sigma_sw"] = np.minimum(s["sigma_sw"], 16 * h / 1.2)
    p = O.params()
    S = vesis.System(s)
    U = torch.empty(S.G, dtype=torch.float32, device="cuda")
    E = torch.empty(3 * S.G, dtype=torch.float32, device="cuda")
    S.energy_field(U, E)
    rng = np.random.default_rng(seed)
    cells = rng.integers(0, n, (2500, 3))
    near = np.floor((s["xyz"] - s["origin"]) / h).astype(int)[:300]      # cells holding atoms
    edge = np.array([[a, b, c] for a in (0, 15, 16, n[0] - 1) for b in (0, 63, 64, n[1] - 1)
                     for c in (0, 31, 32, n[2] - 1)])
    cells = np.concatenate([cells, near, edge])
    U64, E64, bU, bE = field64(s, cells, p)
    idx = torch.from_numpy((cells[:, 0] * n[1] + cells[:, 1]) * n[2] + cells[:, 2]).cuda()
    u = U[idx].double().cpu().numpy()
    e = E.view(3, -1)[:, idx].double().cpu().numpy().T
    assert np.all(np.isfinite(u)) and np.all(np.isfinite(e))
    assert np.all(np.linalg.norm(e - E64, axis=1) <= bE)
    assert np.all(np.abs(u - U64) <= bU)
    U2, E2 = torch.empty_like(U), torch.empty_like(E)
    S.energy_field(U2, E2)
    assert torch.equal(U, U2) and torch.equal(E, E2)     # one order of every sum


GRADIENT_CASES = [
    (1500, (150, 141, 133), 0.4, 11),
    (2000, (257, 130, 65), 0.4, 12),
    (1400, (145, 160, 128), 0.3, 13),
    (1000, (192, 128, 192), 0.5, 14),
    # one column of tiles across y, rows longer than two stages of 256 cells
    (9000, (40, 21, 600), 0.4, 15),
]


@pytest.mark.parametrize("n_atoms,n,h,seed", GRADIENT_CASES)
def test_gradient(n_atoms, n, h, seed):
    """The solvation gradient (solute-solute terms off) against the oracle's,
    labels of the tight start and random ones."""
    import torch
    s = box_system(n_atoms, n, h, seed)
    s["sigma_sw"] = np.minimum(s["sigma_sw"], 16 * h / 1.2)
    s["init"] = {"kind": "tight", "d": s["sigma_sw"]}
    p = O.params(eps_ss=1e30)
    S = vesis.System(s, eps_ss=1e30)
    chi = torch.empty(S.G, dtype=torch.uint8, device="cuda")
    S.init_labels(chi, "tight")
    if seed % 2:
        chi |= torch.from_numpy(synth.random_labels(n, seed, 0.3).reshape(-1)).cuda()
    g = S.atom_forces(chi)
    assert np.array_equal(g, S.atom_forces(chi))
    ref = O.gradient(s, p, chi.cpu().numpy().reshape(tuple(n)))
    # forces of one atom add over cells at 3.5 A and beyond: the terms'
    # relative bound against the largest component
    L = 0.5 * max(n) * h
    tol = 14 * 4 * ULP * L / 3.0 + ULP * (32 + 8 * np.sqrt(4096 * 27)) + 5e-6
    assert np.all(np.abs(g - ref) <= tol * np.abs(ref).max())


def test_additive():
    """E is additive over atoms: the hierarchical field of a solute against
    the sum of the direct fields of its parts (too few atoms for the
    hierarchy), bit for bit repeatable and within FP32 rounding."""
    import torch
    n, h = (150, 141, 133), 0.4
    s = box_system(800, n, h, 7)
    fields = []
    for idx in [np.arange(800)] + [np.arange(k, 800, 4) for k in range(4)]:
        S = vesis.System(synth.subset(s, idx))
        U = torch.empty(S.G, dtype=torch.float32, device="cuda")
        E = torch.empty(3 * S.G, dtype=torch.float32, device="cuda")
        S.energy_field(U, E)
        fields.append(E.double())
    tot = sum(fields[1:])
    rms = tot.square().mean().sqrt()
    # both sides carry the rounding of 800 terms; most cells see |E| of rms
    assert (fields[0] - tot).square().mean().sqrt() <= 2 * ULP * (32 + 8 * np.sqrt(800)) * rms


def test_rejected_steps_leave_no_trace():
    """Trial steps that throw atoms out of the box are evaluated (with the
    atoms in the border tiles) and rejected; the gradient at the start
    afterwards is the same bit for bit."""
    import torch
    n, h = (150, 141, 133), 0.4
    s = box_system(1500, n, h, 8)
    S = vesis.System(s)
    chi = torch.empty(S.G, dtype=torch.uint8, device="cuda")
    S.init_labels(chi, "tight")
    g = S.atom_forces(chi)
    r = S.relax(chi.clone(), s["xyz"], max_outer=1, M0=1e6, max_gd_retries=2)
    assert r["stop_reason"] == 3 and r["gd_trials"] == 3
    assert np.array_equal(r["xyz"], s["xyz"])
    S.set_positions(s["xyz"])
    assert np.array_equal(g, S.atom_forces(chi))
