"""Rounding and interpolation errors of the hierarchical pair sums against 64
bits, beside those of the direct kernels on the same solute cut into parts
(parts of fewer than 400 atoms are summed directly; their fields are added in
64 bits here, which leaves out the rounding of the longer sum that the direct
kernel would form for the whole)."""
import numpy as np
import pytest

import oracle as O
from paper_2208_05524_gb300 import synth, vesis

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def globule(n_atoms, n, h, seed, smax=4.0):
    """Atoms spread evenly over a ball of 0.05 atoms per cubic Angstrom."""
    rng = np.random.default_rng(seed)
    n = np.array(n)
    r = (3 * n_atoms / (0.05 * 4 * np.pi)) ** (1 / 3)
    v = rng.normal(size=(n_atoms, 3))
    xyz = v / np.linalg.norm(v, axis=1)[:, None] * (r * rng.random(n_atoms) ** (1 / 3))[:, None]
    sigma, eps, q = synth._params(rng, n_atoms, 298.0, -3.0)
    sigma = np.minimum(sigma * (smax / sigma.max()), smax)
    z = np.zeros(n_atoms)
    return dict(xyz=xyz, sigma_sw=sigma, eps_sw=eps, q=q, sigma_ss=z, eps_ss=z,
                bonds=np.zeros((0, 2), np.int32), bond_k=np.zeros(0), bond_r0=np.zeros(0), n=n,
                h=h, origin=-0.5 * n * h)


def spread(n_atoms, n, h, seed):
    """The same atoms spread evenly over the box."""
    s = globule(n_atoms, n, h, seed)
    s["xyz"] = np.random.default_rng(seed).uniform(-0.98, 0.98, (n_atoms, 3)) * -s["origin"]
    return s


def _t(a):
    return torch.as_tensor(np.asarray(a, np.float64), device="cuda")


def _centres(s, idx):
    ny, nz = int(s["n"][1]), int(s["n"][2])
    ijk = torch.stack([idx // (ny * nz), (idx // nz) % ny, idx % nz], 1)
    return _t(s["origin"]) + (ijk.double() + 0.5) * s["h"]


def fields64(s, idx):
    """U and E of the cells idx in 64 bits."""
    p = O.params()
    pos, xyz, sg, ep, q = _centres(s, idx), *(_t(s[k]) for k in ("xyz", "sigma_sw", "eps_sw", "q"))
    U, E = [], []
    for a in range(0, len(idx), 8192):
        d = pos[a:a + 8192, None] - xyz[None]
        r = d.square().sum(-1).sqrt().clamp_min(p["rmin"])
        s6 = (sg / r) ** 6
        e = ((q * r ** -3)[..., None] * d).sum(1)
        E.append(e)
        U.append((4 * p["rho_w"] * ep * (s6 * s6 - s6)).sum(1) +
                 O.cfa_prefactor(p) * e.square().sum(1))
    return torch.cat(U), torch.cat(E)


def gradient64(s, chi, E, atoms):
    """The grid gradient of some atoms in 64 bits, for the given field E [3][G]
    (Eq. GradientG; clamped pairs keep the r^-3 E part)."""
    p = O.params()
    C = O.cfa_prefactor(p)
    xyz, sg, ep, q = (_t(s[k])[atoms] for k in ("xyz", "sigma_sw", "eps_sw", "q"))
    A, B = 4 * ep * sg ** 12, 4 * ep * sg ** 6
    cells = torch.nonzero(chi == 0).flatten()
    out = torch.zeros(len(atoms), 3, dtype=torch.float64, device="cuda")
    for a in range(0, len(cells), 1 << 18):
        c = cells[a:a + (1 << 18)]
        d = _centres(s, c)[:, None] - xyz[None]
        r = d.square().sum(-1).sqrt()
        far = r >= p["rmin"]
        r = r.clamp_min(p["rmin"])
        e = E[:, c].double().T
        cd = p["rho_w"] * (12 * A * r ** -14 - 6 * B * r ** -8) + \
            6 * C * q * r ** -5 * (d * e[:, None]).sum(-1)
        out += ((cd * far)[..., None] * d).sum(0) - 2 * C * ((q * r ** -3).T @ e)
    return out * s["h"] ** 3


def fields(s):
    """U, E [3][G] and the kind of sums of a system."""
    S = vesis.System(s, far_field=0)
    U = torch.empty(S.G, dtype=torch.float32, device="cuda")
    E = torch.empty(3 * S.G, dtype=torch.float32, device="cuda")
    S.energy_field(U, E)
    kind = S.pair_sums()["fields"]
    S.close()
    return U, E.view(3, -1), kind


def tight(s):
    S = vesis.System(s, far_field=0)
    chi = torch.empty(S.G, dtype=torch.uint8, device="cuda")
    S.init_labels(chi, "tight")
    S.close()
    return chi


def rms(x):
    return float(x.square().mean().sqrt())


# boxes of at least 2e9 pairs: the fewest atoms, spacings at and above the
# resolution line (16 h = 1.2 sigma), a ragged box
FIELDS = [
    (400, (172, 172, 172), 0.4, 4.0),
    (1000, (141, 150, 133), 0.4, 4.0),
    (1000, (166, 166, 166), 0.3, 4.0),
    (2000, (147, 147, 147), 0.5, 4.0),
    (1500, (160, 160, 160), 0.35, 4.66),
]


@pytest.mark.parametrize("n_atoms,n,h,smax", FIELDS)
def test_fields_round_like_direct_sums(n_atoms, n, h, smax):
    """Over solvent cells, the rms errors of U and E are at most 1.5 times
    those of the parts' direct sums."""
    s = globule(n_atoms, n, h, 3, smax)
    U, E, kind = fields(s)
    assert kind == "hierarchical"
    sol = torch.nonzero(tight(s) == 0).flatten()
    pick = np.random.default_rng(5).integers(0, len(sol), 60000)
    idx = sol[torch.as_tensor(pick, device="cuda")]
    U64, E64 = fields64(s, idx)
    m = -(-n_atoms // 250)
    lj, Ed = 0.0, 0.0
    C = O.cfa_prefactor(O.params())
    for k in range(m):
        u, e, kind = fields(synth.subset(s, np.arange(k, n_atoms, m)))
        assert kind == "direct"
        u, e = u[idx].double(), e[:, idx].double()
        lj = lj + u - C * e.square().sum(0)
        Ed = Ed + e
    Ud = lj + C * Ed.square().sum(0)
    assert rms(U[idx].double() - U64) <= 1.5 * rms(Ud - U64)
    assert rms(E[:, idx].double().T - E64) <= 1.5 * rms(Ed.T - E64)


def test_few_atoms_are_summed_directly():
    """Below 400 atoms the direct sums round less far from the solute."""
    for n_atoms, kind in ((256, "direct"), (399, "direct"), (400, "hierarchical")):
        assert fields(globule(n_atoms, (256, 200, 200), 0.4, 1))[2] == kind


# globules, and atoms spread over the box: cubes, boxes long in x (narrow
# columns) and in z (rows of more than two stages of 256 cells), flat boxes
GRADIENTS = [
    (globule, 1000, (166, 166, 166), 0.3),
    (globule, 1200, (700, 100, 110), 0.4),
    (globule, 2000, (140, 141, 600), 0.4),
    (spread, 1000, (600, 600, 17), 0.4),
    (spread, 400, (2048, 2048, 4), 0.4),
    (spread, 2000, (925, 70, 70), 0.4),
]


@pytest.mark.parametrize("make,n_atoms,n,h", GRADIENTS)
def test_gradient_rounds_like_direct_sums(make, n_atoms, n, h):
    """For the same labels and field, the rms error over 64 atoms is at most
    1.25 times that of the direct kernel on the atoms in parts (both carry the
    rounding of the FP32 coordinates and of the near rows)."""
    s = make(n_atoms, n, h, 4)
    chi, E = tight(s), fields(s)[1]
    args = dict(far_field=0, eps_ss=1e30)
    S = vesis.System(s, **args)
    assert S.pair_sums()["gradient"] == "hierarchical"
    g = S.atom_forces(chi, E=E.reshape(-1))
    S.close()
    gd = np.zeros_like(g)
    m = -(-n_atoms // 350)
    for k in range(m):
        S = vesis.System(synth.subset(s, np.arange(k, n_atoms, m)), **args)
        assert S.pair_sums()["gradient"] == "direct"
        gd[k::m] = S.atom_forces(chi, E=E.reshape(-1))
        S.close()
    atoms = np.random.default_rng(6).choice(n_atoms, 64, replace=False)
    ref = gradient64(s, chi, E, torch.as_tensor(atoms, device="cuda")).cpu().numpy()
    err = np.sqrt(np.mean((g[atoms] - ref) ** 2))
    assert err <= 1.25 * np.sqrt(np.mean((gd[atoms] - ref) ** 2))


@pytest.mark.parametrize("make,n_atoms,n,kind", [
    (spread, 2000, (70, 70, 925), "direct"),        # 4383 us direct, 8316 by nodes
    (spread, 2000, (925, 70, 70), "hierarchical"),  # 4687, 1501
    (spread, 700, (65, 65, 1400), "direct"),        # 2404, 8702
    (spread, 1000, (17, 600, 600), "direct"),       # 3028, 4056
    (spread, 1000, (600, 600, 17), "hierarchical"), # 3522, 1346
    (globule, 1000, (166, 166, 167), "hierarchical"),
])
def test_gradient_rule_follows_the_shape(make, n_atoms, n, kind):
    """Long z and boxes a few columns wide keep the direct gradient; the fields
    are hierarchical in all of these."""
    S = vesis.System(make(n_atoms, n, 0.4, 1))
    assert S.pair_sums() == dict(fields="hierarchical", gradient=kind)
    S.close()
