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
