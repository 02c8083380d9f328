"""Bookkeeping of the hierarchical sums' tiles on boxes cut anywhere: every
pair of an atom and a cell is counted once, and node values are kept for the
tiles that hold cells alone."""
import numpy as np
import pytest

import oracle as O
from paper_2208_05524_gb300 import vesis
from test_gpu_tree_accuracy import spread

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_atoms,n", [
    (1500, (150, 141, 133)),     # tiles of every level cut
    (1000, (192, 161, 177)),     # whole tiles and one or two cells more
    (2000, (925, 70, 70)),       # one or two tiles of the coarser levels across
    (1000, (600, 600, 17)),
    (2000, (140, 141, 600)),
])
def test_single_solvent_cell(n_atoms, n):
    """Solvent in one cell, charges only: the gradient is one pair term per
    atom (the r^-3 and r^-5 terms never cancel), so a pair missed or met twice
    stands out at full size.  Far terms are interpolated to better than 1e-5 of
    the largest on the tile, at most 40 times the smallest; FP32 coordinates
    give 14 x 2^-24 x 185 A / 3 A."""
    s = spread(n_atoms, n, 0.4, 2)
    s["eps_sw"] = np.zeros(n_atoms)
    S = vesis.System(s, far_field=0, eps_ss=1e30)
    assert S.pair_sums()["gradient"] == "hierarchical"
    rng = np.random.default_rng(3)
    N = np.array(n)
    cells = [N - 1, 0 * N, N // 2, (N - 1) * [1, 0, 0], (N - 1) * [0, 1, 1]]
    cells += [np.minimum(np.array(c), N - 1) for c in ((15, 16, 31), (63, 64, 32), (127, 48, 15))]
    cells += list(rng.integers(0, N, (16, 3)))
    chi = torch.ones(S.G, dtype=torch.uint8, device="cuda")
    E = torch.zeros(3 * S.G, dtype=torch.float32, device="cuda")
    C = O.cfa_prefactor(O.params())
    for c in cells:
        at = int((c[0] * n[1] + c[1]) * n[2] + c[2])
        e = rng.normal(size=3).astype(np.float32)
        chi[at] = 0
        E.view(3, -1)[:, at] = torch.from_numpy(e).cuda()
        g = S.atom_forces(chi, E=E)
        chi[at] = 1
        E.view(3, -1)[:, at] = 0.0
        d = s["origin"] + (c + 0.5) * s["h"] - s["xyz"]
        r = np.linalg.norm(d, axis=1)[:, None]
        assert r.min() > 0.2
        ref = -2 * C * s["q"][:, None] * s["h"] ** 3 * (
            r ** -3 * e - 3 * r ** -5 * (d @ e.astype(np.float64))[:, None] * d)
        err = np.linalg.norm(g - ref, axis=1)
        assert np.all(err <= 1e-3 * np.linalg.norm(ref, axis=1)), c
    S.close()


@pytest.mark.parametrize("n_atoms,n", [(400, (2048, 2048, 4)), (1500, (1, 1500, 1500))])
def test_workspace_of_flat_boxes(n_atoms, n):
    """Device memory per cell: 56 bytes of grid scratch and sweep state, 6.9
    per cell of a whole tile for the node values (16 / 4 and 16 / 1 times that
    on boxes 4 and 1 cells thick), 4 for the coarser levels and lists, and
    allocation granularity."""
    torch.cuda.synchronize()
    a = torch.cuda.mem_get_info()[0]
    S = vesis.System(spread(n_atoms, n, 0.4, 5))
    used = a - torch.cuda.mem_get_info()[0]
    assert S.pair_sums()["fields"] == "hierarchical"
    thin = 16 / min(n)
    assert used <= (56 + 1.5 * 6.9 * thin + 32) * S.G + 300e6
    S.close()


def test_without_room_for_the_workspace():
    """A system whose grid fits but whose hierarchical workspace (80 MB here)
    does not is created all the same and sums directly."""
    s = spread(1500, (150, 141, 133), 0.4, 2)
    chi = torch.ones(150 * 141 * 133, dtype=torch.uint8, device="cuda")
    chi[::3] = 0

    def sums():
        S = vesis.System(s)
        U = torch.empty(S.G, dtype=torch.float32, device="cuda")
        S.energy_field(U)
        kind = S.pair_sums()
        g = S.atom_forces(chi)
        S.close()
        return kind, U, g

    kind, U, g = sums()
    assert kind == dict(fields="hierarchical", gradient="hierarchical")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    a = torch.cuda.mem_get_info()[0]
    S = vesis.System(s)
    used = a - torch.cuda.mem_get_info()[0]
    S.close()
    # half the workspace is left once the rest (and U) has its place
    full = torch.empty(a - used - U.nbytes + (40 << 20), dtype=torch.uint8, device="cuda")
    try:
        kind, Ud, gd = sums()
    finally:
        del full
        torch.cuda.empty_cache()
    assert kind == dict(fields="direct", gradient="direct")
    small = U.abs() < 1.0
    assert torch.allclose(U[small], Ud[small], rtol=1e-3, atol=1e-5)
    assert np.abs(g - gd).max() <= 1e-4 * np.abs(g).max()


def test_autotune_leaves_hierarchical_sums_alone():
    """Nothing to choose: one time for all shapes, and the shapes set before;
    a gradient below its line is still tuned."""
    s = spread(1500, (150, 141, 133), 0.4, 2)
    chi = torch.zeros(150 * 141 * 133, dtype=torch.uint8, device="cuda")
    S = vesis.System(s)
    S.set_tiles(16, 2)
    r = S.autotune(chi, reps=1)
    ms = r["ms"]
    assert ms["energy_pencil4"] == ms["energy_pencil8"] == ms["energy_pencil16"] > 0.0
    assert ms["force_atoms2"] == ms["force_atoms4"] > 0.0
    assert S.get_tiles() == (16, 2)
    S.close()
    S = vesis.System(spread(700, (150, 141, 140), 0.4, 2))
    assert S.pair_sums() == dict(fields="hierarchical", gradient="direct")
    ms = S.autotune(torch.zeros(S.G, dtype=torch.uint8, device="cuda"), reps=1)["ms"]
    assert ms["energy_pencil4"] == ms["energy_pencil8"] == ms["energy_pencil16"] > 0.0
    assert ms["force_atoms2"] > 0.0 and ms["force_atoms4"] > 0.0
    S.close()
