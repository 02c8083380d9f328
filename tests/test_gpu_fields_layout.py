"""The direct energy kernel stores four cells at a time where rows and arrays
allow it and one by one elsewhere: the same bits on every row length, alignment
of U and E and pencil length, and nothing written around them."""
import numpy as np
import pytest

import oracle as O
from paper_2208_05524_gb300 import synth, vesis

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nz", [1, 2, 3, 4, 5, 8, 9, 12, 20])
def test_fields_at_any_alignment(nz):
    n, h = (7, 6, nz), 0.4
    s = synth.single_ion(n=8, h=h)
    s["n"], s["origin"] = np.array(n), -0.5 * np.array(n) * h
    S = vesis.System(s, far_field=0)
    G = S.G
    U0 = torch.empty(G, dtype=torch.float32, device="cuda")
    E0 = torch.empty(3 * G, dtype=torch.float32, device="cuda")
    S.energy_field(U0, E0)
    Uo, _, Eo = O.fields(s, O.params(far_field=0))
    # the FP32 rounding of one atom's terms: coordinates, distance, powers
    tol = 64 * 2.0 ** -24
    assert np.all(np.abs(U0.cpu().numpy() - Uo.ravel()) <= tol * np.abs(Uo).max())
    for pencil in (4, 8, 16):
        S.set_tiles(pencil, 4)
        for u in (0, 1, 2, 4):
            for e in (0, 3, 4):
                Ub = torch.full((G + 12,), 7.0, dtype=torch.float32, device="cuda")
                Eb = torch.full((3 * G + 12,), 7.0, dtype=torch.float32, device="cuda")
                S.energy_field(Ub[u:u + G], Eb[e:e + 3 * G])
                assert torch.equal(Ub[u:u + G], U0) and torch.equal(Eb[e:e + 3 * G], E0)
                assert bool((Ub[:u] == 7.0).all()) and bool((Ub[u + G:] == 7.0).all())
                assert bool((Eb[:e] == 7.0).all()) and bool((Eb[e + 3 * G:] == 7.0).all())
    S.close()
