"""The flip sweep's load forms, estimates and tile dealing against the oracle:
rows of W and U at every alignment, ties between equal flip energies, energies
of extreme size, and more tiles than one bitmap word per block holds."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2208_05524_gb300 import synth

pytestmark = pytest.mark.gpu


def _blob(n, seed):
    x = [(np.arange(v) - 0.5 * v) / (0.5 * v) for v in n]
    d = x[0][:, None, None] ** 2 + x[1][None, :, None] ** 2 + x[2][None, None, :] ** 2
    return (d < 0.4 + 0.2 * synth.random_field(n, seed=seed, scale=1.0)).astype(np.uint8)


ROUNDS = 200
# (cells, U offset in elements, kernel options, kind of U)
CASES = {
    "rows_of_8": ((24, 20, 32), 0, {}, "random"),
    "odd_rows": ((21, 19, 29), 0, {}, "random"),
    "odd_rows_stencil": ((21, 19, 29), 0, {"kernel": "sin2", "sin2_lambda": 2.0}, "random"),
    "rows_of_4": ((10, 13, 12), 0, {}, "random"),
    "short_rows": ((18, 17, 3), 0, {}, "random"),
    "unaligned_u": ((24, 20, 32), 1, {}, "random"),
    "ties": ((24, 24, 24), 0, {}, "constant"),
    "extremes": ((24, 20, 27), 0, {}, "extreme"),
    "many_tiles": ((9, 105, 1393), 0, {}, "random"),
}


@pytest.mark.parametrize("case", CASES)
def test_sweep_forms(case):
    """Identical rounds, flips and labels over at most 200 rounds; the summed
    dE to FP64 rounding: at most 10^5 terms of one sign, 10^5 / 2^53 = 1.1e-11."""
    import paper_2208_05524_gb300.vesis as vs
    n, off, kw, kind = CASES[case]
    h = 0.3
    s = synth.single_ion(n=8, h=h)
    s["n"] = np.array(n)
    s["origin"] = -0.5 * np.array(n) * h
    chi0 = _blob(n, 41)
    U32 = (synth.random_field(n, seed=43, scale=0.05) - 0.02).astype(np.float32)
    if kind == "constant":
        U32[:] = np.float32(-0.01)
    elif kind == "extreme":
        U32[::5] *= np.float32(1e30)
        U32[1::5] *= np.float32(1e-30)
    sc = O.surface_constants(s, O.params(**kw))
    ref = chi0.copy()
    ro = O.blsm_parallel(ref, U32.astype(np.float64), sc, max_rounds=ROUNDS)
    assert ro["rounds"] > 0
    S = vs.System(s, **kw)
    buf = torch.zeros(U32.size + off, dtype=torch.float32, device="cuda")
    U = buf[off:]
    U.copy_(torch.from_numpy(U32.reshape(-1)))
    for mode in (-1, 0, 1):
        S.set_sweep_stamps(mode)
        chi = torch.from_numpy(chi0.reshape(-1).copy()).cuda()
        r = S.blsm_relax(chi, U, max_rounds=ROUNDS, terms=False)
        assert r["rounds"] == ro["rounds"] and r["flips"] == ro["flips"], mode
        assert np.array_equal(chi.cpu().numpy(), ref.reshape(-1)), mode
        assert r["dE_sum"] == pytest.approx(ro["dE_sum"], rel=1.2e-11), mode
