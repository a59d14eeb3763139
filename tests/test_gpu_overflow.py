"""fp32 contractions of 128 channels at the ends of fp32's range: an operand
beyond bf16's largest value, and sums that overflow, give what fp32 arithmetic
gives (a finite energy, an infinite one), not a NaN."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from helpers import TOL_F32
from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu
C = 128


def model(change):
    """One layer, l_max = 1; `change` gets views of b1, W2, Wr and wo."""
    spec = S.cons_spec(1, C, 1)
    blob = S.cons_weights(spec, 5)
    o = spec.n_species * C + 2 * spec.K * C + 2 * C * C
    b1, W2 = blob[o:o + C], blob[o + C:o + C + C * C].reshape(C, C)
    Wr, wo = blob[-C * C - 2 * C:-2 * C].reshape(C, C), blob[-C:]
    change(b1, W2, Wr, wo)
    return spec, blob


def energy(spec, blob, n_rep, forces=False):
    sy = S.water_192(6)
    ctx = core.Context(cons=(spec, blob))
    d = core.DeviceSystem([sy] * n_rep)
    nb = core.nbr_build(ctx, d, spec.rc + 0.5)
    E, F = core.energy_forces_cons(ctx, d, nb, with_prior=False, forces=forces)
    ctx.sync()
    return sy, E.cpu().numpy(), None if F is None else F.cpu().numpy()


@pytest.mark.parametrize("n_rep", [1, 60])      # narrow and wide tiles
@pytest.mark.parametrize("big", [3.0e38, 3.4e38])   # 3.39e38 is bf16's largest
def test_operand_beyond_the_largest_bf16(big, n_rep):
    def change(b1, W2, Wr, wo):
        b1[0] = np.float32(big)
        W2[:, 0] = (W2[:, 0] * 1e-31).astype(np.float32)

    spec, blob = model(change)
    sy, E, F = energy(spec, blob, n_rep, forces=True)
    Eo, Fo = O.cons_energy_forces(sy, spec, blob)
    assert np.all(np.abs(E - Eo) <= TOL_F32 * abs(Eo))
    assert np.abs(F[:sy.n_atoms] - Fo).max() <= TOL_F32 * np.abs(Fo).max()


@pytest.mark.parametrize("n_rep", [1, 60])
def test_infinite_sums_stay_infinite(n_rep):
    def change(b1, W2, Wr, wo):
        b1[0] = np.float32(3.0e38)
        W2[:, 0] = 2.0                          # 6e38: every feature is +inf
        Wr[:], wo[:] = np.abs(Wr), np.abs(wo)

    _, E, _ = energy(*model(change), n_rep)
    assert np.all(np.isposinf(E))
