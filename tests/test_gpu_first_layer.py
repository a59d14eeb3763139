"""The species-factored first layer (forward sums, adjoint forces, tensor-head
vectors) against the FP64 oracle, where its batching can go wrong: rows longer
than one sweep of 96 candidates, an atom without neighbours, every species in
one row, and each channel count and l_max."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from helpers import TOL_F32, rel_maxabs
from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


def ball(n, radius, seed, n_species=S.N_SPECIES, d_min=0.9):
    """n atoms at least d_min apart in a ball (open boundary), every species
    drawn, and one atom out of everybody's reach."""
    rng = np.random.default_rng(seed)
    x = []
    while len(x) < n - 1:
        p = rng.uniform(-radius, radius, 3)
        if np.linalg.norm(p) <= radius and all(np.linalg.norm(p - q) >= d_min for q in x):
            x.append(p)
    x = np.array(x + [[3 * radius + 20.0, 0.0, 0.0]], np.float32).astype(np.float64)
    sp = rng.integers(0, n_species, n).astype(np.uint8)
    return S.System("ball", x, sp, np.arange(n, dtype=np.int32), np.zeros((0, 2), np.int32), np.zeros(0), np.zeros(3))


@pytest.mark.parametrize("C,lmax", [(C, l) for C in (32, 64, 128) for l in (0, 1, 2)])
def test_first_layer_conservative_force(C, lmax):
    sy = ball(170, 5.2, 11)          # rows of up to 168 neighbours within 5 A
    spec = S.cons_spec(1, C, lmax)
    blob = S.cons_weights(spec, 12)
    ctx = core.Context(cons=(spec, blob))
    d = core.DeviceSystem(sy)
    nb = core.nbr_build(ctx, d, spec.rc + 0.5)
    rows = np.diff(nb.row_ptr.cpu().numpy())
    assert rows.max() > 128 and rows.min() == 0
    E, F = core.energy_forces_cons(ctx, d, nb, with_prior=False)
    Eo, Fo = O.cons_energy_forces(sy, spec, blob)
    assert rel_maxabs(F.cpu().numpy(), Fo) <= TOL_F32
    assert abs(E.item() - Eo) <= TOL_F32 * abs(Eo)
    E2, F2, W = core.energy_forces_cons(ctx, d, nb, with_prior=False, with_virial=True)
    assert torch.equal(F, F2)
    # open boundary: the pair-form virial is -sum F . x of the oracle's forces
    scale = float((np.abs(Fo).sum(1)).sum() * (spec.rc + 0.5))
    assert abs(W.item() + float((Fo * sy.x).sum())) <= 1e-5 * scale


@pytest.mark.parametrize("C,n_l", [(32, 1), (32, 4), (64, 2), (64, 3)])
def test_first_layer_nc_force(C, n_l):
    sy = ball(170, 4.6, 21)
    spec = S.nc_spec(C, rc=4.0, n_l=n_l)
    blob = S.nc_weights(spec, 22)
    ctx = core.Context(nc=(spec, blob))
    d = core.DeviceSystem(sy)
    nb = core.nbr_build(ctx, d, spec.rc + 0.5)
    assert np.diff(nb.row_ptr.cpu().numpy()).max() > 96
    F, net = core.forces_nc(ctx, d, nb, with_bonds=False)
    Fo = O.nc_forces(sy, spec, blob, with_bonds=False)[0]
    assert rel_maxabs(F.cpu().numpy(), Fo) <= TOL_F32
    assert float(net.abs().max()) == 0.0
