"""The fp32 contraction's two tile sizes: a replica's results are the same bits
alone (small tiles) and inside a batch large enough for the large tiles, at
row counts that leave ragged tiles, and the forces match the FP64 oracle;
ragged N and K (the head's 2 H n_c columns) through the distillation."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from helpers import TOL_F32, rel_maxabs
from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,lmax,n_solute", [(32, 2, 21), (64, 1, 33), (128, 2, 27)])
def test_replica_alone_and_in_a_large_batch(C, lmax, n_solute):
    sy = S.capped_molecule_in_droplet(n_solute, 5)
    n_rep = 20000 // sy.n_atoms
    spec = S.cons_spec(2, C, lmax)
    blob = S.cons_weights(spec, 6)
    ctx = core.Context(cons=(spec, blob))

    def forces(systems):
        d = core.DeviceSystem(systems)
        return core.energy_forces_cons(ctx, d, core.nbr_build(ctx, d, spec.rc + 0.5), with_prior=False)

    E1, F1 = forces([sy])
    En, Fn = forces([sy] * n_rep)
    for r in (0, n_rep // 2, n_rep - 1):
        assert torch.equal(F1, Fn[r * sy.n_atoms:(r + 1) * sy.n_atoms])
    assert bool((En == E1[0]).all())
    Eo, Fo = O.cons_energy_forces(sy, spec, blob)
    assert rel_maxabs(F1.cpu().numpy(), Fo) <= TOL_F32


@pytest.mark.parametrize("C,n_l,n_rep", [(32, 1, 1), (64, 3, 1), (64, 1, 110)])
def test_distillation_gradient_is_the_sum_over_the_batch(C, n_l, n_rep):
    """N and K of 2 (8 + n_l) 8 = 144 and 176 columns; the gradient of n equal
    frames is n times that of one, up to fp32 summation order."""
    sy = S.water_192(31)
    spec = S.nc_spec(C, rc=3.5, n_l=n_l)
    blob = S.nc_weights(spec, 32)
    ctx = core.Context(nc=(spec, blob))
    T = np.random.default_rng(33).normal(0.0, 10.0, (sy.n_atoms, 3)).astype(np.float32)

    def grad(k):
        d = core.DeviceSystem([sy] * k)
        nb = core.nbr_build(ctx, d, spec.rc + 0.5)
        loss, g = core.nc_distill_step(ctx, d, nb, torch.from_numpy(np.tile(T, (k, 1))).cuda(), with_grad=True)
        return loss.cpu().numpy(), g.double().cpu().numpy()

    l1, g1 = grad(1)
    ref = O.nc_forces(sy, spec, blob)[0]
    assert abs(l1[0] - ((ref - T) ** 2).sum()) <= 1e-4 * l1[0]
    ln, gn = grad(n_rep + 1)
    assert np.all(ln == l1[0])
    assert np.abs(gn - (n_rep + 1) * g1).max() <= 2e-4 * np.abs(gn).max()


@pytest.mark.parametrize("lmax,n,radius", [(0, 40, 3.4), (1, 70, 4.2), (2, 64, 4.6), (2, 150, 5.2), (2, 300, 7.5)])
def test_tensor_core_layers_over_chunk_edges(lmax, n, radius):
    """Rows from none to more than two chunks of 64 edges and more than the 96
    candidates in flight. The model force within 2e-3 of its RMS of
    the oracle, as every split-bf16 path, and each replica the same bits alone
    and batched."""
    rng = np.random.default_rng(7 + n)
    x = []
    while len(x) < n - 1:
        p = rng.uniform(-radius, radius, 3)
        if np.linalg.norm(p) <= radius and all(np.linalg.norm(p - q) >= 0.9 for q in x):
            x.append(p)
    x = np.array(x + [[60.0, 0.0, 0.0]], np.float32).astype(np.float64)
    sy = S.System("ball", x, rng.integers(0, S.N_SPECIES, n).astype(np.uint8), np.arange(n, dtype=np.int32),
                  np.zeros((0, 2), np.int32), np.zeros(0), np.zeros(3))
    spec = S.cons_spec(3, 128, lmax, bf16=True)
    blob = S.cons_weights(spec, 8)
    ctx = core.Context(cons=(spec, blob))

    def forces(systems):
        d = core.DeviceSystem(systems)
        return core.energy_forces_cons(ctx, d, core.nbr_build(ctx, d, spec.rc + 0.5), with_prior=False)[1]

    F = forces([sy])
    _, Fo = O.cons_energy_forces(sy, spec, blob)
    err = np.abs(F.cpu().numpy() - Fo).max()
    assert err <= 2e-3 * np.sqrt((Fo ** 2).mean())
    other = S.capped_molecule_in_droplet(30, 9)
    Fb = forces([other, sy, other])
    assert torch.equal(F, Fb[other.n_atoms:other.n_atoms + n])
