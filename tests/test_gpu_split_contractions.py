"""fp32 contractions with operands in three bf16 parts: rows around the
128-row tile, both tile widths, every l_max (K and N of 128, 256 and 384)
against the FP64 oracle, and the distillation's contractions just below and
above the row count from which they are used (K of 144 and 176: a last chunk of
one and of three K steps)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from helpers import TOL_F32, rel_maxabs
from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


def cluster(n, seed):
    rng = np.random.default_rng(seed)
    radius, x = 1.35 * n ** (1 / 3), []
    while len(x) < n:
        p = rng.uniform(-radius, radius, 3)
        if np.linalg.norm(p) <= radius and all(np.linalg.norm(p - q) >= 1.0 for q in x):
            x.append(p)
    x = np.array(x, np.float32).astype(np.float64)
    return S.System("cluster", x, rng.integers(0, S.N_SPECIES, n).astype(np.uint8), np.arange(n, dtype=np.int32),
                    np.zeros((0, 2), np.int32), np.zeros(0), np.zeros(3))


@pytest.mark.parametrize("lmax,n", [(0, 128), (1, 127), (2, 1), (2, 33), (2, 129), (1, 257)])
def test_rows_around_a_tile(lmax, n):
    sy = cluster(n, 4)
    spec = S.cons_spec(2, 128, lmax)
    blob = S.cons_weights(spec, 5)
    ctx = core.Context(cons=(spec, blob))
    d = core.DeviceSystem(sy)
    E, F = core.energy_forces_cons(ctx, d, core.nbr_build(ctx, d, spec.rc + 0.5), with_prior=False)
    Eo, Fo = O.cons_energy_forces(sy, spec, blob)
    assert abs(E.item() - Eo) <= TOL_F32 * abs(Eo)
    assert float(np.abs(F.cpu().numpy() - Fo).max()) <= TOL_F32 * max(1e-3, float(np.abs(Fo).max()))
    # wide tiles: the same replica, the same bits
    k = 1 + 8000 // n
    db = core.DeviceSystem([sy] * k)
    Eb, Fb = core.energy_forces_cons(ctx, db, core.nbr_build(ctx, db, spec.rc + 0.5), with_prior=False)
    assert torch.equal(Fb[-n:], F) and bool((Eb == E[0]).all())


@pytest.mark.parametrize("n_l", [1, 3])
def test_gradient_on_both_sides_of_the_row_rule(n_l):
    """The gradient of k equal frames is k times one frame's: 42 frames of 192
    atoms are below 8192 rows, 43 above. Both are fp32 sums, within 2e-5 of the
    largest entry of each other (1e-5 each)."""
    sy = S.water_192(41)
    spec = S.nc_spec(64, rc=3.5, n_l=n_l)
    ctx = core.Context(nc=(spec, S.nc_weights(spec, 42)))
    T = np.random.default_rng(43).normal(0.0, 10.0, (sy.n_atoms, 3)).astype(np.float32)
    g = []
    for k in (42, 43):
        d = core.DeviceSystem([sy] * k)
        nb = core.nbr_build(ctx, d, spec.rc + 0.5)
        _, gr = core.nc_distill_step(ctx, d, nb, torch.from_numpy(np.tile(T, (k, 1))).cuda(), with_grad=True)
        g.append(gr.double().cpu().numpy() / k)
    assert np.abs(g[1] - g[0]).max() <= 2e-5 * np.abs(g[0]).max()
