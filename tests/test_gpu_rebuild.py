"""A state's one-launch rebuild against the separate kernels of nbr_build: the
same rows for a lone atom, replicas with and without neighbours, more cells and
replicas than blocks, and scans of several tiles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


def atoms(n, rng, spread):
    x = rng.uniform(0.0, spread, (n, 3)).astype(np.float32).astype(np.float64) + np.arange(n)[:, None] * [1.3, 0, 0]
    return S.System("atoms", x, np.zeros(n, np.uint8), np.arange(n, dtype=np.int32), np.zeros((0, 2), np.int32),
                    np.zeros(0), np.zeros(3))


def systems(which):
    rng = np.random.default_rng(3)
    if which == "one":
        return [atoms(1, rng, 1.0)]
    if which == "many":
        return [atoms(1 + k % 5, rng, 0.5) for k in range(1500)]
    if which == "ragged":
        return [atoms(300, rng, 4.0), atoms(1, rng, 1.0), atoms(40, rng, 2.0), S.water_192(4)]
    return [S.capped_molecule_in_droplet(200, 5)] * 8


@pytest.mark.parametrize("which", ["one", "many", "ragged", "droplets"])
def test_rows_equal_the_separate_kernels(which):
    sy = systems(which)
    cs, ns = S.cons_spec(1, 32, 1), S.nc_spec(32)
    ctx = core.Context(cons=(cs, S.cons_weights(cs, 1)), nc=(ns, S.nc_weights(ns, 2)))
    m = np.concatenate([s.element_masses() for s in sy])
    d = core.DeviceSystem(sy)
    st = core.MDState(d, S.maxwell_boltzmann(m, 300.0, 5), m.astype(np.float32), seeds=7)
    ig = core.integrator(1.0, 2, 300.0, [1.0] * 5, skin=0.5)
    core.respa_step(ctx, st, ig, 0)
    ctx.sync()
    for which_list in (0, 1):
        got = st.lists(which_list)
        want = core.nbr_build(ctx, d, got.r_list)
        n = want.n_pairs
        assert torch.equal(got.row_ptr, want.row_ptr)
        assert torch.equal(got.col[:n], want.col[:n])
    st.release()
