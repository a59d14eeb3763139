"""The barrier of a state's one-launch rebuild: a block that never comes ends
the wait with DMTS_E_TIMEOUT and leaves the context usable, and a list overflow
inside a rebuild stops every block at the next barrier."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def models():
    cs, ns = S.cons_spec(1, 32, 1), S.nc_spec(32, rc=3.5)
    return (cs, S.cons_weights(cs, 1)), (ns, S.nc_weights(ns, 2))


def run(ctx, n_outer=3):
    sy = S.water_192(4)
    m = sy.element_masses()
    d = core.DeviceSystem(sy)
    st = core.MDState(d, S.maxwell_boltzmann(m, 300.0, 5), m.astype(np.float32), seeds=7)
    core.respa_step(ctx, st, core.integrator(2.0, 2, 300.0, [1.0] * 5, skin=0.3), n_outer)
    ctx.sync()
    x = d.x.clone()
    st.release()
    return x


@pytest.mark.parametrize("absent", [0, 1])
def test_a_block_that_never_comes(models, absent):
    ctx = core.Context(cons=models[0], nc=models[1])
    t0 = time.perf_counter()
    assert core.check_bounded_barrier(ctx, 2000, absent) == core.L.E_TIMEOUT
    assert time.perf_counter() - t0 < 5.0
    assert core.check_bounded_barrier(ctx, 100000, -1) == core.L.OK
    want = run(core.Context(cons=models[0], nc=models[1]))
    assert torch.equal(run(ctx), want)


def test_bad_arguments(models):
    ctx = core.Context(cons=models[0], nc=models[1])
    for limit, absent in ((0, 0), (1000001, 0), (10, 2), (10, -2)):
        assert ctx.lib.dmts_check_bounded_barrier(ctx.handle, limit, absent, core._stream()) == core.L.E_INVALID


def test_overflow_inside_a_rebuild(models):
    """Lists sized for a gas without pairs, then every atom moved into reach of
    all others: the next step's rebuild overflows, the call reports it, nothing
    is left behind for the context's other states."""
    ctx = core.Context(cons=models[0], nc=models[1])
    n = 600
    gas = np.arange(n)[:, None] * np.array([12.0, 0.0, 0.0])
    sy = S.System("gas", gas, np.zeros(n, np.uint8), np.arange(n, dtype=np.int32), np.zeros((0, 2), np.int32),
                  np.zeros(0), np.zeros(3))
    m = sy.element_masses()
    d = core.DeviceSystem(sy)
    st = core.MDState(d, np.zeros((n, 3)), m.astype(np.float32), seeds=7)
    ig = core.integrator(1.0, 2, 300.0, [1.0] * 5, skin=0.5)
    core.respa_step(ctx, st, ig, 1)
    ctx.sync()
    assert st.lists(0).n_pairs == 0
    rng = np.random.default_rng(6)
    d.x.copy_(torch.from_numpy(rng.uniform(0.0, 2.5, (n, 3)).astype(np.float32)).cuda())   # 359,400 pairs
    core.respa_step(ctx, st, ig, 1)
    with pytest.raises(core.L.DmtsError) as e:
        ctx.sync()
    assert e.value.status == core.L.E_NBR_OVERFLOW
    ctx.sync()
    st.release()
    assert torch.equal(run(ctx), run(core.Context(cons=models[0], nc=models[1])))
