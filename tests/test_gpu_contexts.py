"""Contexts of different models on different host threads: kernels whose
shared memory depends on the model's species count are launched side by side."""
import ctypes as ct
import dataclasses
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,lmax", [(128, 2), (64, 1)])
def test_two_threads_with_different_species_counts(C, lmax):
    """20,000 calls on each thread, enqueued back to back: every one is
    accepted and the last ones' bits are those of the call made alone."""
    sy = S.capped_molecule_in_droplet(20, 3)
    jobs = []
    for n_species in (5, 8):
        spec = dataclasses.replace(S.cons_spec(1, C, lmax), n_species=n_species)
        ctx = core.Context(cons=(spec, S.cons_weights(spec, 4)))
        d = core.DeviceSystem(sy)
        nb = core.nbr_build(ctx, d, spec.rc + 0.5)
        jobs.append((ctx, d, nb, core.energy_forces_cons(ctx, d, nb, with_prior=False)[1]))
    torch.cuda.synchronize()
    refused, wrong, start = [], [], threading.Barrier(2)

    def work(ctx, d, nb, want):
        st = torch.cuda.Stream()
        E = torch.empty(1, dtype=torch.float64, device="cuda")
        F = torch.empty_like(want)
        s, n = d.struct(), nb.struct()
        args = (ctx.handle, ct.byref(s), ct.byref(n), E.data_ptr(), F.data_ptr(), None, 0, st.cuda_stream)
        start.wait()
        for k in range(20000):
            if ctx.lib.energy_forces_cons(*args) != core.L.OK:
                refused.append(k)
            if k % 200 == 0:
                st.synchronize()
        st.synchronize()
        wrong.append(not torch.equal(F, want))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not refused, (len(refused), refused[:4])
    assert wrong == [False, False]


def test_three_threads_rebuilding_at_once():
    """States of three contexts stepped from three threads, on streams of
    different priority, every inner step with a rebuild whose grid alone fills
    the GPU: the bits of a state stepped alone."""
    cs, ns = S.cons_spec(1, 32, 0), S.nc_spec(32, rc=3.5)
    n = 10000
    sy = S.water_box(n, 12.42 / 64 ** (1 / 3) * n ** (1 / 3), 1)
    m = sy.element_masses()
    v = S.maxwell_boltzmann(m, 300.0, 5)
    ig = core.integrator(0.1, 5, 300.0, [20.0] * 5, skin=2e-4)

    def state():
        ctx = core.Context(cons=(cs, S.cons_weights(cs, 1)), nc=(ns, S.nc_weights(ns, 2)))
        return ctx, core.MDState(core.DeviceSystem(sy), v, m.astype("float32"), seeds=7)

    def run(ctx, st, stream, out):
        try:
            with torch.cuda.stream(stream):
                for n_outer in (1, 3, 6, 1, 1):
                    core.respa_step(ctx, st, ig, n_outer)
                ctx.sync()
                out.append(st.dsys.x.clone())
                stream.synchronize()
        except Exception as e:   # noqa: BLE001 (reported below)
            out.append(repr(e))

    alone, together = [], []
    ctx, st = state()
    torch.cuda.synchronize()
    run(ctx, st, torch.cuda.Stream(), alone)
    st.release()
    jobs = [state() for _ in range(3)]
    torch.cuda.synchronize()
    threads = [threading.Thread(target=run, args=(*j, torch.cuda.Stream(priority=-k), together))
               for k, j in enumerate(jobs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert [o for o in alone + together if isinstance(o, str)] == []
    assert all(torch.equal(o, alone[0]) for o in together)
    for _, st in jobs:
        st.release()
