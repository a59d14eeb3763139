"""Kernels scheduled before their predecessor has ended, against a process in
which no two kernels overlap (CUDA_LAUNCH_BLOCKING=1: a launch returns when its
kernel has ended): every call that launches them in sequence gives the same
bits, right behind a copy, on the default stream and on another."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2602_14975_gb300 import core  # noqa: E402
from paper_2602_14975_gb300 import synth as S  # noqa: E402

pytestmark = pytest.mark.gpu


def md(ctx, systems, mode, calls):
    m = np.concatenate([s.element_masses() for s in systems])
    d = core.DeviceSystem(systems)
    st = core.MDState(d, S.maxwell_boltzmann(m, 300.0, 5), m.astype(np.float32), seeds=7)
    ig = core.integrator(2.0, 3, 300.0, [1.0] * 5, mode=mode, skin=0.3)
    for n in calls:
        core.respa_step(ctx, st, ig, n)
    out = [d.x.clone(), st.v.clone(), st.f_nc.clone(), st.f_cons.clone(), st.energy.clone()]
    st.release()
    return out


def collect():
    """Every output, enqueued without a wait of its own between the calls."""
    out = {}

    def keep(name, tensors):
        out.update({f"{name}_{k}": t for k, t in enumerate(tensors)})

    sy = S.water_192(3)
    rng = np.random.default_rng(5)
    for n_rep, C, bf16 in ((1, 64, False), (1, 128, True), (12, 128, False), (12, 128, True)):
        cs, ns = S.cons_spec(2, C, 2, bf16=bf16), S.nc_spec(64, bf16=bf16)
        for side in (False, True):
            name = f"{n_rep}_{C}_{bf16}_{side}"
            ctx = core.Context(cons=(cs, S.cons_weights(cs, 1)), nc=(ns, S.nc_weights(ns, 2)))
            d = core.DeviceSystem([sy] * n_rep)
            x = torch.from_numpy(d.x.cpu().numpy() + rng.uniform(-0.05, 0.05, d.x.shape).astype(np.float32)).pin_memory()
            T = torch.from_numpy(rng.normal(0.0, 10.0, d.x.shape).astype(np.float32)).cuda()
            torch.cuda.synchronize()
            with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.current_stream()):
                d.x.copy_(x, non_blocking=True)
                nb, nbn = core.nbr_build(ctx, d, cs.rc + 0.8), core.nbr_build(ctx, d, ns.rc + 0.8)
                keep("list_" + name, (nb.row_ptr, nb.col, nbn.row_ptr, nbn.col))
                d.x.copy_(x, non_blocking=True)
                keep("cons_" + name, core.energy_forces_cons(ctx, d, nb, with_virial=True))
                d.x.copy_(x, non_blocking=True)
                keep("nc_" + name, core.forces_nc(ctx, d, nbn, with_virial=True))
                keep("distill_" + name, core.nc_distill_step(ctx, d, nbn, T, lr=1e-3, step=1, with_grad=True))
                keep("distill2_" + name, core.nc_distill_step(ctx, d, nbn, T, lr=1e-3, step=2, with_grad=True))
                keep("trained_" + name, core.forces_nc(ctx, d, nbn))
                keep("init_" + name, md(ctx, [sy] * n_rep, core.L.MODE_RESPA, (0,)))
                keep("step_" + name, md(ctx, [sy] * n_rep, core.L.MODE_RESPA, (1, 1)))
                keep("sts_" + name, md(ctx, [sy] * n_rep, core.L.MODE_STS, (2,)))
            torch.cuda.synchronize()
    # more rows than the distillation's SIMT contractions take, and a ragged batch
    ns = S.nc_spec(64)
    ctx = core.Context(nc=(ns, S.nc_weights(ns, 2)))
    for name, systems in (("rows", [sy] * 43), ("ragged", [S.capped_molecule_in_droplet(n, 5) for n in (20, 57, 90)])):
        d = core.DeviceSystem(systems)
        T = torch.from_numpy(rng.normal(0.0, 10.0, d.x.shape).astype(np.float32)).cuda()
        nbn = core.nbr_build(ctx, d, ns.rc + 0.8)
        keep("nc_" + name, core.forces_nc(ctx, d, nbn))
        keep("distill_" + name, core.nc_distill_step(ctx, d, nbn, T, with_grad=True))
    torch.cuda.synchronize()
    return {k: t.cpu().numpy() for k, t in out.items()}


def test_same_bits_as_without_any_overlap(tmp_path):
    ref = str(tmp_path / "ref.npz")
    env = dict(os.environ, CUDA_LAUNCH_BLOCKING="1")
    r = subprocess.run([sys.executable, os.path.abspath(__file__), ref], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    want = np.load(ref)
    for _ in range(3):
        got = collect()
        assert set(got) == set(want.files)
        wrong = [k for k in got if not np.array_equal(got[k], want[k])]
        assert not wrong, wrong
    assert all(np.isfinite(v).all() and v.size for v in got.values())


if __name__ == "__main__":
    np.savez(sys.argv[1], **collect())
