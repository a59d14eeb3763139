"""Force calls and distillation steps captured into a caller's own CUDA graph:
replays on changed inputs give the bits of direct calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,bf16", [(64, False), (128, False), (128, True)])
def test_replays_on_changed_inputs(C, bf16):
    sy = S.water_192(3)
    cs, ns = S.cons_spec(2, C, 2, bf16=bf16), S.nc_spec(64, bf16=bf16)
    ctx = core.Context(cons=(cs, S.cons_weights(cs, 1)), nc=(ns, S.nc_weights(ns, 2)))
    d = core.DeviceSystem([sy] * 3)
    nb, nbn = core.nbr_build(ctx, d, cs.rc + 0.8), core.nbr_build(ctx, d, ns.rc + 0.8)
    rng = np.random.default_rng(5)
    T = torch.from_numpy(rng.normal(0.0, 10.0, d.x.shape).astype(np.float32)).cuda()

    def calls():
        return [*core.energy_forces_cons(ctx, d, nb, with_virial=True), *core.forces_nc(ctx, d, nbn),
                *core.nc_distill_step(ctx, d, nbn, T, with_grad=True)]

    x0 = d.x.clone()
    calls()                                     # workspaces allocated
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = calls()
    for _ in range(3):
        d.x.copy_(x0 + torch.from_numpy(rng.uniform(-0.05, 0.05, x0.shape).astype(np.float32)).cuda())
        g.replay()
        got = [t.clone() for t in out]
        for a, b in zip(got, calls()):
            assert torch.equal(a, b)
    ctx.sync()
