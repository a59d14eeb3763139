"""Kernels scheduled before their predecessor has ended: back-to-back calls whose
inputs change in between, without a wait, give the bits of calls that are waited
for one by one, on the default stream and on another, for a size of one wave and
one of several."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [False, True])
@pytest.mark.parametrize("n_rep,C,bf16", [(1, 64, False), (1, 128, True), (12, 128, False), (12, 128, True)])
def test_back_to_back_calls(n_rep, C, bf16, side):
    sy = S.water_192(3)
    cs, ns = S.cons_spec(2, C, 2, bf16=bf16), S.nc_spec(64)
    ctx = core.Context(cons=(cs, S.cons_weights(cs, 1)), nc=(ns, S.nc_weights(ns, 2)))
    d = core.DeviceSystem([sy] * n_rep)
    nb, nbn = core.nbr_build(ctx, d, cs.rc + 0.8), core.nbr_build(ctx, d, ns.rc + 0.8)
    rng = np.random.default_rng(5)
    x0 = d.x.clone()
    dx = [torch.from_numpy(rng.uniform(-0.05, 0.05, x0.shape).astype(np.float32)).cuda() for _ in range(6)]
    st = torch.cuda.Stream() if side else torch.cuda.current_stream()
    torch.cuda.synchronize()

    def calls(wait):
        out = []
        with torch.cuda.stream(st):
            for e in dx:
                torch.add(x0, e, out=d.x)
                E, F = core.energy_forces_cons(ctx, d, nb)
                if wait:
                    torch.cuda.synchronize()
                Fn, net = core.forces_nc(ctx, d, nbn)
                if wait:
                    torch.cuda.synchronize()
                out += [E, F, Fn]
        torch.cuda.synchronize()
        return out

    ref = calls(True)
    for _ in range(3):
        for a, b in zip(calls(False), ref):
            assert torch.equal(a, b)
