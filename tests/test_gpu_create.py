"""A context is complete when it is handed out: nothing of its creation is
still running, so a first call on a stream that does not wait for the legacy
one gives the bits of any later call."""
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,n_l,bf16", [(32, 4, False), (64, 2, False), (64, 2, True)])
def test_first_call_on_a_stream_of_its_own(C, n_l, bf16):
    sy = S.water_192(3)
    spec = S.nc_spec(C, rc=3.5, n_l=n_l, bf16=bf16)
    blob = S.nc_weights(spec, 4)
    d = core.DeviceSystem(sy)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    first = []
    for _ in range(20):
        ctx = core.Context(nc=(spec, blob))
        assert torch.cuda.default_stream().query()
        with torch.cuda.stream(side):
            nb = core.nbr_build(ctx, d, spec.rc + 0.5)
            first.append(core.forces_nc(ctx, d, nb)[0])
    torch.cuda.synchronize()
    want = core.forces_nc(ctx, d, nb)[0]
    for F in first:
        assert torch.equal(F, want)
