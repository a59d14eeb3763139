"""Neighbour rows kept by the count and copied by the fill, at every length
where their sort changes (32, 64, 96, 128 entries ranked, longer ones swept
again), with a candidate set past the staging area, against all pairs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 2, 3, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 255, 256, 257]


def blob_system(n, rng, box):
    x = rng.uniform(0.0, 2.0, (n, 3)).astype(np.float32).astype(np.float64)
    return S.System("blob", x, np.zeros(n, np.uint8), np.arange(n, dtype=np.int32), np.zeros((0, 2), np.int32),
                    np.zeros(0), np.full(3, box))


@pytest.mark.parametrize("box", [0.0, 9.0, 40.0])
def test_rows_of_every_length(box):
    """Replicas whose atoms are all within the cutoff of one another: row i of
    a replica of n atoms is every other one of its atoms, ascending."""
    rng = np.random.default_rng(1)
    spec = S.nc_spec(32, rc=3.5)
    ctx = core.Context(nc=(spec, S.nc_weights(spec, 1)))
    sizes = [l + 1 for l in LENGTHS] + [2100]
    d = core.DeviceSystem([blob_system(n, rng, box) for n in sizes])
    for _ in range(2):                       # the second build reuses the scratch
        nb = core.nbr_build(ctx, d, 4.0)
        row, col = nb.row_ptr.cpu().numpy(), nb.col.cpu().numpy()
        o = 0
        for n in sizes:
            want = np.arange(o, o + n)
            for i in range(n):
                assert np.array_equal(col[row[o + i]:row[o + i + 1]], np.delete(want, i))
            o += n
        assert nb.n_pairs == row[-1]
