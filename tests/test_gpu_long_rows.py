"""Lists whose rows are longer than the count keeps (128) and than the shared
row buffer (256), from staged neighbourhoods and from ones too large to stage,
with room for 128 pairs an atom (the fill an ordinary launch) and with less (an
early one): all pairs, ascending."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,longest", [(1500, 5.0, 128), (3000, 4.6, 128), (3000, 5.6, 128), (3000, 6.0, 256)])
def test_rows_against_all_pairs(n, r, longest):
    edge = (n * 4.19 * 125 / 150) ** (1.0 / 3.0)      # 150 atoms within 5 A
    x = np.random.default_rng(3).uniform(0.0, edge, (n, 3)).astype(np.float32)

    def system(x, box):
        k = len(x)
        return S.System("s", x.astype(np.float64), np.zeros(k, np.uint8), np.arange(k, dtype=np.int32),
                        np.zeros((0, 2), np.int32), np.zeros(0), np.full(3, box))

    gas = system(np.arange(9000)[:, None] * np.float32([9.0, 0.0, 0.0]), 0.0)   # no pairs: room without long rows
    spec = S.nc_spec(32, rc=3.5)
    ctx = core.Context(nc=(spec, S.nc_weights(spec, 1)))
    d = core.DeviceSystem([system(x, edge), gas])
    wide = core.nbr_build(ctx, d, r, capacity=128 * d.n_atoms)
    assert wide.n_pairs < 128 * d.n_atoms
    tight = core.nbr_build(ctx, d, r, capacity=wide.n_pairs)
    assert torch.equal(wide.row_ptr, tight.row_ptr) and torch.equal(wide.col, tight.col)
    row, col = wide.row_ptr.cpu().numpy(), wide.col.cpu().numpy()
    assert np.diff(row).max() > longest and row[n] == row[-1]
    box = float(np.float32(edge))
    for i in range(n):
        q = x.astype(np.float64) - x[i]
        d2 = ((q - box * np.rint(q / box)) ** 2).sum(1)
        got = col[row[i]:row[i + 1]]
        assert np.all(np.diff(got) > 0) and i not in got
        sure = np.flatnonzero(d2 < r * r - 1e-4)
        assert np.isin(sure[sure != i], got).all() and (d2[got] < r * r + 1e-4).all()
