"""Device memory a conservative evaluation takes, against the arrays it needs."""
import ctypes as ct

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu
MB = 1 << 20
ROUNDING = 64 * MB     # some thirty allocations of 2 MB granularity


def growth(spec, n):
    """Device memory taken by the first evaluation of n atoms that have no
    neighbours (the outputs exist already)."""
    ctx = core.Context(cons=(spec, S.cons_weights(spec, 3)))
    one = S.System("one", np.zeros((1, 3)), np.zeros(1, np.uint8), np.zeros(1, np.int32), np.zeros((0, 2), np.int32),
                   np.zeros(0), np.zeros(3))
    d = core.DeviceSystem(one)
    nb = core.nbr_build(ctx, d, spec.rc + 0.5)
    core.energy_forces_cons(ctx, d, nb)      # kernels loaded
    ctx.sync()
    i32 = dict(dtype=torch.int32, device="cuda")
    d.n_atoms = n
    d.x = torch.zeros(n, 3, device="cuda")
    d.species = torch.zeros(n, dtype=torch.uint8, device="cuda")
    d.mol_id, d.bond_ptr = torch.arange(n, **i32), torch.zeros(n + 1, **i32)
    d.rep_off = torch.tensor([0, n], **i32)
    nb = core.NbrList(torch.zeros(n + 1, **i32), torch.zeros(1, **i32), spec.rc + 0.5)
    E, F = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty(n, 3, device="cuda")
    s, l = d.struct(), nb.struct()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    st = ctx.lib.energy_forces_cons(ctx.handle, ct.byref(s), ct.byref(l), E.data_ptr(), F.data_ptr(), None, 0,
                                    torch.cuda.current_stream().cuda_stream)
    assert st == core.L.OK
    ctx.sync()
    taken = before - torch.cuda.mem_get_info()[0]
    fp = core.replica_footprint(ctx, n)
    ctx.close()
    torch.cuda.empty_cache()
    return taken, fp


def test_features_of_the_layers_only():
    """One layer, l_max = 0: its output features, A, q, the pre-activations and
    five MLP and gradient arrays, [n][C] floats each; 10 words per atom besides
    (energy, forces before the prior, fixed-point sums) and the replica map."""
    n, C = 1_000_000, 128
    taken, _ = growth(S.cons_spec(1, C, 0), n)
    assert taken <= n * (4 * C * 9 + 44) + ROUNDING


@pytest.mark.parametrize("C,L,lmax,bf16", [(128, 3, 2, True), (128, 1, 1, True), (64, 2, 1, True), (128, 2, 0, False)])
def test_admission_counts_what_is_allocated(C, L, lmax, bf16):
    """The serving loop's count per replica, less its share of state and lists
    (85 bytes and 288 list words per atom), covers what an evaluation takes and
    exceeds it by no more than the one array it allows for words per atom."""
    n = 1_000_000
    taken, fp = growth(S.cons_spec(L, C, lmax, bf16=bf16), n)
    counted = fp - n * (85 + 4 * 288)
    assert taken <= counted + ROUNDING
    assert counted <= taken + n * 4 * C + ROUNDING
