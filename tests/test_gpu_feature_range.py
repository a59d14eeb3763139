"""Row and channel scales of the tensor-core layers, with features spread over
decades: a model whose channels are held in other units is the same model, and
neighbours whose features differ by decades still add up within the split-bf16
bar. Rows beyond the 96 candidates in flight are among them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from helpers import TOL_BF16_RMS
from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S
from test_gpu_first_layer import ball

pytestmark = pytest.mark.gpu
C, L = 128, 3


def blocks(spec, blob):
    """Views of the blob: emb, per layer (wrad, W1, b1, W2, b2), Wr, br, wo."""
    nl, o = spec.lmax + 1, 0

    def take(*shape):
        nonlocal o
        n = int(np.prod(shape))
        o += n
        return blob[o - n:o].reshape(shape)

    emb = take(spec.n_species, C)
    layers = [(take(nl, spec.K, C), take(C, nl * C), take(C), take(C, C), take(C)) for _ in range(L)]
    return emb, layers, take(C, C), take(C), take(C)


def forces(spec, blob, sy):
    ctx = core.Context(cons=(spec, blob))
    d = core.DeviceSystem(sy)
    nb = core.nbr_build(ctx, d, spec.rc + 0.5)
    F = core.energy_forces_cons(ctx, d, nb, with_prior=False)[1]
    ctx.sync()
    return F, int(np.diff(nb.row_ptr.cpu().numpy()).max())


@pytest.mark.parametrize("decades", [4, 12])
@pytest.mark.parametrize("lmax", [0, 1, 2])
def test_channels_in_other_units(lmax, decades):
    """s_c times 2^e_c and the weights that read it divided by that: every
    product is the same up to exact powers of two, so the forces are the same
    bits. One channel is read by nothing."""
    spec = S.cons_spec(L, C, lmax, bf16=True)
    blob = S.cons_weights(spec, 8)
    for wrad, W1, _, _, _ in blocks(spec, blob)[1]:
        wrad[:, :, 5] = 0.0
    sy = ball(150, 5.2, 3)
    want, longest = forces(spec, blob, sy)
    assert longest > 96
    e = np.round(np.random.default_rng(9).uniform(-0.5, 0.5, C) * decades * np.log2(10.0))
    f = 2.0 ** e
    emb, layers, Wr, _, _ = blocks(spec, blob)
    emb *= f
    for wrad, _, _, W2, b2 in layers:
        wrad /= f
        W2 *= f[:, None]
        b2 *= f
    Wr /= f
    got, _ = forces(spec, blob, sy)
    assert torch.equal(got, want)


@pytest.mark.parametrize("decades", [4, 8])
@pytest.mark.parametrize("lmax", [1, 2])
def test_neighbours_decades_apart(lmax, decades):
    """Species whose features differ by up to `decades` decades (the layers'
    updates as small as the smallest; the energy scaled up so that the forces
    stay far above the fixed-point unit)."""
    spec = S.cons_spec(L, C, lmax, bf16=True, scale=1e-2 * 10.0 ** decades)
    blob = S.cons_weights(spec, 8)
    emb, layers, _, _, _ = blocks(spec, blob)
    emb *= 10.0 ** (-decades * np.array([1.0, 0.5, 0.25, 0.0, 0.75]))[:, None]
    for _, _, _, W2, _ in layers:
        W2 *= 10.0 ** -decades
    blob = blob.astype(np.float32).astype(np.float64)
    for sy in (S.water_192(3), S.capped_molecule_in_droplet(40, 5), ball(110, 5.2, 4)):
        F, _ = forces(spec, blob, sy)
        _, Fo = O.cons_energy_forces(sy, spec, blob)
        assert np.abs(F.cpu().numpy() - Fo).max() <= TOL_BF16_RMS * np.sqrt((Fo ** 2).mean())
