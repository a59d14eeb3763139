"""The distillation gradient's kernels (head adjoint over batches of 16 edges,
layer gradient from the per-species basis sums, tiled weight contractions)
against the FP64 oracle's loss: every count of tensor heads, both channel
counts, rows that leave a part of a batch, an atom without neighbours, every
species, and several slices of atoms."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

pytestmark = pytest.mark.gpu


def cluster(n, radius, seed):
    rng = np.random.default_rng(seed)
    x = []
    while len(x) < n - 1:
        p = rng.uniform(-radius, radius, 3)
        if np.linalg.norm(p) <= radius and all(np.linalg.norm(p - q) >= 1.2 for q in x):
            x.append(p)
    x = np.array(x + [[50.0, 0.0, 0.0]], np.float32).astype(np.float64)
    return S.System("cluster", x, rng.integers(0, S.N_SPECIES, n).astype(np.uint8), np.arange(n, dtype=np.int32),
                    np.zeros((0, 2), np.int32), np.zeros(0), np.zeros(3))


@pytest.mark.parametrize("C,n_l,n,radius", [(32, 1, 64, 4.0), (32, 4, 61, 4.0), (64, 2, 64, 4.0), (64, 3, 150, 6.0),
                                            (64, 2, 600, 10.5)])
def test_gradient_against_the_oracle(C, n_l, n, radius):
    """The oracle's central difference along the gradient itself is its norm
    (relative 1e-4: fp32 forces are within 1e-5, the difference's own error is
    of order h^2), and its differences in entries spread over the blocks are those
    entries (within 1e-3 of the largest)."""
    sy = cluster(n, radius, 3)
    spec = S.nc_spec(C, rc=4.0, n_l=n_l)
    blob = S.nc_weights(spec, 6)
    ctx = core.Context(nc=(spec, blob))
    F = O.nc_forces(sy, spec, blob)[0]
    T = (F + np.random.default_rng(7).normal(0.0, 5.0, F.shape)).astype(np.float32)
    d = core.DeviceSystem(sy)
    nb = core.nbr_build(ctx, d, spec.rc + 0.5)
    loss, grad = core.nc_distill_step(ctx, d, nb, T, lr=0.0, with_grad=True)
    g = grad.double().cpu().numpy()

    def L(b):
        return float(((O.nc_forces(sy, spec, b)[0] - T.astype(np.float64)) ** 2).sum())

    assert abs(loss.item() - L(blob)) <= 1e-4 * L(blob)
    norm = np.linalg.norm(g)
    h = 1e-4
    fd = (L(blob + h * g / norm) - L(blob - h * g / norm)) / (2 * h)
    assert abs(fd - norm) <= 1e-4 * norm, (fd, norm)
    if n > 200:
        return
    fitted = np.flatnonzero(g)
    for k in fitted[np.linspace(0, fitted.size - 1, 8).astype(int)]:
        e = np.zeros_like(blob)
        e[k] = h
        fd = (L(blob + e) - L(blob - e)) / (2 * h)
        assert abs(fd - g[k]) <= 1e-3 * np.abs(g).max(), (k, fd, g[k])


def test_gradient_of_an_empty_row_set():
    """No atom has a neighbour: the learned gradient is zero but for the biases' paths, none of which reach a force."""
    x = np.array([[0.0, 0, 0], [30.0, 0, 0], [0, 30.0, 0]])
    sy = S.System("gas", x, np.zeros(3, np.uint8), np.arange(3, dtype=np.int32), np.zeros((0, 2), np.int32),
                  np.zeros(0), np.zeros(3))
    spec = S.nc_spec(64, rc=4.0)
    blob = S.nc_weights(spec, 6)
    ctx = core.Context(nc=(spec, blob))
    d = core.DeviceSystem(sy)
    nb = core.nbr_build(ctx, d, spec.rc + 0.5)
    _, grad = core.nc_distill_step(ctx, d, nb, np.ones((3, 3), np.float32), lr=0.0, with_grad=True)
    assert not bool(grad.any())
