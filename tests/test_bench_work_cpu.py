"""The per-kernel work bench.py rates its profile by: the kernels' own loops,
counted here a second time by walking them."""
import dataclasses
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
from paper_2602_14975_gb300 import synth as S  # noqa: E402


def adjoint_fma_per_channel(lmax, K):
    """(pair, lower neighbour): the multiply-adds (or lone products) of k_mp_bwd's
    two loops for one channel."""
    pair = lower = 0
    for l in range(lmax + 1):
        pair += 2 * K          # R and R'
        lower += K             # R
        for _ in range(2 * l + 1):
            pair += 2 + 1 + 1 + 1      # Gam (two), its sum with Y, beta, the sender sum with Y
            lower += 1
        pair += 1 + 1          # rho, sender role
        lower += 1
    return pair, lower


@pytest.mark.parametrize("C,lmax,bf16", [(128, 2, True), (128, 2, False), (64, 1, True), (64, 1, False), (128, 0, True)])
def test_work_of_the_layers(C, lmax, bf16):
    cs, ns = S.cons_spec(3, C, lmax, bf16=bf16), S.nc_spec(64, bf16=bf16)
    w = bench.kernel_work(cs, ns)
    nlm, K, nl = (lmax + 1) ** 2, cs.K, lmax + 1
    assert w["first_fwd"]["edge"] == sum(2 * K for _ in range(nlm))
    assert w["nc_mp_fwd"]["edge"] == 2 * K * 4
    pair, lower = adjoint_fma_per_channel(lmax, K)
    assert w["mp_bwd"]["edge"] == pytest.approx(2 * (pair + lower) * C / 2 + 51 * 16 + 46.5)
    if bf16 and C == 128:
        blocks = -(-nlm * K // 16)
        assert w["mp_fwd"]["tensor_edge"] == w["mp_fwd"]["edge"] == 3 * 2 * 16 * blocks * C
    else:
        assert w["mp_fwd"]["tensor_edge"] == 0
        assert w["mp_fwd"]["edge"] == 2 * C * sum(K + 1 + 2 * l + 1 for l in range(nl))


def test_no_layer_is_counted_that_a_kernel_does_not_run():
    """One launch of a later layer's kernel is the same work in a model of any
    depth: the first layer has rows of its own."""
    ns = S.nc_spec(64, bf16=True)
    a, b = (bench.kernel_work(S.cons_spec(L, 128, 2, bf16=True), ns) for L in (2, 4))
    assert a == b and set(a) == {"first_fwd", "first_bwd", "nc_mp_fwd", "mp_fwd", "mp_bwd"}
    few = bench.kernel_work(dataclasses.replace(S.cons_spec(2, 128, 2, bf16=True), n_species=2), ns)
    assert few["first_fwd"]["atom"] < a["first_fwd"]["atom"] and few["first_fwd"]["edge"] == a["first_fwd"]["edge"]


def test_factored_layer_is_far_below_the_unfactored_count():
    w = bench.kernel_work(S.cons_spec(3, 128, 2, bf16=True), S.nc_spec(64, bf16=True))
    assert w["first_fwd"]["edge"] * 50 < 2 * (8 * 3 + 9) * 128
    assert w["nc_mp_fwd"]["edge"] * 30 < 2 * (8 * 2 + 2 + 4) * 64
