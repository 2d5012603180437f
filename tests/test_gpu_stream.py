"""The packed stream of the consecutive-lane configurations against the CSR it is made from.

The stream changes what is read, not the products or their order: configurations 9-11 (stream)
give the bits of configurations 12-14 (16-bit index over the CSR's own values) wherever both
exist, and stay within the row-sum bound of the oracle elsewhere: rows of 0, 1, 31 .. 33 and
127 .. 129 entries and long ones, and chunks of 32 entries whose columns span 65,535, 65,536 and
more (those read their columns from the CSR).
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import INDEX16_TWIN, dev, host, make_ddc, require_cuda, spmv_bound

pytestmark = pytest.mark.gpu


def _products(ddc, V, J, g, x):
    from paper_1503_01721_gb300 import api
    pi, d = torch.full((J,), float("nan"), device="cuda"), torch.full((V,), float("nan"), device="cuda")
    api.beamlet_price(ddc.h, dev(g, torch.float32), pi)
    api.dose_forward(ddc.h, dev(x, torch.float32), d)
    return host(pi), host(d)


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("cfg", [9, 10, 11])
def test_row_lengths_and_column_spans(dtype, cfg):
    require_cuda()
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(5)
    V = 200000
    rows = [np.arange(0, 3 * n, 3) for n in (0, 1, 31, 32, 33, 127, 128, 129, 1300, 5000)] * 12
    far = [np.array([0, 65535]), np.array([3, 65539]), np.concatenate([np.arange(40), 190000 + np.arange(60)])]
    rows = rows + far
    vox = np.concatenate(rows).astype(np.int32)
    blt = np.concatenate([np.full(len(r), j) for j, r in enumerate(rows)]).astype(np.int32)
    val = rng.uniform(0.05, 1.0, len(vox)).astype(np.float32)
    J = len(rows)
    g, x = synth.random_vector(V, 1), synth.random_vector(J, 2, 0.0, 1.0)
    g[[7, 190059]] = 3.0  # read through a near and a far column
    pi, d = _products(make_ddc((vox, blt, val), dtype, cfg, V, J), V, J, g, x)
    vq, _ = oracle.quantize_ddc(J, blt, val, dtype)
    D = oracle.ddc_matrix(V, J, vox, blt, vq)
    pr, dr = oracle.beamlet_price(D, g), oracle.dose_forward(D, x)
    assert np.all(np.abs(pi - pr) <= spmv_bound(abs(D).T @ np.abs(g.astype(np.float64)), np.bincount(blt, minlength=J)))
    assert np.all(np.abs(d - dr) <= spmv_bound(abs(D) @ np.abs(x.astype(np.float64)), np.bincount(vox, minlength=V)))


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
def test_same_bits_as_the_16_bit_index_and_zero_padding_is_not_read(dtype):
    require_cuda()
    c = synth.make_case("cfg1", seed=0)
    g, x = synth.random_vector(c.V, 3), synth.random_vector(c.J, 4, 0.0, 1.0)
    g[0] = np.inf  # the padding of a record points at its chunk's base, never multiplied
    for z, twin in INDEX16_TWIN.items():
        a = _products(make_ddc(c, dtype, z, brick=True), c.V, c.J, g, x)
        b = _products(make_ddc(c, dtype, twin, brick=True), c.V, c.J, g, x)
        assert all(np.array_equal(u.view(np.uint32), v.view(np.uint32)) for u, v in zip(a, b))


@pytest.mark.parametrize("K,bpc,cfg", [(1, 16, 9), (31, 8, 4), (33, 5, 9), (256, 3, 11), (257, 4, 10), (1024, 1, 9),
                                       (1025, 2, 5)])  # at most 1024 CPs: a list of the active ones
def test_rows_of_the_active_cps(K, bpc, cfg):
    """Every row of the active CPs and no other is written, with the full pass's bits."""
    require_cuda()
    from paper_1503_01721_gb300 import api
    rng = np.random.default_rng(K)
    V, J = 500, K * bpc
    blt = np.repeat(np.arange(J, dtype=np.int32), 6)
    vox = np.concatenate([np.sort(rng.choice(V, 6, replace=False)) for _ in range(J)]).astype(np.int32)
    ddc = make_ddc((vox, blt, rng.uniform(0.1, 1, len(vox)).astype(np.float32)), "f32", cfg, V, J)
    g = dev(synth.random_vector(V, 3), torch.float32)
    full = torch.empty(J, device="cuda")
    api.beamlet_price(ddc.h, g, full)
    for active in (rng.random(K) < 0.5, np.zeros(K, bool), np.ones(K, bool)):
        pi = torch.full((J,), 7.0, device="cuda")
        api.beamlet_price(ddc.h, g, pi, dev(active.astype(np.uint8), torch.uint8), bpc)
        want = np.where(np.repeat(active, bpc), host(full), np.float32(7.0))
        assert np.array_equal(host(pi).view(np.uint32), want.view(np.uint32))
