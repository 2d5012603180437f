"""The packed stream where a handle is known to hold it (api.ddc_stream_bytes): CSR(D) rows of every
length and column span, active CPs whose rows outnumber the warps of a launch, plans with FP32
refinement, and the matrices that get no stream.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import dev, host, make_ddc, require_cuda, spmv_bound

pytestmark = pytest.mark.gpu

VB = {"f32": 4, "bf16": 2, "fp8": 1}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    require_cuda()
    import __graft_entry__
    __graft_entry__.build()


def _strided_rows(n_rows, n_cols, length, seed):
    """n_rows rows of `length` entries, columns start + step * i: (row, column, value) arrays."""
    rng = np.random.default_rng(seed)
    step = rng.integers(1, n_cols // length + 1, n_rows)
    start = (rng.random(n_rows) * (n_cols - step * (length - 1))).astype(np.int64)
    col = (start[:, None] + step[:, None] * np.arange(length)).astype(np.int32).reshape(-1)
    return (np.repeat(np.arange(n_rows, dtype=np.int32), length), col,
            rng.uniform(0.05, 1.0, n_rows * length).astype(np.float32))


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("cfg", [9, 10, 11])
def test_dose_over_row_lengths_and_column_spans(dtype, cfg):
    """CSR(D) with rows of 1 .. 5000 entries (whole records and remainders) and 32-entry chunks that
    span 65,535, 65,539 and more beamlets."""
    from paper_1503_01721_gb300 import api
    rng = np.random.default_rng(6)
    J = 200000
    rows = [np.arange(0, 3 * n, 3) for n in (1, 31, 32, 33, 127, 128, 129, 255, 256, 257, 1300, 5000)] * 12
    rows += [np.arange(j, j + 1000) for j in (10, 70000, 130001, 198000)]
    rows += [np.array([0, 65535]), np.array([3, 65539]), np.concatenate([np.arange(40), 190000 + np.arange(60)]),
             np.concatenate([np.arange(128), 190000 + np.arange(128)])]
    blt = np.concatenate(rows).astype(np.int32)
    vox = np.concatenate([np.full(len(r), i) for i, r in enumerate(rows)]).astype(np.int32)
    val = rng.uniform(0.05, 1.0, len(vox)).astype(np.float32)
    V = len(rows)
    ddc = make_ddc((vox, blt, val), dtype, cfg, V, J)
    n_rec = sum((len(r) + 127) // 128 for r in rows)
    assert api.ddc_stream_bytes(ddc.h) == (n_rec * (16 + 128 * (2 + VB[dtype])) + (V + 1) * 4, 0)
    x = synth.random_vector(J, 2, 0.0, 1.0)
    x[[65535, 65539, 190059]] = 3.0
    d = torch.full((V,), float("nan"), device="cuda")
    api.dose_forward(ddc.h, dev(x, torch.float32), d)
    vq, _ = oracle.quantize_ddc(J, blt, val, dtype)
    D = oracle.ddc_matrix(V, J, vox, blt, vq)
    err = np.abs(host(d) - oracle.dose_forward(D, x))
    assert np.all(err <= spmv_bound(abs(D) @ np.abs(x.astype(np.float64)), np.bincount(vox, minlength=V)))


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("K,bpc,length,cfg", [(60, 400, 256, 9),   # 24,000 rows: more than 20,000 warps of any launch
                                              (1000, 29, 128, 10), (1024, 32, 255, 11), (7, 3500, 383, 9)])
def test_active_cps_with_rows_beyond_a_wave(dtype, K, bpc, length, cfg):
    """Every row of the active CPs and no other is written, with the full pass's bits."""
    from paper_1503_01721_gb300 import api
    V, J = 4000, K * bpc
    blt, vox, val = _strided_rows(J, V, length, K)
    ddc = make_ddc((vox, blt, val), dtype, cfg, V, J)
    assert api.ddc_stream_bytes(ddc.h)[1] > 0
    rng = np.random.default_rng(K)
    g = synth.random_vector(V, 3)
    full = torch.empty(J, device="cuda")
    api.beamlet_price(ddc.h, dev(g, torch.float32), full)
    vq, _ = oracle.quantize_ddc(J, blt, val, dtype)
    D = oracle.ddc_matrix(V, J, vox, blt, vq)
    err = np.abs(host(full) - oracle.beamlet_price(D, g))
    assert np.all(err <= spmv_bound(abs(D).T @ np.abs(g.astype(np.float64)), np.full(J, length)))
    last = np.zeros(K, bool)
    last[-1] = True
    for active in (rng.random(K) < 0.5, np.zeros(K, bool), np.ones(K, bool), last):
        pi = torch.full((J,), 7.0, device="cuda")
        api.beamlet_price(ddc.h, dev(g, torch.float32), pi, dev(active.astype(np.uint8), torch.uint8), bpc)
        want = np.where(np.repeat(active, bpc), host(full), np.float32(7.0))
        assert np.array_equal(host(pi).view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("cfg", [9, 10, 11])
def test_windows_with_empty_segments(dtype, cfg):
    """The rows inside the leaf-travel windows have the full pass's bits, with windows that end in
    mid run, empty ones between and after them, and more rows than a launch has warps."""
    from paper_1503_01721_gb300 import api
    from types import SimpleNamespace
    K, nr, nc, length, V = 50, 40, 37, 256, 4000
    J = K * nr * nc
    mlc = SimpleNamespace(K=K, n_rows=nr, n_cols=nc, arc_first_cp=np.array([0], np.int32), travel_cols=2,
                          interdigitation=False, machine=None)
    blt, vox, val = _strided_rows(J, V, length, 8)
    ddc = make_ddc((vox, blt, val), dtype, cfg, V, J)
    assert api.ddc_stream_bytes(ddc.h)[1] > 0
    rng = np.random.default_rng(9)
    occ = (rng.random(K) < 0.2).astype(np.uint8)
    occ[[0, K - 1]] = 1  # the list ends with segments without a row
    lv = np.sort(rng.integers(0, nc + 1, (K, nr, 2)), -1).astype(np.int16)
    g = dev(synth.random_vector(V, 3), torch.float32)
    full, pi = torch.empty(J, device="cuda"), torch.full((J,), 7.0, device="cuda")
    api.beamlet_price(ddc.h, g, full)
    api.beamlet_price_windowed(ddc.h, mlc, dev(occ, torch.uint8), dev(lv, torch.int16), g, pi)
    need = np.zeros((K, nr, nc), bool)  # a leaf moves 2 columns per CP from each occupied neighbour
    at = np.flatnonzero(occ)
    for k in np.flatnonzero(occ == 0):
        near = [q for q in (at[at < k].max(initial=-1), at[at > k].min(initial=K)) if 0 <= q < K]
        for r in range(nr):
            lo = max([0] + [int(lv[q, r, 0]) - 2 * abs(k - q) for q in near])
            hi = min([nc] + [int(lv[q, r, 1]) + 2 * abs(k - q) for q in near])
            need[k, r, lo:max(lo, hi)] = True
    need = need.reshape(-1)
    assert need.sum() > 20000
    want = np.where(need, host(full), np.float32(7.0))
    assert np.array_equal(host(pi).view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
def test_refined_plan_reads_the_float32_values(dtype):
    """FP32 refinement on a handle whose CSR(D) holds a stream of the stored values: the final dose
    is the float32 matrix's (1e-5; the stored values are off by 2^-9 and more)."""
    from paper_1503_01721_gb300 import api
    from test_gpu_cg import TIGHT, gpu_plan
    c = synth.make_case("cfg1", seed=0)
    ddc = make_ddc(c, dtype=dtype, tile_cfg=9, refine=True, brick=True)
    assert min(api.ddc_stream_bytes(ddc.h)) > 0
    F, st, cps, lv, y, dose = gpu_plan(ddc, c, 6, TIGHT)
    assert st["refined"] == 1
    d_ref = oracle.dose_forward(oracle.ddc_matrix(c.V, c.J, c.vox, c.blt, c.val), oracle.aperture_fluence(c.mlc, cps, lv, y))
    assert np.max(np.abs(dose - d_ref)) <= 1e-5 * np.max(np.abs(d_ref))
    # the same apertures as on a handle without a stream
    plain = make_ddc(c, dtype=dtype, tile_cfg=4, refine=True, brick=True)
    assert api.ddc_stream_bytes(plain.h) == (0, 0)
    assert list(gpu_plan(plain, c, 6, TIGHT)[2]) == list(cps)


@pytest.mark.parametrize("rows,why", [([np.arange(0, 60, 10)] * 400, "short rows: records would be padding"),
                                      ([np.arange(128) * 2200] * 200, "far columns: chunks span 65,536 and more")])
def test_a_refused_stream_leaves_the_csr(rows, why):
    from paper_1503_01721_gb300 import api
    V, J = 300000, len(rows)
    vox = np.concatenate(rows).astype(np.int32)
    blt = np.concatenate([np.full(len(r), j) for j, r in enumerate(rows)]).astype(np.int32)
    val = np.random.default_rng(3).uniform(0.05, 1.0, len(vox)).astype(np.float32)
    g = synth.random_vector(V, 1)
    out = []
    for cfg in (9, 4):
        ddc = make_ddc((vox, blt, val), "f32", cfg, V, J)
        assert api.ddc_stream_bytes(ddc.h)[1] == 0, why
        pi = torch.empty(J, device="cuda")
        api.beamlet_price(ddc.h, dev(g, torch.float32), pi)
        out.append(host(pi))
    D = oracle.ddc_matrix(V, J, vox, blt, val)
    bound = spmv_bound(abs(D).T @ np.abs(g.astype(np.float64)), np.bincount(blt, minlength=J))
    for pi in out:
        assert np.all(np.abs(pi - oracle.beamlet_price(D, g)) <= bound)


def test_the_stream_gives_way_when_memory_is_short():
    """With less than half of the device's memory left a build takes no stream, and its products are
    the CSR's: the stream is optional, what a later build or plan allocates is not."""
    from paper_1503_01721_gb300 import api
    c = synth.make_case("cfg1", seed=0)
    g = dev(synth.random_vector(c.V, 1), torch.float32)
    out = []
    _, total = torch.cuda.mem_get_info()
    for held in (int(0.55 * total), 0):
        block = torch.empty(held, dtype=torch.uint8, device="cuda")
        for kw in ({"tile_cfg": 9}, {"autotune": True}):
            ddc = api.Ddc(c.V, c.J, dev(c.vox, torch.int32), dev(c.blt, torch.int32), dev(c.val, torch.float32),
                          dtype="bf16", **kw)
            bytes_ = api.ddc_stream_bytes(ddc.h)
            assert bytes_ == (0, 0) if held else bytes_[1] > 0 or "autotune" in kw
            if "tile_cfg" in kw:
                pi = torch.empty(c.J, device="cuda")
                api.beamlet_price(ddc.h, g, pi)
                out.append(host(pi))
            ddc.close()
        del block
        torch.cuda.empty_cache()
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))


def test_which_passes_read_a_stream():
    from paper_1503_01721_gb300 import api
    c = synth.make_case("cfg1", seed=0)

    def reads(**kw):
        ddc = make_ddc(c, "bf16", **kw)
        return api.ddc_stream_reads(ddc.h)
    assert reads(tile_cfg=9) == {"D": True, "Dt": True, "windows": True}
    assert reads(tile_cfg=4) == {"D": False, "Dt": False, "windows": False}
    assert reads(tile_cfg=12, index16=True) == {"D": False, "Dt": False, "windows": False}
