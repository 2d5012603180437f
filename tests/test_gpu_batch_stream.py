"""Batches on handles that hold the packed stream: every plan as cg_plan runs it alone.

The batched D^T g reads the streams when every plan's matrix holds one, each plan's own form in a
mixed batch.  On this case (pencil beams in brick order) the stream is 15% ahead in the batch's own
timing of its configurations; a late launch may decide one such timing, so it is taken up to five times.
"""
import numpy as np
import pytest
import torch

import synth
from gpu_util import host, make_ddc, require_cuda
from test_gpu_cg import TIGHT, gpu_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("cfgs", [(9, 10), (11, 4)])  # both hold the stream, one of two
def test_batch_equals_single_plans(dtype, cfgs):
    require_cuda()
    import __graft_entry__
    __graft_entry__.build()
    from paper_1503_01721_gb300 import api
    n, opts = 5, api.BBOptions(**TIGHT)
    cases = [synth.make_case("cfg1", seed=s) for s in (0, 1)]
    ddcs = [make_ddc(c, dtype, cfg, brick=True) for c, cfg in zip(cases, cfgs)]
    assert [api.ddc_stream_bytes(d.h)[1] > 0 for d in ddcs] == [cfg >= 9 for cfg in cfgs]
    for _ in range(5):
        batch = api.Batch([(d.h, c.mlc, api.VoxelParams.from_numpy(c.structs), n) for d, c in zip(ddcs, cases)], opts)
        if batch.info()["spmv_cfg"] >= 9:
            break
    if cfgs == (9, 10):
        assert batch.info()["spmv_cfg"] in (9, 10, 11)
    F, _ = batch.run()
    for i, (ddc, c) in enumerate(zip(ddcs, cases)):
        F1, _, cps1, lv1, _, dose1 = gpu_plan(ddc, c, n, TIGHT)
        cps, lv = torch.empty(n, dtype=torch.int32), torch.empty(n * c.mlc.n_rows * 2, dtype=torch.int16)
        dose = torch.empty(c.V)
        batch.result(i, cps, lv, None, dose)
        assert list(cps) == list(cps1) and np.array_equal(host(lv).reshape(lv1.shape), lv1)
        assert abs(F[i] - F1) <= 1e-5 * F1
        assert np.max(np.abs(host(dose) - dose1)) <= 1e-3 * np.max(dose1)
