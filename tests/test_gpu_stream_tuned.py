"""Autotuned handles beside the packed stream: what the tuner keeps is what it reads, and whatever it chose,
the products have the bits of the same configurations built outright."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import dev, host, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("case,brick", [("cfg1", True), ("cfg1", False), ("ragged", True), ("tiny", False)])
def test_tuned_handle(dtype, case, brick):
    require_cuda()
    import __graft_entry__
    __graft_entry__.build()
    from paper_1503_01721_gb300 import api
    c = synth.make_case(case, seed=0)
    grid = (c.geom.nx, c.geom.ny, c.geom.nz) if brick else None
    coo = [dev(c.vox, torch.int32), dev(c.blt, torch.int32), dev(c.val, torch.float32)]
    tuned = api.Ddc(c.V, c.J, *coo, dtype=dtype, autotune=True, vox_grid=grid)
    info = tuned.info()
    if api.ddc_stream_bytes(tuned.h)[0]:  # CSR(D)'s stream is kept only to be read
        assert info["cfg_D"] in (9, 10, 11)
    fixed = api.Ddc(c.V, c.J, *coo, dtype=dtype, tile_cfg=info["cfg_D"], tile_cfg_Dt=info["cfg_Dt"], vox_grid=grid)
    g, x = dev(synth.random_vector(c.V, 3), torch.float32), dev(synth.random_vector(c.J, 4, 0.0, 1.0), torch.float32)
    out = []
    for h in (tuned.h, fixed.h):
        pi, d = torch.empty(c.J, device="cuda"), torch.empty(c.V, device="cuda")
        api.beamlet_price(h, g, pi)
        api.dose_forward(h, x, d)
        out.append((host(pi), host(d)))
    assert all(np.array_equal(a.view(np.uint32), b.view(np.uint32)) for a, b in zip(*out))
    # a plan (windowed passes, in the configuration and form timed for them) and a batch on the tuned handle
    vox = api.VoxelParams.from_numpy(c.structs)
    F, st = api.cg_plan(tuned.h, c.mlc, vox, 2)
    batch = api.Batch([(tuned.h, c.mlc, vox, 2)] * 2)
    Fb, _ = batch.run()
    assert st["n_apertures"] == 2 and all(abs(f - F) <= 1e-4 * F for f in Fb)
