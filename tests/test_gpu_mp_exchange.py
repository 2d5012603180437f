"""The master problem's exchange between CTAs, at the sizes where its paths change.

With at least as many CTAs as columns each CTA owns one column and polls its slots with
every thread; with fewer CTAs a warp owns a column.  The CTAs are the 256-voxel blocks of
the problem up to those that fit on the GPU; up to 4 apertures four fit on an SM, up to
44 two, then one.  Each case against the FP64 oracle's optimum from converged options, with the
bounds of the other master-problem tests (float32 products, F within 1e-4 of the optimum).
"""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import dev, host, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,n", [(1, 1), (31, 4), (257, 5),          # 1, 1 and 2 CTAs
                                 (2048, 8), (2304, 8), (2560, 9),    # 8, 9 and 10 CTAs around n + 1 columns
                                 (11520, 44), (11521, 45), (12544, 48),
                                 (77824, 4), (200000, 3),            # 304 and 608 CTAs
                                 (120000, 44), (120001, 49), (60000, 96)])
def test_master_problem_over_the_exchange_paths(V, n):
    require_cuda()
    import __graft_entry__
    from paper_1503_01721_gb300 import api
    __graft_entry__.build()
    rng = np.random.default_rng(V + n)
    DA = (rng.random((V, n)) * (rng.random((V, n)) < 0.3)).astype(np.float32)
    sid = rng.integers(0, 3, V).astype(np.uint8)
    T, wo, wu = (np.array(a, np.float32) for a in ([0.6, 0.5, 1.0], [0.05, 0.3, 1.0], [0.0, 0.0, 1.0]))
    f = lambda a, dt: torch.as_tensor(a).to("cuda", dt)
    vox = api.VoxelParams(f(sid, torch.uint8), f(T, torch.float32), f(wo, torch.float32), f(wu, torch.float32))
    y, z = torch.zeros(n, device="cuda"), torch.empty(V, device="cuda")
    DAd = dev(DA.T, torch.float32)
    rep = api.mp_bb_solve(DAd, vox, y, z, opts=api.BBOptions(2000, 1e-10, 1e-12))
    y64, DA64 = host(y).astype(np.float64), DA.astype(np.float64)
    F, _ = oracle.objective_grad(DA64 @ y64, sid, T, wo, wu)
    _, _, F_opt, _, _, _ = oracle.mp_bb_solve(DA64, sid, T, wo, wu, np.zeros(n),
                                              opts=oracle.BBOptions(max_iter=3000, rel_tol5=1e-13, step_tol=1e-14))
    floor = 1e-6 * V * 1e-3  # an optimum near 0 (fewer voxels than apertures) has no relative bound
    assert abs(rep["F"] - F) <= 1e-5 * F + floor
    if V > 256:  # below, float32 iterates can cycle short of the optimum (31 voxels, 4 apertures do)
        assert F <= F_opt * (1 + 1e-4) + floor
    # a second solve on the same buffers gives the same bits
    y2, z2 = torch.zeros(n, device="cuda"), torch.empty(V, device="cuda")
    rep2 = api.mp_bb_solve(DAd, vox, y2, z2, opts=api.BBOptions(2000, 1e-10, 1e-12))
    assert torch.equal(y, y2) and torch.equal(z, z2) and rep2 == rep
