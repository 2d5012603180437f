"""CUDA graph capture of a masked D^T g pass on a handle that has only run whole passes: the
kernels of the other row numberings are loaded with the first."""
import os
import subprocess
import sys

import pytest

from gpu_util import require_cuda

pytestmark = pytest.mark.gpu

CODE = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import numpy as np, torch, synth
from gpu_util import dev, host, make_ddc
from paper_1503_01721_gb300 import api
c = synth.make_case("cfg1", seed=0)
bpc = c.mlc.n_rows * c.mlc.n_cols
ddc = make_ddc(c, {dtype!r}, {cfg}, brick=False)
g = dev(synth.random_vector(c.V, 3), torch.float32)
full = torch.empty(c.J, device="cuda")
api.beamlet_price(ddc.h, g, full)
rng = np.random.default_rng(1)
active = dev((rng.random(c.mlc.K) < 0.5).astype(np.uint8), torch.uint8)
pi = torch.full((c.J,), 7.0, device="cuda")
torch.cuda.synchronize()
graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
with torch.cuda.graph(graph, stream=s):
    api.beamlet_price(ddc.h, g, pi, active, bpc)
for _ in range(2):
    pi.fill_(7.0)
    graph.replay()
    torch.cuda.synchronize()
    want = np.where(np.repeat(host(active) != 0, bpc), host(full), np.float32(7.0))
    assert np.array_equal(host(pi).view(np.uint32), want.view(np.uint32))
print("captured")
"""


@pytest.mark.parametrize("dtype,cfg", [("f32", 9), ("bf16", 11), ("fp8", 10), ("f32", 4)])
def test_capture_after_a_whole_pass(dtype, cfg):
    require_cuda()
    import __graft_entry__
    __graft_entry__.build()
    here = os.path.dirname(os.path.abspath(__file__))
    code = CODE.format(root=os.path.dirname(here), tests=here, dtype=dtype, cfg=cfg)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)  # a process of its own: no kernel is loaded yet
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr[-2000:]
