"""The warp-row kernels of the packed stream keep their registers: compiled for sm_103a, the
variants that hold 64 warps per SM (32 registers) and the 40-register one spill nothing to local
memory, in any numbering of the rows and value type (ptxas prints it; no GPU needed)."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def ptxas_lines(tmp_path_factory):
    from paper_1503_01721_gb300 import build
    out = tmp_path_factory.mktemp("spmv") / "spmv.o"
    cmd = [build.nvcc()] + build.NVCC_FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, "spmv.cu"), "-o", str(out)]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("nvcc is not here")
    assert r.returncode == 0, r.stderr
    return r.stderr


def _spills(text, kernel):
    """(entry, bytes of spill stores, bytes of spill loads) of every entry whose name holds `kernel`."""
    found = re.findall(r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", text,
                       flags=re.S)
    return [(name, int(st), int(ld)) for name, st, ld in found if kernel in name]


def test_stream_kernels_spill_nothing(ptxas_lines):
    entries = _spills(ptxas_lines, "spmv_warp_row_x_kernel")
    assert len(entries) >= 9
    assert [e for e in entries if e[1] or e[2]] == []


def test_batched_stream_kernels_spill_nothing(ptxas_lines):
    """Batches whose plans all hold the stream (BF16 at 512 threads apart, which spills a little for
    twice the warps)."""
    entries = [e for e in _spills(ptxas_lines, "spmv_rows_batched_kernel") if "BatchFormE2E" in e[0]]
    assert len(entries) == 9
    assert len([e for e in entries if e[1] or e[2]]) <= 1
    assert [e for e in entries if (e[1] or e[2]) and not ("Li512ELi4E" in e[0] and "bfloat16" in e[0])] == []
