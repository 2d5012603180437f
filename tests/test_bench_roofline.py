"""What the benchmark says about a pass that reads the packed stream: the kernel that ran and the bytes
that moved (no GPU needed)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _kernels(function):
    """{configuration: template arguments} of a dispatch function of csrc/spmv.cu, and the function's text."""
    src = open(os.path.join(ROOT, "paper_1503_01721_gb300", "csrc", "spmv.cu")).read()
    body = src[src.index(f"RowFn {function}(int cfg) {{"):]
    body = body[:body.index("\n}\n")]
    return {int(c): (k, f"<{t},{u}>") for c, k, t, u in
            re.findall(r"case (\d+): return (\w+)<NUM, (\d+), (\d+), VT>;", body)}, body


def test_kernel_names_are_the_library_s():
    import bench
    csr, body = _kernels("row_kernel_for")
    assert "default: return spmv_warp_row_kernel<NUM, 512, 4, VT>;" in body
    csr[6] = ("spmv_warp_row_kernel", "<512,4>")
    assert {c: k + a for c, (k, a) in csr.items()} == {c: bench.SPMV_KERNELS[c] for c in range(4, 15)}
    strm, body = _kernels("stream_kernel_for")
    assert "default: return spmv_warp_row_x_kernel<NUM, 512, 4, VT>;" in body
    strm[11] = ("spmv_warp_row_x_kernel", "<512,4>")
    assert {c: k + a for c, (k, a) in strm.items()} == bench.STREAM_KERNELS


def test_stream_pass_moves_its_records():
    from paper_1503_01721_gb300 import roofline
    rows, n = 1000, 1313  # 11 records a row
    for dtype, rec in (("f32", 784), ("bf16", 528), ("fp8", 400)):
        csr = roofline.spmv_bytes(rows * n, rows, 5000, rows, dtype)
        moved = roofline.stream_bytes(rows * 11 * rec + 4 * (rows + 1), rows, 5000, rows)
        assert moved == rows * 11 * rec + 12 * (rows + 1) + 4 * 5000 + 4 * rows
        assert moved < 0.85 * csr  # a rate over the CSR's bytes is no fraction of a peak
