"""What the compiler reports of the kernels whose speed rests on their values staying in registers."""
import os
import re
import subprocess

from paper_2305_09887_b200 import build


def spills(source, tmp_path):
    """{kernel: bytes of spill stores} of a source file."""
    obj = os.path.join(tmp_path, "out.o")
    out = subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, source), "-o", obj],
                         check=True, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True).stdout
    return {m.group(1): int(m.group(2)) for m in
            re.finditer(r"Compiling entry function '(\w+)'[^\n]*\n[^\n]*Function properties[^\n]*\n[^\n]*?(\d+) bytes spill stores", out)}


def test_input_gradient_of_a_few_classes_does_not_spill(tmp_path):
    got = {k: v for k, v in spills("dgrad_narrow.cu", tmp_path).items() if "dgrad_narrow_kernel" in k}
    assert len(got) == 8 and not any(got.values()), got


def test_window_tiles_keep_their_epilogue_in_registers(tmp_path):
    got = {k: v for k, v in spills("spmm_tc.cu", tmp_path).items() if "spmm_dense_kernel" in k}
    assert len(got) == 3 and all(v <= 8 for v in got.values()), got


def test_gathers_with_self_loops_keep_their_rows_in_registers(tmp_path):
    got = {k: v for k, v in spills("spmm.cu", tmp_path).items() if "spmm_kernelILi2ELi2E" in k}  # 257 to 512 values
    assert len(got) == 1 and not any(got.values()), got
