"""Registers of the conversion kernels, as the assembler reports them: their launches count on eight blocks of 256 threads an SM, which is 32, and
kernels that hold a row in registers do not hold it in memory instead."""
import re
import subprocess

from paper_2409_16626_b200 import build as B

SR = 4


def report_of(source, tmp_path):
    cmd = [B.NVCC] + B.FLAGS + ["-Xptxas", "-v", "-cubin", B.CSRC + "/" + source, "-o", str(tmp_path / "out.cubin")]
    return subprocess.run(cmd, check=True, capture_output=True, text=True).stderr


def test_encode_kernels_leave_room_for_eight_blocks_an_sm(tmp_path):
    report = report_of("hif8_convert.cu", tmp_path)
    kernels = re.findall(r"Compiling entry function '\w*?convert_kernelILi(\d)ELi(\d)ELb(\d)ELb(\d)ELb\dELb(\d)E\w*'.*?(\d+) bytes spill stores.*?Used (\d+) registers", report, re.S)
    encode = [(int(src), int(mode), int(spill), int(regs)) for src, mode, fq, amax, slots, spill, regs in kernels
              if fq == "0" and amax == "0" and slots == "0" and int(mode) != SR]
    assert len(encode) >= 3 * 4  # source formats, rounding methods
    assert [k for k in encode if k[2] or k[3] > 32] == []


def test_kernels_that_hold_a_row_spill_little(tmp_path):
    report = report_of("hif8_channel.cu", tmp_path)
    kernels = re.findall(r"Compiling entry function '\w*?row_channel_kernelILi(\d)ELi(\d)ELi(\d)E\w*'.*?(\d+) bytes spill stores", report, re.S)
    assert len(kernels) == 3 * 5 * 3  # source formats, rounding methods, forms
    assert [k for k in kernels if int(k[3]) > 48] == []
