"""Registers of the conversion kernels, as the assembler reports them: their launches count on eight blocks of 256 threads an SM, which is 32."""
import re
import subprocess

from paper_2409_16626_b200 import build as B

SR = 4


def test_encode_kernels_leave_room_for_eight_blocks_an_sm(tmp_path):
    cmd = [B.NVCC] + B.FLAGS + ["-Xptxas", "-v", "-cubin", B.CSRC + "/hif8_convert.cu", "-o", str(tmp_path / "convert.cubin")]
    report = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
    kernels = re.findall(r"Compiling entry function '\w*?convert_kernelILi(\d)ELi(\d)ELb(\d)ELb(\d)E\w*'.*?(\d+) bytes spill stores.*?Used (\d+) registers", report, re.S)
    encode = [(int(src), int(mode), int(spill), int(regs)) for src, mode, fq, amax, spill, regs in kernels if fq == "0" and amax == "0" and int(mode) != SR]
    assert len(encode) >= 3 * 4  # source formats, rounding methods
    assert [k for k in encode if k[2] or k[3] > 32] == []
