"""Power-of-two scaling by the exponent field (PrecF64::scale2) against the product, bit for bit:
zeros, subnormals, the smallest normals, values whose result is subnormal, the largest finite values,
infinities, NaN, of both signs, at every factor that the transforms use, and 2^20 random bit patterns
(tests/scale2_check.cu).  On the CPU the same table through a model of the exponent arithmetic."""
import os
import shutil
import struct
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1501_04552_gb300", "csrc")
FACTORS = [-1] + [-3 * k for k in range(4, 10)]      # one half, 1/N^3 for N = 16 .. 512


def table():
    bits = [0, 1, 2, 3, 0x7FFFFFFFFFFFF, 0x8000000000000, 0xFFFFFFFFFFFFF,             # zero, subnormals
            0x7FEFFFFFFFFFFFFF, 0x7FE0000000000000, 0x7FDFFFFFFFFFFFFF,                # largest finite values
            0x7FF0000000000000, 0x7FF0000000000001, 0x7FF8000000000000, 0x7FFFFFFFFFFFFFFF,
            0x3FF0000000000000, 0x3FEFFFFFFFFFFFFF]
    for e in range(1, 40):                           # around the smallest normals: results that are subnormal
        bits += [(e << 52) | m for m in (0, 1, 0x8000000000001, 0xFFFFFFFFFFFFF)]
    return [(b | s, p) for p in FACTORS for b in bits for s in (0, 1 << 63)]


def model(bits, p):
    """the field arithmetic of scale2 in 32-bit words; None where it multiplies"""
    hi, m32 = bits >> 32, 0xFFFFFFFF
    d = ((struct.unpack("<Q", struct.pack("<d", 2.0 ** p))[0] >> 32) - 0x3FF00000) & m32
    e = hi & 0x7FF00000
    f = (e + d) & m32
    if (e - 0x00100000) & m32 < 0x7FE00000 and (f - 0x00100000) & m32 < 0x7FE00000:
        return (((hi + d) & m32) << 32) | (bits & m32)
    return None


def test_field_arithmetic_is_the_product():
    taken = 0
    for bits, p in table():
        got = model(bits, p)
        if got is not None:
            x = struct.unpack("<d", struct.pack("<Q", bits))[0]
            assert got == struct.unpack("<Q", struct.pack("<d", x * 2.0 ** p))[0], (hex(bits), p)
            taken += 1
    assert taken > len(table()) // 3


@pytest.mark.gpu
def test_scale2_is_the_product(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "scale2_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC,
                    "-o", exe, os.path.join(HERE, "scale2_check.cu")], check=True)
    rows = table()
    out = subprocess.run([exe], input="".join("%x %d\n" % r for r in rows), check=True, capture_output=True, text=True).stdout
    words = out.split("\n")[-2].split()
    assert int(words[1]) == len(rows) + (1 << 20)
    assert int(words[3]) == 0, out
    assert int(words[5]) > (1 << 19)      # subnormal inputs and results among them are not flushed
