"""Write drt_fftrig.h: sin and cos of i / 32, i = 0..205, each as two FP32 numbers (high, low), from their power series in
60-digit decimal arithmetic.

  python paper_2205_00237_gb300/csrc/gen_fftrig.py     # rewrites drt_fftrig.h beside this script
"""
import os
import struct
from decimal import Decimal as D, getcontext

getcontext().prec = 60
N = 206


def sincos(x):
    s, c, term, k = D(0), D(0), D(1), 0
    while abs(term) > D(10) ** -55 or k < 4:
        if k % 2 == 0:
            c += term if k % 4 == 0 else -term
        else:
            s += term if k % 4 == 1 else -term
        k += 1
        term = term * x / k
    return s, c


def two(x):
    f32 = lambda v: struct.unpack("<f", struct.pack("<f", float(v)))[0]   # noqa: E731
    h = f32(x)
    return "%sf, %sf" % (h.hex(), f32(x - D(h)).hex())


def main():
    src = ("// Generated by gen_fftrig.py: sin and cos of i / 32, i = 0..205, as (sin high, sin low, cos high, cos low).\n"
           "#pragma once\n\nnamespace drt {\n\nstatic __device__ const float4 kFFTrig[%d] = {\n" % N)
    for i in range(N):
        s, c = sincos(D(i) / 32)
        src += "    {%s, %s},\n" % (two(s), two(c))
    src += "};\n\n}  // namespace drt\n"
    with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "drt_fftrig.h"), "w") as f:
        f.write(src)


if __name__ == "__main__":
    main()
