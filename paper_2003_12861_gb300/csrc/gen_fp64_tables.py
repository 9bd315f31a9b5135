"""Generate fp64_tables.h: tables of the generic event kernel's FP64
functions (fp64_math.cuh), computed from the mathematics with mpmath at 50
digits.

* 2^(j/256), j = 0..255, as a double and the rounded rest, and the degree-4
  Chebyshev economisation of (e^r - 1 - r) / r^2 on |r| <= ln2/512
  (table-driven reduction of P. T. P. Tang, ACM TOMS 15 (1989)).
* erfc about the points -7, -6 7/8, ..., 0 and erfcx(z) = exp(z^2) erfc(z)
  about 0, 1/8, ..., 8: per point the degree-10 Chebyshev interpolant on
  +-1/16 in monomials of the distance.

Run: python paper_2003_12861_gb300/csrc/gen_fp64_tables.py
"""
import os

import mpmath as mp

mp.mp.dps = 50
HERE = os.path.dirname(os.path.abspath(__file__))


def interpolant(f, half, n):
    """Monomials of the degree-n Chebyshev interpolant of f on [-half, half]."""
    N = n + 1
    xs = [mp.cos(mp.pi * (k + mp.mpf(1) / 2) / N) for k in range(N)]
    fx = [f(half * x) for x in xs]
    c = [2 * mp.fsum(fx[k] * mp.cos(mp.pi * j * (k + mp.mpf(1) / 2) / N) for k in range(N)) / N for j in range(N)]
    c[0] /= 2
    T = [[mp.mpf(0)] * N for _ in range(N)]
    T[0][0] = mp.mpf(1)
    if N > 1:
        T[1][1] = mp.mpf(1)
    for k in range(2, N):
        for j in range(N):
            T[k][j] = (2 * T[k - 1][j - 1] if j > 0 else 0) - T[k - 2][j]
    return [mp.fsum(c[k] * T[k][j] for k in range(N)) / half ** j for j in range(N)]


def hexf(x):
    return float(x).hex()


def main():
    out = ["// Generated by gen_fp64_tables.py from the mathematics (mpmath, 50 digits). Do not edit.", "#pragma once",
           "namespace rf {"]
    half = mp.log(2) / 512
    c = interpolant(lambda r: mp.mpf(1) / 2 + r / 6 + r * r / 24 + r ** 3 / 120 + r ** 4 / 720 + r ** 5 / 5040, half, 2)
    out.append("constexpr double kExp64_2 = %s, kExp64_3 = %s, kExp64_4 = %s;" % tuple(map(hexf, c)))
    step = mp.log(2) / 256
    # 34 significant bits: its product with |k| < 2^19 is exact
    e = mp.floor(mp.log(step, 2))
    c1 = float(mp.nint(step / mp.mpf(2) ** (e - 33)) * mp.mpf(2) ** (e - 33))
    out.append("constexpr double kExp64_K = %s, kExp64_C1 = %s, kExp64_C2 = %s;" % (hexf(1 / step), c1.hex(), hexf(step - mp.mpf(c1))))
    v = []
    for j in range(256):
        t = mp.mpf(2) ** (mp.mpf(j) / 256)
        v += [hexf(t), hexf(t - mp.mpf(float(t)))]
    out.append("static __device__ __align__(16) const double kExp64[512] = {" + ",".join(v) + "};")
    rows = []
    for i in range(-56, 1):
        rows.append(interpolant(lambda d: mp.erfc(mp.mpf(i) / 8 + d), mp.mpf(1) / 16, 10))
    for i in range(0, 65):
        rows.append(interpolant(lambda d: mp.exp((mp.mpf(i) / 8 + d) ** 2) * mp.erfc(mp.mpf(i) / 8 + d), mp.mpf(1) / 16, 10))
    out.append("constexpr int kTailRow = 12;  // doubles a row: 11 coefficients and the rounded rest of the first")
    out.append("static __device__ __align__(16) const double kTail64[%d] = {" % (12 * len(rows)) +
               ",".join(",".join(map(hexf, r + [r[0] - mp.mpf(float(r[0]))])) for r in rows) + "};")
    out.append("}  // namespace rf")
    with open(os.path.join(HERE, "fp64_tables.h"), "w") as fh:
        fh.write("\n".join(out) + "\n")


if __name__ == "__main__":
    main()
