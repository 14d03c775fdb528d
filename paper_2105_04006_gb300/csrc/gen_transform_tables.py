"""Constant tables of the transform kernels, written at build time.

Usage: python gen_transform_tables.py OUT.inc

The transform evaluates the trig sums of a run of bins by spreading the
observations onto a uniform periodic grid of twice as many cells with a
Kaiser-Bessel window psi, an FFT, and a division by psi's Fourier transform
(the nonuniform FFT of Dutt & Rokhlin 1993 with the window of Jackson et al.
1991):

  psi(x) = I0(beta sqrt(1 - (2x/w)^2)) / I0(beta),  |x| <= w/2,
  psi^(xi) = w / I0(beta) sinh(s) / s,  s = sqrt(beta^2 - (pi w xi)^2).

The aliasing error at offset xi, sqrt(sum_{p != 0} psi^(xi + p)^2) / psi^(xi),
is at most 1.6e-7 at the edge of the run and 5e-8 rms (w = 8, the FP32
kernels) and 4.8e-15 and 1.1e-15 (w = 16, FP64) for |xi| <= 1/4, beta being
the minimiser of the former.
"""
import math
import sys


def i0(x):
    term, total, k = 1.0, 1.0, 1
    while term > 1e-18 * total:
        term *= (x / (2.0 * k)) ** 2
        total += term
        k += 1
    return total


def psi(x, w, beta):
    z = 1.0 - (2.0 * x / w) ** 2
    return i0(beta * math.sqrt(z)) / i0(beta) if z >= 0.0 else 0.0


def psi_hat(xi, w, beta):
    s = math.sqrt(beta * beta - (math.pi * w * xi) ** 2)
    return w / i0(beta) * math.sinh(s) / s


def window_polys(w, beta, deg):
    """Row r: monomial coefficients in u = frac - 1/2 of psi(r - (w/2 - 1) - frac), 0 <= frac < 1,
    from the Chebyshev interpolant at 64 nodes cut to degree deg."""
    n = 64
    rows = []
    for r in range(w):
        th = [math.pi * (k + 0.5) / n for k in range(n)]
        f = [psi(r - (w // 2 - 1) - (0.5 * math.cos(a) + 0.5), w, beta) for a in th]
        cheb = [(2.0 if j else 1.0) / n * math.fsum(v * math.cos(j * a) for v, a in zip(f, th))
                for j in range(deg + 1)]
        # sum_j cheb_j T_j(2u) -> monomials in x = 2u -> in u
        t0, t1 = [1.0], [0.0, 1.0]
        mono = [0.0] * (deg + 1)
        for j in range(deg + 1):
            for d, v in enumerate(t0):
                mono[d] += cheb[j] * v
            t2 = [0.0] + [2.0 * v for v in t1]
            for d, v in enumerate(t0):
                t2[d] -= v
            t0, t1 = t1, t2
        rows.append([v * 2.0 ** d for d, v in enumerate(mono)])
    return rows


def emit(out, decl, values, fmt, per_line=8):
    out.write("%s = {\n" % decl)
    for i in range(0, len(values), per_line):
        out.write("  " + ", ".join(fmt(v) for v in values[i:i + per_line]) + ",\n")
    out.write("};\n")


def f32(v):
    s = "%.9g" % v
    return (s if any(c in s for c in ".en") else s + ".0") + "f"


def f64(v):
    s = "%.17g" % v
    return s if any(c in s for c in ".en") else s + ".0"


def c32(v):
    return "{%s, %s}" % (f32(v[0]), f32(v[1]))


def unit(num, den):
    a = 2.0 * math.pi * num / den
    return math.cos(a), math.sin(a)


def main(path):
    w, beta, deg, m = 8, 0.742 * 8 * math.pi, 8, 4096
    with open(path, "w") as out:
        out.write("// written by gen_transform_tables.py\n")
        polys = window_polys(w, beta, deg)
        # kTfPoly[d][r]: coefficient of u^d for the cell r - 3 cells from the observation's own
        emit(out, "__device__ const float kTfPoly[%d * %d]" % (deg + 1, w),
             [polys[r][d] for d in range(deg + 1) for r in range(w)], f32)
        # kTfDeconv[256 s + t]: 1 / psi^ at the offset of thread t's s-th output, t/16 + 16 (t%16) + 256 s - m/4
        emit(out, "__device__ const float kTfDeconv[%d]" % (m // 2),
             [1.0 / psi_hat((t // 16 + 16 * (t % 16) + 256 * s - m // 4) / m, w, beta)
              for s in range(8) for t in range(256)], f32)
        # twiddles of the 4096-point transform's first two radix-16 passes
        emit(out, "__device__ const float2 kTfTw1[15 * 256]",
             [unit(p * b, 4096) for p in range(1, 16) for b in range(256)], c32, 4)
        emit(out, "__device__ const float2 kTfTw2[15 * 16]",
             [unit(r * d, 256) for r in range(1, 16) for d in range(16)], c32, 4)


if __name__ == "__main__":
    main(sys.argv[1])
