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
import struct
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


def window_sub_polys(w, beta, deg, n_sub):
    """[s][r][d]: monomial coefficients in v of psi(r - (w/2 - 1) - (s + 1/2 + v) / n_sub), |v| <= 1/2."""
    n = 12
    th = [math.pi * (k + 0.5) / n for k in range(n)]
    cosj = [[math.cos(j * a) for a in th] for j in range(deg + 1)]
    # Chebyshev polynomials in monomials of x = 2v
    mono = [[1.0], [0.0, 1.0]]
    while len(mono) <= deg:
        nxt = [0.0] + [2.0 * v for v in mono[-1]]
        for d, v in enumerate(mono[-2]):
            nxt[d] -= v
        mono.append(nxt)
    out = []
    for s in range(n_sub):
        rows = []
        for r in range(w):
            f = [psi(r - (w // 2 - 1) - (s + 0.5 + 0.5 * c) / n_sub, w, beta) for c in cosj[1]]
            cheb = [(2.0 if j else 1.0) / n * math.fsum(v * c for v, c in zip(f, cosj[j])) for j in range(deg + 1)]
            rows.append([math.fsum(cheb[j] * mono[j][d] for j in range(deg + 1) if d < len(mono[j])) * 2.0 ** d
                         for d in range(deg + 1)])
        out.append(rows)
    return out


def deconv_poly(w, beta, deg):
    """Monomial coefficients in z = (4 xi)^2, 0 <= z <= 1, of 1 / psi^(xi)."""
    n = 64
    th = [math.pi * (k + 0.5) / n for k in range(n)]
    f = [1.0 / psi_hat(0.25 * math.sqrt(0.5 * math.cos(a) + 0.5), w, beta) for a in th]
    cheb = [(2.0 if j else 1.0) / n * math.fsum(v * math.cos(j * a) for v, a in zip(f, th)) for j in range(deg + 1)]
    # T_j(2z - 1) in powers of z
    t0, t1, c = [1.0], [-1.0, 2.0], [0.0] * (deg + 1)
    for j in range(deg + 1):
        for d, v in enumerate(t0):
            c[d] += cheb[j] * v
        t2 = [0.0] * (len(t1) + 1)
        for d, v in enumerate(t1):
            t2[d] -= 2.0 * v
            t2[d + 1] += 4.0 * v
        for d, v in enumerate(t0):
            t2[d] -= v
        t0, t1 = t1, t2
    return c


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


def single(v):
    return struct.unpack("f", struct.pack("f", v))[0]


def two(v):
    """A double as a two-float pair (48 of its bits)."""
    h = single(v)
    return "%s, %s" % (f32(h), f32(single(v - h)))


def dd(v):
    return "{%s}" % two(v)


def dd2(v):
    return "{%s, %s}" % (two(v[0]), two(v[1]))


def c32(v):
    return "{%s, %s}" % (f32(v[0]), f32(v[1]))


def unit(num, den):
    """(cos, sin) of 2 pi num / den, the angle reduced to the first octant first."""
    num %= den
    q, r = divmod(8 * num, den)  # octant and remainder / den
    s = r if q % 2 == 0 else den - r
    a = 2.0 * math.pi * s / (8 * den)
    c, v = math.cos(a), math.sin(a)
    if q in (1, 2, 5, 6):
        c, v = v, c
    return (-c if q in (2, 3, 4, 5) else c), (-v if q >= 4 else v)


def main(path):
    w, beta, deg, m = 8, 0.742 * 8 * math.pi, 8, 4096
    with open(path, "w") as out:
        out.write("// written by gen_transform_tables.py\n")
        polys = window_polys(w, beta, deg)
        out.write("#if defined(LSP_TF_TABLES_F32) || defined(LSP_TF_TABLES_LONG)\n")
        # kTfPoly[d][r]: coefficient of u^d for the cell r - 3 cells from the observation's own
        emit(out, "__device__ const float kTfPoly[%d * %d]" % (deg + 1, w),
             [polys[r][d] for d in range(deg + 1) for r in range(w)], f32)
        out.write("#endif\n")
        out.write("#ifdef LSP_TF_TABLES_F32\n")
        # kTfDeconv[256 s + t]: 1 / psi^ at the offset of thread t's s-th output, t/16 + 16 (t%16) + 256 s - m/4
        emit(out, "__device__ const float kTfDeconv[%d]" % (m // 2),
             [1.0 / psi_hat((t // 16 + 16 * (t % 16) + 256 * s - m // 4) / m, w, beta)
              for s in range(8) for t in range(256)], f32)
        # twiddles of the 4096-point transform's first two radix-16 passes
        emit(out, "__device__ const float2 kTfTw1[4 * 256]",
             [unit(p * b, 4096) for p in (1, 2, 4, 8) for b in range(256)], c32, 4)
        emit(out, "__device__ const float2 kTfTw2[4 * 16]",
             [unit(r * d, 256) for r in (1, 2, 4, 8) for d in range(16)], c32, 4)
        out.write("#endif\n")
        # one long object: e^{2 pi i n / 4096}, e^{2 pi i n / 2^24}, and 1 / psi^ as a polynomial in (4 xi)^2
        out.write("#ifdef LSP_TF_TABLES_LONG\n")
        emit(out, "__device__ const float2 kUnit[4096]", [unit(k, 4096) for k in range(4096)], c32, 4)
        emit(out, "__device__ const float2 kFine[4096]", [unit(k, 1 << 24) for k in range(4096)], c32, 4)
        emit(out, "__device__ const float4 kUnitD[4096]", [unit(k, 4096) for k in range(4096)], dd2, 2)
        emit(out, "__device__ const float4 kFineD[4096]", [unit(k, 1 << 24) for k in range(4096)], dd2, 2)
        emit(out, "__device__ const float kDeconvPoly[9]", deconv_poly(w, beta, 8), f32)
        emit(out, "__device__ const float2 kDeconvPolyD[17]", deconv_poly(16, 0.741 * 16 * math.pi, 16), dd, 4)
        out.write("#endif\n")
        out.write("#ifdef LSP_TF_TABLES_F64\n")
        w, beta, deg, n_sub = 16, 0.741 * 16 * math.pi, 5, 64
        polys = window_sub_polys(w, beta, deg, n_sub)
        # kTfPolyD[(6 sub + d) 16 + r]: coefficient of v^d, sub-interval sub of a cell, cell r - 7
        out.write("#endif\n#if defined(LSP_TF_TABLES_F64) || defined(LSP_TF_TABLES_LONG)\n")
        emit(out, "__device__ const float2 kTfPolyD[%d]" % (n_sub * (deg + 1) * w),
             [polys[s][r][d] for s in range(n_sub) for d in range(deg + 1) for r in range(w)], dd, 4)
        out.write("#endif\n#ifdef LSP_TF_TABLES_F64\n")
        emit(out, "__device__ const float2 kTfDeconvD[%d]" % (m // 2),
             [1.0 / psi_hat((t // 16 + 16 * (t % 16) + 256 * s - m // 4) / m, w, beta)
              for s in range(8) for t in range(256)], dd, 4)
        emit(out, "__device__ const float4 kTfTwD1[15 * 256]",
             [unit(p * b, 4096) for p in range(1, 16) for b in range(256)], dd2, 2)
        emit(out, "__device__ const float4 kTfTwD2[15 * 16]",
             [unit(r * d, 256) for r in range(1, 16) for d in range(16)], dd2, 2)
        out.write("#endif\n")


if __name__ == "__main__":
    main(sys.argv[1])
