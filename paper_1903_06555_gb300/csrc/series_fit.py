"""Coefficients of the sampled-kernel interpolation (series_kernel.cuh).

For one visibility [GC](., dw) and its panel sums are even functions of rho
band-limited to R cycles per grid pixel.  Sampled at rho = i / (4 R) -- half
the spacing the sampling theorem needs, so |omega| <= pi / 2 radian per
sample -- such a function f is, on the interval [p, p + 1] of sample units
with t = 2 (x - p) - 1 in [-1, 1],

    f(x) ~ sum_m t^m  sum_d  C[m][d] (f(p + 1 + d) + (-1)^m f(p - d)).

The weights at a point x are the least-squares ones over the band,
(A + eps^2 I)^-1 b(x) with A_ij = sinc((i - j) / 2) and b_j(x) =
sinc((x - j) / 2) (eps bounds the weights, so that rounding of the samples
is not amplified: the absolute weights sum to 1.9 in FP32 and 2.1 in FP64);
they are then interpolated in t by a polynomial through its Chebyshev points.

    FP32: 20 samples, 8 terms:  error <= 5.9e-8 at the band's edge, 5e-9
          over its lower half;
    FP64: 40 samples, 14 terms: error <= 1.2e-15.

Run:  python series_fit.py > series_coef.cuh
"""
import mpmath as mp

mp.mp.dps = 50


def fit(half, terms, eps):
    n = 2 * half
    idx = [i - (half - 1) for i in range(n)]

    def sinc(t):
        return mp.mpf(1) if t == 0 else mp.sin(mp.pi * t / 2) / (mp.pi * t / 2)

    A = mp.matrix(n, n)
    for i in range(n):
        for j in range(n):
            A[i, j] = sinc(mp.mpf(idx[i] - idx[j]))
        A[i, i] += mp.mpf(eps) ** 2
    inv = A ** -1
    t = [mp.cos(mp.pi * (k + mp.mpf(1) / 2) / terms) for k in range(terms)]
    W = mp.matrix(terms, n)
    V = mp.matrix(terms, terms)
    for k in range(terms):
        b = mp.matrix(n, 1)
        for j in range(n):
            b[j] = sinc((t[k] + 1) / 2 - idx[j])
        w = inv * b
        for j in range(n):
            W[k, j] = w[j]
        for m in range(terms):
            V[k, m] = t[k] ** m
    C = (V ** -1) * W
    # column of sample p + 1 + d; the mirrored one equals it times (-1)^m
    return [[C[m, half + d] for d in range(half)] for m in range(terms)]


def emit(name, ctype, half, terms, eps, suffix, digits):
    C = fit(half, terms, eps)
    print(f"__constant__ {ctype} {name}[{terms}][{half}] = {{")
    for row in C:
        vals = [mp.nstr(v, digits, min_fixed=0, max_fixed=0) + suffix for v in row]
        if suffix:
            vals = ["{%s, %s}" % (v, v) for v in vals]
        lines, cur = [], ""
        for v in vals:
            if len(cur) + len(v) > 88:
                lines.append(cur)
                cur = ""
            cur += v + ", "
        lines.append(cur)
        print("    {" + "\n     ".join(s.rstrip() for s in lines).rstrip(",") + "},")
    print("};")


if __name__ == "__main__":
    print("// Printed by series_fit.py in this directory (the definition is there); FP32\n"
          "// values twice, for paired arithmetic.  Included by series_kernel.cuh.\n"
          "#pragma once\n")
    emit("c_series_f", "float2", 10, 8, "1e-8", "f", 10)
    print()
    emit("c_series_d", "double", 20, 14, "1e-17", "", 20)
