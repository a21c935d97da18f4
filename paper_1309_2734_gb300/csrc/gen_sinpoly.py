"""Writes sinpoly.h: sin(2 pi d) / d, |d| <= 1/4, as a polynomial of degree 4 in u = d^2.

The accurate direct form on the tensor cores folds a signed turn r to a quarter of a turn: -cos(2 pi r) is the sine at
|r| - 1/4 and sin(2 pi r) that at r, or at 1/2 - |r| with r's sign, so both come from one odd polynomial, whose last
operation is a product and rounds once.

Method: Lawson's iteratively reweighted least squares (a standard route to the minimax polynomial) on Chebyshev nodes of
u in [0, 1/16], weighted by d (fit error 3.3e-9).  The coefficients, rounded to single precision, are then moved by whole
float steps, one at a time, while that lowers the RMS error of the evaluation in single precision (signed 32-bit turn ->
float, fold, FMA Horner steps) over the turns.

Run:  python gen_sinpoly.py > sinpoly.h
"""
import numpy as np


def fit(deg=4, nodes=6000, iters=400):
    k = np.arange(nodes)
    u = (np.cos(np.pi * (k + 0.5) / nodes) + 1.0) / 32.0
    d = np.sqrt(u)
    f = np.sin(2.0 * np.pi * d) / np.maximum(d, 1e-30)
    V = np.vander(u, deg + 1, increasing=True)
    wt = np.ones_like(u)
    for _ in range(iters):
        s = np.sqrt(wt) * d
        c, *_ = np.linalg.lstsq(V * s[:, None], f * s, rcond=None)
        wt = wt * np.abs(V @ c - f) * d
        wt = np.maximum(wt / wt.mean(), 1e-12)
    return c, float(np.max(np.abs(V @ c - f) * d))


def f32(x):
    return np.asarray(x).astype(np.float32).astype(np.float64)


TURNS = np.arange(1 << 17, dtype=np.int64) * (1 << 15) + (1 << 14) - (1 << 31)
R = f32(TURNS.astype(np.float64)) * 2.0 ** -32
THETA = 2 * np.pi * TURNS / 2.0 ** 32
COS, SIN = np.cos(THETA), np.sin(THETA)
D = np.abs(R) - 0.25
M = np.copysign(np.minimum(np.abs(R), 0.5 - np.abs(R)), R)


def sine(c, d):
    u = f32(d * d)
    p = np.full_like(u, c[-1])
    for a in c[-2::-1]:
        p = f32(p * u + a)
    return f32(d * p)


def rms(c):
    a, b = sine(c, D) + COS, sine(c, M) - SIN
    return float(np.sqrt(((a * a).mean() + (b * b).mean()) / 2))


def moved(v, steps):
    return float((np.array([v], np.float32).view(np.int32) + np.int32(steps)).view(np.float32)[0])


def main():
    c, err = fit()
    c = f32(c)
    start = best = rms(c)
    for _ in range(6):
        before = best
        for i in range(len(c)):
            for k in (1, -1, 2, -2, 4, -4, 16, -16, 64, -64, 256, -256):
                old = c[i]
                c[i] = moved(old, k)
                r = rms(c)
                if r < best * (1 - 1e-6):
                    best = r
                else:
                    c[i] = old
        if best == before:
            break
    print("// Generated by gen_sinpoly.py; do not edit.")
    print("// sin(2 pi d) = d (S0 + S1 u + ... + S4 u^4), u = d^2, |d| <= 1/4.")
    print(f"// Fit error {err:.1e}; RMS error of a turn's entries in single precision {best:.2e} ({start:.2e} as rounded).")
    print("#pragma once")
    for i, v in enumerate(c):
        print(f"#define CGH_SIN_{i} {float(v)!r}f")


if __name__ == "__main__":
    main()
