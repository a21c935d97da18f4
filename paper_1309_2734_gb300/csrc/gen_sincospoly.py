"""Writes sincospoly.h: sqrt(2) sin(pi r) / r and sqrt(2) cos(pi r), |r| <= 1/2, as polynomials of degree 4 in u = r^2.

The tensor-core direct form takes the sine and cosine of half a turn's angle and doubles it: with s = sqrt(2) sin(pi r)
and c = sqrt(2) cos(pi r), cos(2 pi r) = 1 - s^2 and sin(2 pi r) = s c, so no quadrant is selected.

Method: Lawson's iteratively reweighted least squares (a standard route to the minimax polynomial) on Chebyshev nodes
of u in [0, 1/4], the sine weighted by r (fit errors 3.3e-9 and 4.7e-8).  The coefficients, rounded to single
precision, are then moved by whole float steps, one at a time, while that lowers the RMS error of the evaluation in
single precision (signed 32-bit turn -> float, FMA Horner steps) over the turns: 1.72e-7 to 1.20e-7.

Run:  python gen_sincospoly.py > sincospoly.h
"""
import numpy as np


def fit(fun, weight, deg, nodes=6000, iters=400):
    k = np.arange(nodes)
    u = 0.125 * (np.cos(np.pi * (k + 0.5) / nodes) + 1.0)
    f, W = fun(u), weight(u)
    V = np.vander(u, deg + 1, increasing=True)
    wt = np.ones_like(u)
    for _ in range(iters):
        s = np.sqrt(wt) * W
        c, *_ = np.linalg.lstsq(V * s[:, None], f * s, rcond=None)
        wt = wt * np.abs(V @ c - f) * W
        wt = np.maximum(wt / wt.mean(), 1e-12)
    return c


def f32(x):
    return np.asarray(x).astype(np.float32).astype(np.float64)


TURNS = np.arange(1 << 17, dtype=np.int64) * (1 << 15) + (1 << 14) - (1 << 31)
R = f32(TURNS.astype(np.float64)) * 2.0 ** -32
U = f32(R * R)
THETA = 2 * np.pi * TURNS / 2.0 ** 32


def rms(S, C):
    hs, hc = np.full_like(U, S[-1]), np.full_like(U, C[-1])
    for i in range(len(S) - 2, -1, -1):
        hs, hc = f32(hs * U + S[i]), f32(hc * U + C[i])
    s = f32(R * hs)
    a, b = f32(1 - s * s) - np.cos(THETA), f32(s * hc) - np.sin(THETA)
    return np.sqrt((a * a).mean() + (b * b).mean())


def moved(v, steps):
    return float((np.array([v], np.float32).view(np.int32) + np.int32(steps)).view(np.float32)[0])


def main():
    root = np.sqrt
    S = f32(root(2) * fit(lambda u: np.sin(np.pi * root(u)) / np.maximum(root(u), 1e-30), root, 4))
    C = f32(root(2) * fit(lambda u: np.cos(np.pi * root(u)), np.ones_like, 4))
    best = rms(S, C)
    for _ in range(6):
        before = best
        for arr in (S, C):
            for i in range(len(arr)):
                for k in (1, -1, 2, -2, 4, -4, 16, -16, 64, -64, 256, -256):
                    old = arr[i]
                    arr[i] = moved(old, k)
                    r = rms(S, C)
                    if r < best * (1 - 1e-6):
                        best = r
                    else:
                        arr[i] = old
        if best == before:
            break
    print("// Generated by gen_sincospoly.py; do not edit.")
    print("// sqrt(2) sin(pi r) = r (S0 + S1 u + ... + S4 u^4) and sqrt(2) cos(pi r) = C0 + C1 u + ... + C4 u^4, "
          "u = r^2, |r| <= 1/2.")
    print("#pragma once")
    for name, arr in (("HSIN", S), ("HCOS", C)):
        for i, v in enumerate(arr):
            print(f"#define CGH_{name}_{i} {float(v)!r}f")


if __name__ == "__main__":
    main()
