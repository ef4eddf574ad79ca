"""Generate lskum_fluxtable.h: the tables of the fixed-point split fluxes.

Run from the repository root:  python paper_2406_07441_gb300/csrc/gen_fluxtable.py
(needs mpmath; the generated header is committed, so building does not).

The split flux of a Maxwellian along its own direction of motion needs, with
S = |u_d| sqrt(beta),
  E(S) = erfc(S)/2           (A = 1 - E or E),
  K(S) = exp(-S^2)/(2 sqrt pi) - S E(S)
(the mass moment is rho/sqrt(beta) times K, or K + S on the downstream side).
K' = -E, K'' = -E' = exp(-S^2)/sqrt(pi) > 0: both functions fall, convex.
On each interval [j/256, (j+1)/256) of [0, 2.5), with t the position in it,
  E = e0 - t (|e1| - t (e2 + t (e3 + t (e4 + t e5)))),
  K = k0 - t (e0 h - t (|e1| h/2 - t (k3 + t (k4 + t k5)))),   h = 1/256:
E by the Chebyshev interpolant of degree 5 (error below 2^-63), K by the
integral of E's leading terms and a cubic tail interpolated at Chebyshev
points.  Fixed point: e0, |e1|, e2 in units of 2^-63, k0 in units of 2^-61,
e3, e4, e5 of 2^-57, 2^-58, 2^-59 and k3, k4, k5 of 2^-58, 2^-59, 2^-60 (each
32-bit high product with t halves the unit).  The generator runs the
kernels' integer steps (lskum_fixflux.cuh) exactly and checks them against
mpmath.

e^(j/2048), j = 0 .. 1423 (0 to ln 2 and a little beyond), in units of 2^-62.
"""
import os

import mpmath as mp

HERE = os.path.dirname(os.path.abspath(__file__))
OUT = os.path.join(HERE, "lskum_fluxtable.h")
ROWS, STEP_LOG2 = 640, 8   # [0, 2.5) in intervals of 2^-8
EXP_ROWS = 1424


def E(x):
    return mp.erfc(x) / 2


def K(x):
    return mp.exp(-x * x) / (2 * mp.sqrt(mp.pi)) - x * E(x)


def monomial_fit(f, n):
    """Coefficients of the degree-n interpolant of f at Chebyshev points of [0, 1]."""
    N = n + 1
    xs = [(1 + mp.cos(mp.pi * (k + mp.mpf(1) / 2) / N)) / 2 for k in range(N)]
    A = mp.matrix(N, N)
    b = mp.matrix(N, 1)
    for i, x in enumerate(xs):
        for j in range(N):
            A[i, j] = x ** j
        b[i] = f(x)
    c = mp.lu_solve(A, b)
    return [c[j] for j in range(N)]


def fx(v, s):
    return int(mp.nint(v * mp.mpf(2) ** s))


def row(j):
    h = mp.mpf(1) / 2 ** STEP_LOG2
    x0 = j * h
    c = monomial_fit(lambda t: E(x0 + t * h), 5)
    e0, e1, e2 = fx(c[0], 63), fx(-c[1], 63), max(fx(c[2], 63), 0)
    # half a unit is added where the next term's high product is rounded down
    half = mp.mpf(1) / 2
    e3, e4, e5 = fx(c[3] + half / 2 ** 57, 57), fx(c[4] + half / 2 ** 58, 58), fx(c[5], 59)
    q0, q1 = mp.mpf(e0) / 2 ** 63 * h, mp.mpf(e1) / 2 ** 63 * h / 2
    k0 = K(x0)
    k = monomial_fit(lambda t: (k0 - q0 * t + q1 * t * t - K(x0 + t * h)) / t ** 3, 2)
    k3, k4, k5 = fx(k[0] + half / 2 ** 58, 58), fx(k[1] + half / 2 ** 59, 59), fx(k[2], 60)
    for v in (e3, e4, e5, k3, k4, k5):
        assert abs(v) < 2 ** 31
    return e0, e1, e2, fx(k0, 61), e3, e4, e5, k3, k4, k5


def mulh_t(a, b):
    """The kernels' truncated high product of two unsigned 64-bit words."""
    ah, al, bh, bl = a >> 32, a & 0xffffffff, b >> 32, b & 0xffffffff
    return ah * bh + (ah * bl >> 32) + (al * bh >> 32)


def evaluate(r, S):
    """The kernels' integer steps for S in units of 2^-61: (E 2^63, K 2^61)."""
    e0, e1, e2, k0, e3, e4, e5, k3, k4, k5 = r
    t = (S << 11) & (2 ** 64 - 1)
    th = t >> 33
    a = e4 + (th * e5 >> 32)
    a = e3 + (th * a >> 32)
    d = e2 + (th * a >> 25)
    assert 0 <= d < 2 ** 64
    d = e1 - mulh_t(t, d)
    assert 0 <= d < 2 ** 64
    ee = e0 - mulh_t(t, d)
    a = k4 + (th * k5 >> 32)
    a = k3 + (th * a >> 32)
    d = (e1 >> 11) - (th * a >> 28)
    assert 0 <= d < 2 ** 64
    d = (e0 >> 10) - mulh_t(t, d)
    assert 0 <= d < 2 ** 64
    return ee, k0 - mulh_t(t, d)


def main(out=OUT):
    with mp.workdps(40):
        rows = [row(j) for j in range(ROWS)]
        worst = [mp.mpf(0), mp.mpf(0)]
        for j, r in enumerate(rows):
            for k in range(12):
                S = (j << 53) + ((1 << 53) * k // 11 - (k == 11))
                ee, kk = evaluate(r, S)
                x = mp.mpf(S) / mp.mpf(2) ** 61
                worst[0] = max(worst[0], abs(mp.mpf(ee) / mp.mpf(2) ** 63 - E(x)))
                worst[1] = max(worst[1], abs(mp.mpf(kk) / mp.mpf(2) ** 61 - K(x)))
        # within 2^-56.4 and 2^-57, below a quarter of FP64's own rounding of A and of the mass moment
        assert worst[0] < mp.mpf(2) ** -56.4 and worst[1] < mp.mpf(2) ** -57, [mp.log(w, 2) for w in worst]
        ex = [fx(mp.exp(mp.mpf(j) / 2048), 62) for j in range(EXP_ROWS)]
        ln2 = fx(mp.log(2), 58)
        c = fx(1 / mp.log(2), 30)
    lines = [
        "// Generated by gen_fluxtable.py (mpmath); do not edit.",
        "// Tables of the fixed-point split fluxes; see gen_fluxtable.py for the method.",
        "#pragma once",
        "",
        "namespace lskum {",
        "",
        f"constexpr int kFluxRows = {ROWS};      // intervals of 2^-{STEP_LOG2} on [0, 2.5)",
        f"constexpr int kFluxExpRows = {EXP_ROWS};  // e^(j/2048)",
        f"constexpr unsigned long long kFluxLn2 = {ln2}ull;  // ln 2 in units of 2^-58",
        f"constexpr int kFluxInvLn2 = {c};  // 1/ln 2 in units of 2^-30",
        "",
        "// Structure of arrays in 16-byte words (a warp's reads of one word spread",
        "// over the banks): (e0, |e1|), (k0, e2), (e3, e4, e5, k3), then (k4, k5).",
        f"__device__ unsigned long long kFluxTable[{7 * ROWS + EXP_ROWS}] = {{",
    ]

    def pack(lo, hi):
        return (lo & 0xffffffff) | (hi & 0xffffffff) << 32

    words = []
    for f in (lambda r: (r[0], r[1]), lambda r: (r[3], r[2]), lambda r: (pack(r[4], r[5]), pack(r[6], r[7])),
              lambda r: (pack(r[8], r[9]),)):
        for r in rows:
            words += f(r)
    words += ex
    for j in range(0, len(words), 5):
        lines.append("    " + ", ".join(f"{v}ull" for v in words[j:j + 5]) + ",")
    lines += ["};", "", "}  // namespace lskum", ""]
    with open(out, "w") as f:
        f.write("\n".join(lines))
    return [float(mp.log(w, 2)) for w in worst]


if __name__ == "__main__":
    print(main())
