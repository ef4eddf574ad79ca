// Kinetic split fluxes of reconstructed states in 64-bit fixed point.
//
// An SM's FP64 unit takes a warp instruction in 19 cycles, so each of its four
// schedulers, all asking, issues one in 76 (64, the latency, when it asks
// alone); a 32x32-bit multiply-add takes a scheduler 4.5, an integer add or
// shift 2 (measured).
// A flux evaluated in FP64, or in FP64 with single operations moved to the
// integer pipes, is bound by that unit (or by unpacking, normalising and
// packing each result: about 80 cycles for a correctly rounded multiply).
// Here a whole flux stays in fixed point: every quantity is an unsigned
// 64-bit magnitude with a fixed unit (its sign apart), so a product is three
// 32-bit multiplies and two adds (15 cycles, measured), a sum two adds, and
// nothing is normalised.  Units are chosen so that each result's error is
// below that of the FP64 form for quantities of order one; the sums over a
// point's neighbours are exact integers.  The fluxes are linear in the
// density, so a point in thin gas has its whole stencil's densities scaled up
// by a power of two (fx_shift) and its sums scaled back.  Measured against 80
// bits, 20,000 states of 0.6 < T < 0.85 per line, rms in 2^-53 of the sum of a
// component's terms' magnitudes, in parentheses FP64 (the momentum across the
// axis, which adds to that along the other, is below 0.25 of the larger of the
// two):
//                             mass         along        energy
//   M 0.02  rho 1             0.15 (1.2)   0.16 (0.7)   0.63 (1.6)
//           rho 1e-6 .. 1/2   0.20 (1.4)   0.29 (0.7)   1.15 (1.6)
//   M 1.2   rho 1             0.10 (1.1)   0.14 (1.1)   0.24 (1.3)
//           rho 1e-6 .. 1/2   0.11 (4.3)   0.21 (4.0)   0.41 (4.3)
// Cold gas at rest (T < 0.4, M < 0.1: no adiabatic flow has it) is the one
// place behind FP64: energy 2.7 (1.6).
//
// The state's ranges, in units with a free stream of density 1 and speed of
// sound 1: 1/4 < T = p/rho < 2, i.e. 0.5 < 2 beta < 4 (to 2^-10); |u|, |v| < 4;
// |2 beta u|, |2 beta v| < 4; ln(rho beta^2.5) in (-16, 0); rho/sqrt(beta) < 4;
// |S| < 2.5 and a mass moment below 4 along each axis (densities times 2^sh).  They hold for subsonic to moderately supersonic flow; a state
// outside (or not finite) is reported and its point is evaluated in FP64.
#pragma once
#include <cmath>
#include <cstdint>

#include "lskum_fixmath.cuh"

namespace lskum {

// Table layout (kFluxTable, 64-bit words; R = kFluxRows): R pairs (e0, |e1|),
// R pairs (k0, e2), R pairs of packed (e3, e4), (e5, k3), R words (k4, k5),
// then e^(j/2048).
constexpr int kFluxTableR = 640, kFluxTableExp = 1424;
constexpr int kFluxTableWords = 7 * kFluxTableR + kFluxTableExp;
constexpr uint64_t kLn2Fx = 199786072581291495ull;  // ln 2 in 2^-58
constexpr int32_t kInvLn2Fx = 1549082005;           // 1/ln 2 in 2^-30

LSKUM_HD uint32_t umulhi32(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
LSKUM_HD int32_t mulhi32(int32_t a, int32_t b)
{
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}

// High 64 bits of the product of two unsigned words without the low words'
// product and the cross products' low halves: at most 3 units below it.
LSKUM_HD uint64_t mulh_t(uint64_t a, uint64_t b)
{
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + umulhi32(ah, bl) + umulhi32(al, bh);
}

// 1/sqrt of the float with these bits, to FP32 accuracy.
LSKUM_HD float rsqrt_seed(uint32_t bits)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(bits)));
    return y;
#else
    float x;
    std::memcpy(&x, &bits, sizeof x);
    return 1.0f / sqrtf(x);
#endif
}

// |z| in units of 2^-s for |z| < 2^(64 - s), truncated.
LSKUM_HD uint64_t fix_mag(double z, int s)
{
    const uint64_t b = f64_bits(z);
    const uint32_t hi = (uint32_t)(b >> 32);
    const int n = 1086 - s - (int)((hi >> 20) & 0x7ffu);  // >= 0 in range
    const uint64_t M = (((uint64_t)((hi & 0x000fffffu) | 0x00100000u) << 32) | (uint32_t)b) << 11;
    return M >> (n < 63 ? n : 63);
}

// x with its sign flipped where m is all ones (m: 0 or -1).
LSKUM_HD uint64_t neg_if(uint64_t x, int32_t m)
{
    const uint64_t mm = (uint64_t)(int64_t)m;
    return (x ^ mm) - mm;
}

// What the split fluxes of one state need, in both axes of its frame: |u| and
// |v| (2^-62) with their signs (0 or -1), sqrt(beta) (2^-63), rho/sqrt(beta)
// (2^-62) and p (2^-62), both times 2^sh, 3T + |u|^2/2 (2^-60, T = p/rho).
struct FxState {
    uint64_t u, v, sb, rs, p, h;
    int32_t su, sv;
};

// The power of two that a point's densities are scaled by, from the high words
// of its own state's rho and 1/sqrt(beta): brings rho/sqrt(beta) to 1/2 or
// more (their exponents and mantissas added as integers: log2 within 0.18).
LSKUM_HD uint32_t fx_shift(uint32_t rho, uint32_t isb)
{
    const int32_t e = (int32_t)((rho + isb - 0x3ff00000u) >> 20) - 1023;  // floor(log2)
    return e >= -1 ? 0u : (e < -25 ? 24u : (uint32_t)(-1 - e));
}

// Do q-variables with these high words lie outside fx_state's ranges?
// (-4 < z3 < -0.5 (1 + 2^-10); |z1|, |z2| < 4; |z0| < 16)
LSKUM_HD bool fx_outside(uint32_t h0, uint32_t h1, uint32_t h2, uint32_t h3)
{
    return !(h3 - 0xbfe00400u < 0xc0100000u - 0xbfe00400u) | ((h1 & 0x7fffffffu) >= 0x40100000u) |
           ((h2 & 0x7fffffffu) >= 0x40100000u) | ((h0 & 0x7fffffffu) >= 0x40300000u);
}

// The state of q-variables z (Eq. 14 inverted) with z[1], z[2] along the
// frame's axes.  bad: bit 31 set when the state leaves the ranges above (the
// values are then meaningless but every table index stays in range).
LSKUM_HD void fx_state(const uint64_t *tab, double z0, double z1, double z2, double z3, FxState &s, uint32_t &bad,
                       uint32_t sh = 0)
{
    const uint32_t h0 = (uint32_t)(f64_bits(z0) >> 32), h1 = (uint32_t)(f64_bits(z1) >> 32);
    const uint32_t h2 = (uint32_t)(f64_bits(z2) >> 32), h3 = (uint32_t)(f64_bits(z3) >> 32);
    uint32_t b = fx_outside(h0, h1, h2, h3) ? 0x80000000u : 0u;
    s.su = (int32_t)h1 >> 31;
    s.sv = (int32_t)h2 >> 31;
    const uint64_t beta = fix_mag(z3, 62);  // 2 beta in 2^-62 = beta in 2^-63
    // 1/sqrt(beta): an FP32 seed y0 (31 bits), e = 1 - beta y0^2 (|e| < 2^-20),
    // y0 (1 + e/2 + 3 e^2/8); the next term is below 2^-61
    const float y0 = rsqrt_seed(((h3 & 0x7fffffffu) - (897u << 20)) << 3 | (uint32_t)(f64_bits(z3) & 0xffffffffu) >> 29);
    const uint32_t Y = (uint32_t)(y0 * 1073741824.0f);            // 2^-30, < 2^31
    const uint64_t pr = mulh_t(beta, ((uint64_t)Y * Y) << 2);   // beta y0^2 in 2^-61
    const int64_t e = (int64_t)(1ull << 61) - (int64_t)pr;        // 2^-61; as e/2: 2^-62
    const int32_t eh = (int32_t)(e >> 17);                        // 2^-44
    const int64_t c = e + ((3 * ((int64_t)eh * eh)) >> 29);       // e/2 + 3 e^2/8 in 2^-62
    const int32_t ch = (int32_t)(c >> 32);
    const uint64_t isb = ((uint64_t)Y << 33) + ((uint64_t)((int64_t)(int32_t)Y * ch) << 3) +
                         (((uint64_t)Y * (uint32_t)c) >> 29);     // 2^-63
    const uint64_t ib = mulh_t(isb, isb);                         // 1/beta in 2^-62 = T in 2^-63
    const uint64_t u = mulh_t(fix_mag(z1, 62), ib);               // 2^-61
    const uint64_t v = mulh_t(fix_mag(z2, 62), ib);
    s.u = u << 1;
    s.v = v << 1;
    const uint64_t k = (mulh_t(s.u, s.u) >> 1) + (mulh_t(s.v, s.v) >> 1);  // |u|^2/2 in 2^-60
    const uint64_t bk = mulh_t(beta, k);                          // beta |u|^2/2 in 2^-59
    // |u|, |v| < 4, |u|^2/2 < 8, beta |u|^2 < 16
    b |= (uint32_t)((u | v | k) >> 32) | ((uint32_t)(bk >> 32) + 0x40000000u);
    s.h = 3 * (ib >> 3) + k;
    // a = z0 + beta |u|^2 = ln(rho beta^2.5) in (-16, 0), 2^-58
    const int64_t a = (int64_t)(neg_if(fix_mag(z0, 58), (int32_t)h0 >> 31) + bk);
    const int32_t ah = (int32_t)(a >> 32);                        // 2^-26
    b |= ~((uint32_t)ah & ((uint32_t)ah << 1));
    // a = r - nk ln 2 with 0 <= r < ln 2 (1 + 2^-20), e^a = 2^-nk e^(j/2048) e^x
    const uint32_t nk = (uint32_t)(-(mulhi32(ah, kInvLn2Fx) >> 24)) & 31u;
    const uint64_t r = (uint64_t)a + (uint64_t)nk * (uint32_t)kLn2Fx +
                       ((uint64_t)(nk * (uint32_t)(kLn2Fx >> 32)) << 32);
    const uint32_t rh = (uint32_t)(r >> 32), j0 = rh >> 15;
    const uint32_t j = j0 < (uint32_t)kFluxTableExp ? j0 : (uint32_t)kFluxTableExp - 1;
    const uint64_t x = (((uint64_t)(rh & 0x7fffu) << 32) | (uint32_t)r) << 6;  // 2^-64, < 2^-11
    // e^x - 1 = x + x P, P = x/2 + x^2/6 + x^3/24 (the next term, x^5/120, is below 2^-61)
    const uint32_t xh = (uint32_t)(x >> 21);                      // 2^-43
    const uint32_t x2 = umulhi32(xh, xh);                         // x^2 in 2^-54
    const uint32_t x36 = umulhi32(x2, 715827883u) + (umulhi32(umulhi32(x2, xh), 178956971u) >> 11);
    const uint64_t P = (x >> 1) + ((uint64_t)x36 << 10);
    const uint64_t tj = tab[7 * kFluxTableR + j];                 // 2^-62
    const uint64_t V = tj + mulh_t(tj, x + mulh_t(x, P));
    // rho/sqrt(beta) = e^a beta^-3; p = rho T
    const uint64_t ib3 = mulh_t(mulh_t(ib, ib), ib);              // 2^-58
    const uint64_t r0 = mulh_t(V, ib3);                           // 2^-56; 2^sh rho/sqrt(beta) in 2^-62: << 6 - t
    const int32_t t = (int32_t)nk - (int32_t)sh, m = t < 6 ? t : 6;
    b |= (r0 >> (58 + (t < 5 ? t : 5))) != 0 ? 0x80000000u : 0u;  // 2^sh rho/sqrt(beta) < 4 (r0 < 2^63)
    s.rs = (r0 << (6 - m)) >> (t - m);
    s.p = mulh_t(s.rs, isb);                                      // rho/beta in 2^-61 = p in 2^-62
    s.sb = mulh_t(beta, isb) << 1;                                // 2^-63
    bad |= b;
}

// One split flux of state s along an axis of its frame, for the upwind (pos)
// or downwind half: a, sa the velocity along the axis, o across it.  With
// w = +a or -a the velocity towards the half's side, S = w sqrt(beta),
// J = K(|S|) + max(S, 0): the mass moment is rm = rho/sqrt(beta) J, and the
// flux is sg (rm, rm h + w p A / 2) for mass and energy, rm w + p A for the
// momentum along and sg rm o across, A = (1 + erf S)/2 (sg = 1 if pos, else
// -1, left to the caller's weight).  Units: rm 2^-59, ga and go 2^-57, g3 2^-55.
struct FxFlux {
    uint64_t rm, ga, go, g3;
};

LSKUM_HD void fx_flux(const uint64_t *tab, const FxState &s, uint64_t a, int32_t sa, uint64_t o, int32_t so,
                      bool pos, FxFlux &f, uint32_t &bad)
{
    const int32_t neg = sa ^ (pos ? 0 : -1);  // -1: w < 0
    const uint64_t S = mulh_t(a, s.sb);       // 2^-61
    const uint32_t Sh = (uint32_t)(S >> 32);
    bad |= Sh | (Sh + 0x30000000u);           // |S| < 2.5
    const uint32_t i0 = Sh >> 21, iv = i0 < (uint32_t)kFluxTableR ? i0 : (uint32_t)kFluxTableR - 1;
#ifdef __CUDA_ARCH__
    const ulonglong2 *t2 = reinterpret_cast<const ulonglong2 *>(tab);
    const ulonglong2 q0 = t2[iv], q1 = t2[kFluxTableR + iv], q2 = t2[2 * kFluxTableR + iv];
    const uint64_t e0 = q0.x, e1 = q0.y, k0 = q1.x, e2 = q1.y, c0 = q2.x, c1 = q2.y;
#else
    const uint64_t e0 = tab[2 * iv], e1 = tab[2 * iv + 1], k0 = tab[2 * kFluxTableR + 2 * iv],
                   e2 = tab[2 * kFluxTableR + 2 * iv + 1], c0 = tab[4 * kFluxTableR + 2 * iv],
                   c1 = tab[4 * kFluxTableR + 2 * iv + 1];
#endif
    const uint64_t c2 = tab[6 * kFluxTableR + iv];
    const uint64_t t = S << 11;              // position in the interval, 2^-64
    const int32_t th = (int32_t)(t >> 33);   // 2^-31
    int32_t p = (int32_t)(uint32_t)(c0 >> 32) + mulhi32(th, (int32_t)(uint32_t)c1);
    p = (int32_t)(uint32_t)c0 + mulhi32(th, p);
    uint64_t d = e2 + (uint64_t)(((int64_t)th * p) >> 25);
    d = e1 - mulh_t(t, d);
    const uint64_t E = e0 - mulh_t(t, d);    // 2^-63
    p = (int32_t)(uint32_t)c2 + mulhi32(th, (int32_t)(uint32_t)(c2 >> 32));
    p = (int32_t)(uint32_t)(c1 >> 32) + mulhi32(th, p);
    d = (e1 >> 11) - (uint64_t)(((int64_t)th * p) >> 28);
    d = (e0 >> 10) - mulh_t(t, d);
    const uint64_t K = k0 - mulh_t(t, d);    // 2^-61
    const uint64_t m = (uint64_t)(int64_t)neg;
    const uint64_t A = neg ? E : (1ull << 63) - E;   // 2^-63
    const uint64_t J = K + (S & ~m);                 // 2^-61
    f.rm = mulh_t(s.rs, J);
    bad |= (uint32_t)(f.rm >> 32) + 0x60000000u;     // rm < 4: differences fit 63 bits
    const uint64_t pA = mulh_t(s.p, A);              // 2^-61
    f.ga = (pA >> 4) + (mulh_t(f.rm, a) ^ m) - m;
    f.go = neg_if(mulh_t(f.rm, o), so);
    f.g3 = mulh_t(f.rm, s.h) + ((mulh_t(a, pA) >> 5) ^ m) - m;
}

// Sum over a point's neighbours of weight x flux difference, exact: the weight
// is wh + 2^-24 wl, both integers, |wl| <= 2^23 (in units of a power of two
// per point, chosen at create so that sum |wh| < 2^30; at most 510 terms).
struct FxSum {
    int64_t hh, l, r;
};

// The two signed parts of a word that was biased by 2^31: high 2^32 + low.
LSKUM_HD void split_word(uint64_t biased, int32_t &high, int32_t &low)
{
#ifdef __CUDA_ARCH__
    // (opaque: from a shift the compiler forms some of the products with the
    // high part as 64x64-bit ones)
    asm("mov.b64 {%0, %1}, %2;" : "=r"(low), "=r"(high) : "l"(biased));
#else
    low = (int32_t)(uint32_t)biased;
    high = (int32_t)(uint32_t)(biased >> 32);
#endif
    low ^= (int32_t)0x80000000;
}

LSKUM_HD void fx_add(FxSum &s, int32_t wh, int32_t wl, uint64_t Gi, uint64_t G0)
{
    const uint64_t D = Gi - G0 + 0x80000000ull;  // |Gi - G0| < 2^62.4
    int32_t dh, dl;
    split_word(D, dh, dl);
    s.hh += (int64_t)wh * dh;
    s.l += (int64_t)wh * dl;
    s.r += (int64_t)wl * dh;
}

// The sum as a double, in units of 2^32 of the flux's unit times the weight's
// (left out: 8 bits of l, 2^-24 of a unit of the flux in all, and wl's
// products with the differences' low words, below that unit each).
LSKUM_HD double fx_total(const FxSum &s)
{
    return fma((double)((s.l >> 8) + s.r), 0x1p-24, (double)s.hh);  // |l >> 8| + |r| < 2^63
}

}  // namespace lskum
