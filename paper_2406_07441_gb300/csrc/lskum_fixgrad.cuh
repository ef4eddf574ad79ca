// Weighted least-squares sums of q-variables in 64-bit fixed point.
//
// The q-derivatives are sums over a point's neighbours of weight x difference:
// 12 FP64 instructions per slot in the first pass and 16 in each inner
// iteration, at 76 cycles each with all four schedulers of an SM competing for
// its FP64 unit.  As integers a weight (31 bits and up to 28 more) times a
// difference (63 bits) is four 32-bit multiply-adds into 64-bit sums, 4.5
// cycles each, and the sum is exact.
//
// A point's derivatives are kept as differences: G_x = X dq/dx with X a power
// of two such that the weights times X add up to less than 1, so |G_x| is at
// most the largest difference of q over the stencil (the same for y, with its
// own power, whatever the stencil's aspect ratio), and q and G share a unit:
// 2^-59 for the first component (|q| < 8), 2^-60 for the others (|q| < 4), times
// a power of two for the first three components of a case whose free stream
// comes near those bounds (fix_shift: from M 2.14 on; FP64's unit in the last
// place of such a value is 2^-51 or more).
// The inner iterations' coefficients absorb the ratios of their points'
// powers.  A value out of range (or not finite) is stored as a mark, with its
// FP64 value beside; points that meet a mark are evaluated in FP64.
#pragma once
#include <cmath>
#include <cstdint>

#include "lskum_fixflux.cuh"

namespace lskum {

constexpr int64_t kFixMark = INT64_MIN;
constexpr int kMaxGradBits = 28;     // a weight's bits below its integer part
constexpr int kMinGradBits = 20;     // what a point needs for the fixed-point form
constexpr int kMaxGradShift = 10;    // largest power of two of a fast inner iteration's coefficients
constexpr int kMaxGradExp = 900;     // largest |exponent| of X or Y of a fast point
constexpr int kGradNoScale = 32000;  // weights without a scale (not finite): the result is NaN

// A case's powers of two, from its free stream's q: bits 0 to 7 of the first
// component (to three quarters of its bound or less), 8 up of the second and
// third (the fourth is -1.4 in every free stream).
constexpr int kMaxFixShift = 20;
inline int fix_shift(const double q[4])
{
    int s0 = 0, s1 = 0;
    while (s0 < kMaxFixShift && !(std::fabs(q[0]) <= 6.0 * (1 << s0))) s0++;
    while (s1 < kMaxFixShift && !(std::fabs(q[1]) <= 3.0 * (1 << s1) && std::fabs(q[2]) <= 3.0 * (1 << s1))) s1++;
    return s0 | s1 << 8;
}

// -log2 of component c's unit in a case with these powers.
LSKUM_HD int fix_unit(int c, int shift = 0)
{
    return c == 0 ? 59 - (shift & 255) : (c < 3 ? 60 - (shift >> 8) : 60);
}

// Component c of q, to the nearest unit, or the mark.
LSKUM_HD int64_t fix_q(double q, int c, int shift = 0)
{
    const int32_t h = (int32_t)(f64_bits(q) >> 32);
    const int unit = fix_unit(c, shift);
    if ((h & 0x7fffffff) >= ((c == 0 ? 0x401fffff + (59 << 20) : 0x400fffff + (60 << 20)) - (unit << 20))) return kFixMark;
    if ((h & 0x7fffffff) < (1022 - unit) << 20) return 0;  // less than half a unit
    return (int64_t)neg_if((fix_mag(q, unit + 1) + 1) >> 1, h >> 31);
}

// The mark of a value's high word (a split or a plain word).
LSKUM_HD bool fix_marked(int32_t hi)
{
    return hi == INT32_MIN;
}

// The stored form of G: its two signed parts.
LSKUM_HD void split_g(int64_t g, int32_t &gh, int32_t &gl)
{
    gl = (int32_t)(uint32_t)g;
    gh = (int32_t)((g + 0x80000000ll) >> 32);
}
LSKUM_HD int64_t join_g(int32_t gh, int32_t gl)
{
    return ((int64_t)gh * 4294967296ll) + gl;
}

// Sum of products: weights wh + 2^-b wl with sum |wh| < 2^31 and sum |wl| <
// 2^31 (b: as many bits as that leaves, at most 28, which is a relative 2^-55
// for a weight of 1/16 of the sum), differences dh 2^32 + dl.
struct GradSum {
    int64_t hh, l, r, ll;
};
LSKUM_HD void grad_add(GradSum &s, int32_t wh, int32_t wl, int32_t dh, int32_t dl)
{
    s.hh += (int64_t)wh * dh;
    s.l += (int64_t)wh * dl;
    s.r += (int64_t)wl * dh;
    s.ll += (int64_t)wl * dl;
}
// The sum's part below hh, in units of 2^(32 - b) (the lanes of a point add
// these and hh; what is cut off is below 2^-25 of a unit of the result).
LSKUM_HD int64_t grad_low(const GradSum &s, int b)
{
    return (s.l >> (32 - b)) + s.r + (s.ll >> 32);
}
// The sum over the weights' unit 2^(p - 31), to the nearest unit; false if out of range.
LSKUM_HD bool grad_value(int64_t hh, int64_t low, int b, int p, int64_t &v)
{
    const int s = b - 1 - p;  // > 0
    v = (hh << (1 + p)) + ((low + (1ll << (s - 1))) >> s);
    const int64_t top = hh >> (60 - p);
    return top == 0 || top == -1;
}
LSKUM_HD bool grad_in_range(int64_t g)
{
    const int64_t top = g >> 62;
    return top == 0 || top == -1;
}

}  // namespace lskum
