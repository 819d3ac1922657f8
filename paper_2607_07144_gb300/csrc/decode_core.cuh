// Span decoding core shared by the bulk decoder, the random reads and the
// record reads (Sec. 1 "The code": the symbol is the cell holding the point,
// then p_{k-1} = (p_k - (1-r) V(c_k)) / r).
//
// The decoder never divides.  With m the span length and Q_k = r^(m-k) p_k,
//     Q_m = stored point,   Q_{k-1} = Q_k - (1-r) r^(m-k) V(c_k),
// and Q_0 = r^m p_0 must be back at the anchor (the origin).  Nearest-vertex
// classification of p_k (= cell containment for r <= r_N) is the argmax over
// c of p_k . V(c) because every vertex lies on the unit circle, and that is
// scale-free: argmax_c Q_k . V(c).  The margin of the true point to a cell
// boundary is about r^m in Q space at every step, so Q is kept in exact
// Q1.62 fixed point (int64, units of 2^-62) and the step is one table load
// of T[j][c] = round((1-r) r^j V(c) 2^62), j = m - k, and two subtractions.
//
// Classification takes an fp32 fast path with a certified margin and falls
// back to integer dot products in the rare near-boundary case: the high words
// of the 64x64->128-bit products, each dropping less than 2^-60, so a
// difference of two such dot products is off by less than 2^-59 (and by
// 2^-61 more from the vertices' Q1.62 rounding).  The decision it makes is
// the sign of Q . (V(a) - V(b)) for neighbouring vertices a, b, whose
// magnitude for a point of the true cell is at least
//     r^(m-1) (1 - cos(2 pi / N)) (1 - 2 r)
// (the point after the span's first symbol, (1 - r) V(c), is the closest
// case; a later point's own offset costs at most the factor 1 - 2 r).  With
// span lengths up to 44 / log2(1/r), r^(m-1) >= 2^-44 / r, and r_N ~ pi / N,
// that is at least about 2^-44 * 2 pi / N >= 2^-51.3 for every N <= 1024,
// 2^7 above the error (at N = 1024, L = 5 the bound is 2^-49.1, and that
// value is reached by alternating-neighbour spans):
//   * N = 4: the vertices are the axis directions, exact integer compares;
//   * N <= 8: fp32 scores q . V(c); exact scores when the best two are closer
//     than a bound far above the fp32 error;
//   * N > 8: Voronoi regions of the vertices are angular sectors, so the fp32
//     angle picks the sector; within twice the angle's error bound of a
//     boundary (the bound: 1.2e-5 rad for the arctangent polynomial plus
//     1.5e-6 rad for the fp32 direction, division and reflections, plus 5e-7
//     rad for the coefficients rounded in sector widths, plus N 2^-24 sector
//     widths for the scaling) the two neighbouring sectors are decided by the
//     sign of Q . (V(a) - V(b)).
#pragma once

#include <climits>
#include <type_traits>

#include "fkv_internal.h"

namespace fkvdec {

// atan u ~ u (a1 + a3 u^2 + a5 u^4 + a7 u^6 + a9 u^8) on [0, 1], from
// fit_atan.py: float32 Horner evaluation within 1.18e-5 rad of atan
constexpr float kAtan[5] = {9.998637438e-01f, -3.302824795e-01f, 1.800999194e-01f, -8.509350568e-02f,
                            2.082198113e-02f};

struct Tables {
    const longlong2 *T;   // [L][N] (x, y), shared memory
    const long long *vx;  // [N] V(c) in Q1.62, shared memory
    const long long *vy;
    const float2 *vf;     // [N] V(c) as float, shared memory
    int N;
    float sect_thr;       // sector test: |fraction| below this is decided in fp32
    float sect_a[5];      // kAtan in sector widths (times N / 2 pi)
    int sect_sh;          // floor(2^16 log2(1/r)): the scale of a walk's step
};

// Shared-memory footprint of the tables for (N, L).
__host__ __device__ inline int smem_bytes(int N, int L)
{
    return L * N * 16 + N * 16 + N * 8;
}

// Block-cooperative copy of the tables into `sm` (16-byte aligned).
__device__ inline Tables load(const fkv_decconst *__restrict__ g, const longlong2 *__restrict__ Tg, int N, int L,
                              uint8_t *sm)
{
    longlong2 *T = reinterpret_cast<longlong2 *>(sm);
    long long *vx = reinterpret_cast<long long *>(sm + L * N * 16);
    long long *vy = vx + N;
    float2 *vf = reinterpret_cast<float2 *>(sm + L * N * 16 + N * 16);
    for (int i = threadIdx.x; i < L * N; i += blockDim.x)
        T[i] = Tg[i];
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        vx[i] = g->vx[i];
        vy[i] = g->vy[i];
        vf[i] = make_float2(g->vfx[i], g->vfy[i]);
    }
    Tables t{T, vx, vy, vf, N, g->sect_thr, {}, g->sect_sh};
#pragma unroll
    for (int i = 0; i < 5; ++i)
        t.sect_a[i] = g->sect_a[i];
    return t;
}

// Q . V(c) in units of 2^-60: the high words of the two 128-bit products
// (the error bound is in the header comment).
__device__ __forceinline__ long long exact_dot(const Tables &t, long long X, long long Y, int c)
{
    return __mul64hi(X, t.vx[c]) + __mul64hi(Y, t.vy[c]);
}

static __device__ __noinline__ int classify_exact_all(const Tables &t, long long X, long long Y)
{
    int best = 0;
    long long bs = exact_dot(t, X, Y, 0);
    for (int c = 1; c < t.N; ++c) {
        const long long s = exact_dot(t, X, Y, c);
        if (s > bs) {
            bs = s;
            best = c;
        }
    }
    return best;
}

// fp32 image (qx, qy) of the direction of (X, Y): both scaled by one power of
// two that puts the larger magnitude's top bit at bit 62, then their high
// 32-bit words converted.  Relative to the larger magnitude the image is off
// by at most 2^-30 (the dropped low word) plus one fp32 rounding, like a
// direct conversion; only integer ops and 32-bit conversions are used,
// because 64-bit integer conversions issue at the FP64 rate on this GPU.
__device__ __forceinline__ void direction(long long X, long long Y, float &qx, float &qy)
{
    const unsigned long long ax = X < 0 ? 0ull - static_cast<unsigned long long>(X) : static_cast<unsigned long long>(X);
    const unsigned long long ay = Y < 0 ? 0ull - static_cast<unsigned long long>(Y) : static_cast<unsigned long long>(Y);
    const int sh = max(__clzll(static_cast<long long>(ax | ay)) - 1, 0);
    const unsigned long long xs = static_cast<unsigned long long>(X) << sh;
    const unsigned long long ys = static_cast<unsigned long long>(Y) << sh;
    qx = __int2float_rn(static_cast<int>(static_cast<unsigned>(xs >> 32)));
    qy = __int2float_rn(static_cast<int>(static_cast<unsigned>(ys >> 32)));
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The angle of direction (qx, qy) in sector widths, in [-N/2, N/2]: octant
// reduction to u in [0, 1], atan u (coefficients k, in sector widths) from the
// odd polynomial of fit_atan.py, the octant's reflections.  No subnormal or
// huge coordinates; the larger one is at least `least`, or both are zero.
__device__ __forceinline__ float sector_angle(int N, const float *k, float qx, float qy, float least)
{
    const float ax = fabsf(qx), ay = fabsf(qy);
    const float u = fminf(ax, ay) * rcp_approx(fmaxf(fmaxf(ax, ay), least));
    const float u2 = u * u;
    float a = u * fmaf(fmaf(fmaf(fmaf(k[4], u2, k[3]), u2, k[2]), u2, k[1]), u2, k[0]);
    if (ay > ax)
        a = 0.25f * static_cast<float>(N) - a;
    if (qx < 0.0f)
        a = 0.5f * static_cast<float>(N) - a;
    return copysignf(a, qy);
}

// The sector, by adding 1.5 2^23; f receives the distance to its centre.
__device__ __forceinline__ int sector_of(int N, const float *k, float qx, float qy, float least, float &f)
{
    const float a = sector_angle(N, k, qx, qy, least);
    const float big = a + 12582912.0f;
    f = a - (big - 12582912.0f);               // in [-0.5, 0.5]
    const int c = __float_as_int(big) - 0x4B400000;
    return c < 0 ? c + N : c;
}

// The sector of (X, Y), imaged by the integers (qx, qy).
__device__ __forceinline__ int classify_sector(const Tables &t, long long X, long long Y, float qx, float qy)
{
    float f;
    const int N = t.N, c = sector_of(N, t.sect_a, qx, qy, 1.0f, f);
    // away from a sector boundary by more than the angle's error allows
    if (fabsf(f) < t.sect_thr)
        return c;
    // else the nearer of the two sectors by exact products
    const int c1 = f > 0.0f ? (c + 1 < N ? c + 1 : 0) : (c > 0 ? c - 1 : N - 1);
    const long long d = exact_dot(t, X, Y, c) - exact_dot(t, X, Y, c1);
    return d > 0 ? c : (d < 0 ? c1 : min(c, c1));
}

__device__ __forceinline__ int classify_axes(long long X, long long Y)
{
    const long long ax = X < 0 ? -X : X, ay = Y < 0 ? -Y : Y;
    if (ax >= ay)
        return X >= 0 ? 0 : 2;
    return Y >= 0 ? 1 : 3;
}

template <int N>
__device__ __forceinline__ int classify_scores(const Tables &t, long long X, long long Y)
{
    float qx, qy;
    direction(X, Y, qx, qy);
    float b1 = -INFINITY, b2 = -INFINITY;
    int bi = 0;
#pragma unroll
    for (int c = 0; c < N; ++c) {
        const float s = fmaf(qx, t.vf[c].x, qy * t.vf[c].y);
        b2 = fmaxf(b2, fminf(s, b1));
        bi = s > b1 ? c : bi;
        b1 = fmaxf(b1, s);
    }
    if (b1 - b2 > 0x1p-18f * (fabsf(qx) + fabsf(qy)))
        return bi;
    return classify_exact_all(t, X, Y);
}

__device__ __forceinline__ int classify_angle(const Tables &t, long long X, long long Y)
{
    float qx, qy;
    direction(X, Y, qx, qy);
    return classify_sector(t, X, Y, qx, qy);
}

// round(v * 2^62) to nearest, saturated to int64 (NaN gives INT64_MIN), from
// the binary64 fields with integer ops: v = m 2^(e - 1075), so v 2^62 =
// m 2^10 / 2^(1023 - e), and m 2^10 < 2^63 leaves room for half a unit.
__device__ __forceinline__ long long to_q62(double v)
{
    const long long b = __double_as_longlong(v);
    const unsigned long long frac = static_cast<unsigned long long>(b) & 0xFFFFFFFFFFFFFull;
    const int k = 1023 - static_cast<int>((b >> 52) & 0x7FF);
    if (k < 0) {                               // |v| >= 2, infinity or NaN
        if (k == -1024 && frac)
            return LLONG_MIN;
        return b < 0 ? LLONG_MIN : LLONG_MAX;
    }
    // (m 2^10 + 2^k / 2) >> k; PTX shifts by 64 and more give zero, as does
    // the zero and subnormal exponent (k = 1023)
    unsigned long long mag;
    asm("{\n\t.reg .b64 h;\n\t"
        "shl.b64 h, %2, %3;\n\t"
        "shr.u64 h, h, 1;\n\t"
        "add.u64 h, h, %1;\n\t"
        "shr.u64 %0, h, %3;\n\t}"
        : "=l"(mag)
        : "l"((frac | (1ull << 52)) << 10), "l"(1ull), "r"(k));
    return b < 0 ? -static_cast<long long>(mag) : static_cast<long long>(mag);
}

// Decode `steps` symbols backward from Q (the span's stored point in Q1.62):
// step j = 0 .. steps-1 emits the symbol at offset m-1-j of the span.
// `emit(j, c)` receives each symbol.  Any Q, of any size: random reads,
// retrieval, and spans that are no code point.  UNROLL steps of the loop (0: the
// compiler's choice): random reads of N <= 8 take few, since their lanes walk
// different numbers of steps and part ways in the remainder of an unrolled loop.
// 4.2 M reads of N = 4, spans of 8: 64 us by two steps, 88 as the compiler
// unrolls it; of 44: 209 and 214.  NC: the alphabet's size where it is known, 0 else.
template <int UNROLL, int NC, class Classify, class Emit>
__device__ __forceinline__ void walk_by(const Tables &t, long long &X, long long &Y, int steps, Classify classify,
                                        Emit emit)
{
    const longlong2 *T = t.T;
    auto step = [&](int j) {
        const int c = classify(X, Y);
        emit(j, c);
        const longlong2 w = T[c];
        X = static_cast<long long>(static_cast<unsigned long long>(X) - static_cast<unsigned long long>(w.x));
        Y = static_cast<long long>(static_cast<unsigned long long>(Y) - static_cast<unsigned long long>(w.y));
        T += NC > 0 ? NC : t.N;
    };
    if constexpr (UNROLL > 0) {
#pragma unroll UNROLL
        for (int j = 0; j < steps; ++j)
            step(j);
    } else {
        for (int j = 0; j < steps; ++j)
            step(j);
    }
}

// The cell test of an alphabet: sectors (N > 8), the axes (N = 4), scores.
enum Cell { kSectors, kAxes, kScores };

template <Cell CELL, int UNROLL = 0, class Emit>
__device__ __forceinline__ void walk(const Tables &t, long long &X, long long &Y, int steps, Emit emit)
{
    if (CELL == kSectors) {
        walk_by<UNROLL, 0>(t, X, Y, steps, [&](long long x, long long y) { return classify_angle(t, x, y); }, emit);
    } else if (CELL == kAxes) {
        walk_by<UNROLL, 4>(t, X, Y, steps, [](long long x, long long y) { return classify_axes(x, y); }, emit);
    } else {
        auto scores = [&](auto n) {
            walk_by<UNROLL, n.value>(
                t, X, Y, steps, [&](long long x, long long y) { return classify_scores<n.value>(t, x, y); }, emit);
        };
        switch (t.N) {
        case 3: scores(std::integral_constant<int, 3>()); break;
        case 5: scores(std::integral_constant<int, 5>()); break;
        case 6: scores(std::integral_constant<int, 6>()); break;
        case 7: scores(std::integral_constant<int, 7>()); break;
        default: scores(std::integral_constant<int, 8>()); break;
        }
    }
}

// The walk of a random read, by the steps that its cell test's loop unrolls best
// (sectors: 1 M reads of N = 64 29 us, 31 rolled; of N = 1024 in a ragged batch of
// 20,000 streams 39.4, 51.3 rolled; scores: 4.2 M reads of N = 8, spans of 2, 66 us
// rolled, 80 by two steps).
template <Cell CELL, class Emit>
__device__ __forceinline__ void walk_read(const Tables &t, long long &X, long long &Y, int steps, Emit emit)
{
    walk<CELL, CELL == kSectors ? 0 : CELL == kAxes ? 2 : 1>(t, X, Y, steps, emit);
}

template <class Emit>
static __device__ __noinline__ void walk_any(const Tables &t, long long &X, long long &Y, int steps, Emit emit)
{
    walk<kSectors>(t, X, Y, steps, emit);
}

// The walk of a code point for N > 8, where Voronoi regions are sectors.  A
// code point's scale is known: |p_k| is in [1 - 2r, 1] (each p_k = V(c) +
// r (p_{k-1} - V(c))), so step j's Q is within r^j [1 - 2r, 1] and a shift by
// floor(j log2(1/r)) puts its magnitude in (0.24, 1] of the full scale (1 - 2r
// >= 0.48 for N >= 9).  The direction is then one shift of each coordinate's
// words and a 32-bit conversion, off by less than 2^-28 of its length.
// Bound: instruction issue (62 % issue active; 88 instructions a symbol with
// the span's set-up and stores).  50.3 M symbols of 6-symbol spans decode in
// 0.170 ms; 0.216 ms with the magnitude found by leading-zero counts, two
// 64-bit shifts, a division with its range cases and conversions for the
// rounding (the planar decoder 0.089 against 0.119 ms for 25.1 M).
// A Q that is no code point gets symbols of some kind (always in [0, N)) and
// fails the anchor check: no other point is within 2^-4 r^m of the sum of the
// steps taken.
template <class Emit>
__device__ __forceinline__ void walk_sectors(const Tables &t, long long &X, long long &Y, int steps, Emit emit)
{
    const longlong2 *T = t.T;
    int sh16 = 0;
    for (int j = 0; j < steps; ++j, T += t.N, sh16 += t.sect_sh) {
        const int sh = sh16 >> 16;
        const float qx = __int2float_rn(static_cast<int>((static_cast<unsigned long long>(X) << sh) >> 32));
        const float qy = __int2float_rn(static_cast<int>((static_cast<unsigned long long>(Y) << sh) >> 32));
        const int c = classify_sector(t, X, Y, qx, qy);
        emit(j, c);
        const longlong2 w = T[c];
        X = static_cast<long long>(static_cast<unsigned long long>(X) - static_cast<unsigned long long>(w.x));
        Y = static_cast<long long>(static_cast<unsigned long long>(Y) - static_cast<unsigned long long>(w.y));
    }
}

// Decode the m symbols of the span stored as p.  start() gives the receiver
// emit(j, c) of a walk from its beginning; false when the walk does not end at
// the anchor (|Q_0| <= lim), the symbols then being those of the general walk.
// The decoders and random reads are compiled for each cell test.  With all of
// them in one kernel, chosen at each symbol, 134 M symbols took 0.402 ms for
// N = 3 (0.318 now), 0.224 for N = 4 (0.170), 0.672 for N = 8 (0.517), 0.416 for
// N = 256 (0.412); 4.2 M random reads 0.648 / 0.297 / 0.459 / 0.111 (0.418 /
// 0.219 / 0.377 / 0.100).
template <Cell CELL, class Start>
__device__ __forceinline__ bool decode_point(const Tables &t, double2 p, int m, long long lim, Start start)
{
    long long X = to_q62(p.x), Y = to_q62(p.y);
    auto off = [&] { return X > lim || X < -lim || Y > lim || Y < -lim; };
    if (CELL != kSectors) {
        walk<CELL>(t, X, Y, m, start());
        return !off();
    }
    walk_sectors(t, X, Y, m, start());
    if (!off())
        return true;
    long long X2 = to_q62(p.x), Y2 = to_q62(p.y);
    walk_any(t, X2, Y2, m, start());
    return false;
}

}  // namespace fkvdec
