// Span codec kernels: the iterated-map code of Sec. 1 "The code", applied
// span-parallel (one span per thread) for encoding, decoding, random reads
// and tail appends (Sec. 2, Table 1).
//
// Encoding must reproduce the binary64 walk bit for bit, with explicit
// round-to-nearest operations (no FMA contraction): d = p - V(c); t = r * d;
// p = V(c) + t per coordinate.  The FP64 pipe (two lanes a clock per SM)
// bounds it, so the bulk encoders keep off that pipe what they can: the first
// symbols of a span come from a table, and the product runs on the integer
// pipe (or, for r = 1/2, not at all).
//
// Decoding only has to recover the symbols, so it runs in exact 64-bit
// fixed point (Q1.62) on the integer pipes with no division at all (see
// decode_core.cuh).
#include <string.h>

#include <type_traits>

#include "decode_core.cuh"

namespace {

constexpr int kThreads = 256;   // spans per block
constexpr int kMaxSpan = 44;    // floor(44 / log2(1/r)) with r <= 1/2

// Symbols are uint8 for alphabets N <= 256 and uint16 up to FKV_MAX_N; every
// kernel that touches symbols is instantiated for both.
template <typename Sym>
__host__ __device__ constexpr int stage_bytes() { return kThreads * kMaxSpan * static_cast<int>(sizeof(Sym)) + 32; }
// Block size of the bulk decoders: 256 spans per chunk for uint8 symbols; for
// uint16 (N up to 1024, 104 KB of decoder tables per block) one 1024-thread
// block per SM shares the tables.
template <typename Sym>
__host__ __device__ constexpr int dec_threads() { return sizeof(Sym) == 1 ? 256 : 1024; }
// Shared staging of one decoded chunk: dec_threads spans of L symbols plus
// the 16-byte realignment slack.
template <typename Sym>
__host__ __device__ inline int dec_stage_bytes(int L)
{
    return (dec_threads<Sym>() * L * static_cast<int>(sizeof(Sym)) + 32 + 15) & ~15;
}
template <typename Sym>
__host__ __device__ constexpr int vtab_len() { return sizeof(Sym) == 1 ? 256 : FKV_MAX_N; }

// Copy len bytes from global src into shared buf so that buf[off + i] =
// src[i], off = src mod 16: aligned 16-byte vectors inside the range, single
// bytes at the two ragged ends.  Never touches bytes outside [src, src+len).
__device__ __forceinline__ int stage_in(uint8_t *buf, const uint8_t *src, int len)
{
    const int off = static_cast<int>(reinterpret_cast<uintptr_t>(src) & 15);
    const uint8_t *a = src - off;
    const int total = off + len;
    const int nv = (total + 15) >> 4;
    for (int v = threadIdx.x; v < nv; v += blockDim.x) {
        const int b0 = v << 4;
        if (b0 >= off && b0 + 16 <= total) {
            *reinterpret_cast<uint4 *>(buf + b0) = __ldg(reinterpret_cast<const uint4 *>(a + b0));
        } else {
            const int lo = b0 > off ? b0 : off;
            const int hi = b0 + 16 < total ? b0 + 16 : total;
            for (int q = lo; q < hi; ++q)
                buf[q] = a[q];
        }
    }
    return off;
}

// The mirror of stage_in: dst[i] = buf[off + i], off = dst mod 16.
__device__ __forceinline__ void stage_out(uint8_t *dst, const uint8_t *buf, int len, int off)
{
    uint8_t *a = dst - off;
    const int total = off + len;
    const int nv = (total + 15) >> 4;
    for (int v = threadIdx.x; v < nv; v += blockDim.x) {
        const int b0 = v << 4;
        if (b0 >= off && b0 + 16 <= total) {
            *reinterpret_cast<uint4 *>(a + b0) = *reinterpret_cast<const uint4 *>(buf + b0);
        } else {
            const int lo = b0 > off ? b0 : off;
            const int hi = b0 + 16 < total ? b0 + 16 : total;
            for (int q = lo; q < hi; ++q)
                a[q] = buf[q];
        }
    }
}

// stage_out by one warp.
__device__ __forceinline__ void stage_out_warp(uint8_t *dst, const uint8_t *buf, int len, int off)
{
    uint8_t *a = dst - off;
    const int total = off + len;
    const int nv = (total + 15) >> 4;
    for (int v = threadIdx.x & 31; v < nv; v += 32) {
        const int b0 = v << 4;
        if (b0 >= off && b0 + 16 <= total) {
            *reinterpret_cast<uint4 *>(a + b0) = *reinterpret_cast<const uint4 *>(buf + b0);
        } else {
            const int lo = b0 > off ? b0 : off;
            const int hi = b0 + 16 < total ? b0 + 16 : total;
            for (int q = lo; q < hi; ++q)
                a[q] = buf[q];
        }
    }
}

// Sec. 1 forward map for a run of symbols from (x, y), binary64, no FMA.
// A symbol >= N takes a NaN vertex, so its span's point comes out NaN.
template <typename Sym>
__device__ __forceinline__ double2 encode_span(const Sym *s, int m, const double2 *sV, int N, double r,
                                               double x, double y)
{
    for (int k = 0; k < m; ++k) {
        const unsigned c = s[k];
        const double2 v = c < static_cast<unsigned>(N) ? sV[c] : make_double2(__longlong_as_double(-1ll),
                                                                              __longlong_as_double(-1ll));
        const double dx = __dsub_rn(x, v.x);
        const double dy = __dsub_rn(y, v.y);
        const double tx = __dmul_rn(r, dx);
        const double ty = __dmul_rn(r, dy);
        x = __dadd_rn(v.x, tx);
        y = __dadd_rn(v.y, ty);
    }
    return make_double2(x, y);
}

// What the bulk encoders use of a context.
struct EncArgs {
    const double2 *V;     // [N]
    const double2 *pre;   // [N^pre_k] the point after pre_k symbols from the anchor, first symbol most significant
    int N, L, pre_k;
    double r;
};

// Calls, so that the compiler does not run the rare case for every lane.
static __device__ __noinline__ double mul_fp64(double a, double b) { return __dmul_rn(a, b); }
static __device__ __noinline__ double mul_add_fp64(double r, double d, double v)
{
    return __dadd_rn(v, __dmul_rn(r, d));
}
static __device__ __noinline__ long long floor_fp64(double x) { return __double2ll_rd(x); }

// r d rounded to nearest even, as __dmul_rn(r, d), on the integer pipe: the
// 53-bit mantissas, aligned to the top of 64 bits, multiply to a 128-bit
// product whose upper word is rounded at its 53rd bit (the lower word only as
// a sticky bit).  r is a normal number with mantissa word m11 (shifted left by
// 11) and exponent field er.  Far-out exponents (zero, subnormal, huge, NaN)
// take the FP64 product.  About 30 instructions, while a binary64 operation
// holds its pipe for 16 clocks, 64 issue slots of the SM.
struct RatioMul {
    double r;
    unsigned long long m11;
    int er;
    __device__ __forceinline__ explicit RatioMul(double r_) : r(r_)
    {
        const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(r_));
        m11 = (b << 11) | (1ull << 63);
        er = static_cast<int>(b >> 52);
    }
    // The rounded mantissa of r d, 2^52 .. 2^53, and *top, the product's
    // top bit: |r d| = mantissa 2^(e + er + top - 2098), e d's exponent field.
    __device__ __forceinline__ unsigned long long mantissa(unsigned hi, unsigned lo, int &top) const
    {
        const unsigned dh = __funnelshift_l(lo, hi, 11) | 0x80000000u, dl = lo << 11;
        const unsigned rh = static_cast<unsigned>(m11 >> 32), rl = static_cast<unsigned>(m11);
        const unsigned long long p00 = static_cast<unsigned long long>(dl) * rl;
        const unsigned long long a = static_cast<unsigned long long>(dh) * rl + (p00 >> 32);
        const unsigned long long b = static_cast<unsigned long long>(dl) * rh + static_cast<unsigned>(a);
        unsigned long long h = static_cast<unsigned long long>(dh) * rh + (a >> 32) + (b >> 32);
        h |= (static_cast<unsigned>(b) | static_cast<unsigned>(p00)) != 0u ? 1ull : 0ull;
        top = static_cast<int>(h >> 63);
        const int drop = 10 + top;
        const unsigned odd = (static_cast<unsigned>(h) >> drop) & 1u;
        h += (512u << top) - 1u + odd;
        return h >> drop;
    }
    __device__ __forceinline__ double operator()(double d) const
    {
        const unsigned hi = static_cast<unsigned>(__double2hiint(d)), lo = static_cast<unsigned>(__double2loint(d));
        const int e = static_cast<int>((hi >> 20) & 0x7FFu);
        if (static_cast<unsigned>(e - 512) >= 588u)
            return mul_fp64(r, d);
        int top;
        const unsigned long long h = mantissa(hi, lo, top);
        const unsigned th = static_cast<unsigned>(h >> 32) + (static_cast<unsigned>(e + er - 1024 + top) << 20);
        return __hiloint2double(static_cast<int>(th | (hi & 0x80000000u)), static_cast<int>(static_cast<unsigned>(h)));
    }
    // v + r d, both operations rounded to nearest even, for |v| in [0.7, 1]:
    // the sum as well on the integer pipe, in units of 2^-62.  v is a whole
    // number of them; the product, below 1/2, keeps in its last bit whether
    // bits under it were dropped, and since the sum is above 1/8 at least six
    // bits lie between that bit and the place of rounding, which it therefore
    // never turns.  Larger and far smaller products take the FP64 operations.
    __device__ __forceinline__ double plus(double v, double d) const
    {
        const unsigned hi = static_cast<unsigned>(__double2hiint(d)), lo = static_cast<unsigned>(__double2loint(d));
        int top;
        const unsigned long long h = mantissa(hi, lo, top);
        const unsigned sh = 2044u - (((hi >> 20) & 0x7FFu) + static_cast<unsigned>(er + top));
        if (sh > 63u)
            return mul_add_fp64(r, d, v);
        const unsigned long long w = h << 8;
        unsigned long long t = w >> sh;
        t |= t << sh != w ? 1ull : 0ull;
        const unsigned vhi = static_cast<unsigned>(__double2hiint(v)), vlo = static_cast<unsigned>(__double2loint(v));
        const unsigned long long vm = static_cast<unsigned long long>((vhi & 0xFFFFFu) | 0x100000u) << 32 | vlo;
        unsigned long long q = vm << (((vhi >> 20) & 0x7FFu) - 1013u);
        q = static_cast<int>(vhi ^ hi) < 0 ? q - t : q + t;
        const int lz = __clz(static_cast<int>(static_cast<unsigned>(q >> 32))) - 1;   // 0 .. 3
        q <<= lz;
        q += 511u + ((static_cast<unsigned>(q) >> 10) & 1u);
        q >>= 10;
        const unsigned qh = static_cast<unsigned>(q >> 32) + (static_cast<unsigned>(1022 - lz) << 20);
        return __hiloint2double(static_cast<int>(qh | (vhi & 0x80000000u)), static_cast<int>(static_cast<unsigned>(q)));
    }
};

// Shared vertex table of the bulk encoders: for r = 1/2 the multiples 2^j V(c)
// at [j N + c], j = 0 .. L; else V(c) with the larger coordinate first, and
// whether that is y.
template <bool HALF, typename Sym>
struct EncTable {
    double2 v[HALF ? 4 * (kMaxSpan + 1) : vtab_len<Sym>()];
    uint8_t turned[HALF ? 16 : vtab_len<Sym>()];
    __device__ __forceinline__ void load(const EncArgs &a)
    {
        if (HALF) {
            for (int i = threadIdx.x; i < (a.L + 1) * a.N; i += blockDim.x) {
                const double2 p = a.V[i % a.N];
                const double up = __longlong_as_double(static_cast<long long>(1023 + i / a.N) << 52);
                v[i] = make_double2(p.x * up, p.y * up);
            }
        } else {
            for (int i = threadIdx.x; i < a.N; i += blockDim.x) {
                const double2 p = a.V[i];
                const bool turn = (__double2hiint(p.y) & 0x7FFFFFFF) > (__double2hiint(p.x) & 0x7FFFFFFF);
                v[i] = turn ? make_double2(p.y, p.x) : p;
                turned[i] = turn;
            }
        }
    }
};

// The vertices as they are (encode_few).
template <typename Sym>
struct PlainTable {
    double2 v[vtab_len<Sym>()];
    __device__ __forceinline__ void load(const EncArgs &a)
    {
        for (int i = threadIdx.x; i < a.N; i += blockDim.x)
            v[i] = a.V[i];
    }
};

// One span from the anchor: its first pre_k symbols from the table, the rest
// walked, the product on the integer pipe.  With r = 1/2 (HALF) the product
// is exact, and the walk keeps S = 2^j p (scaling by powers of two commutes
// with the roundings): S <- 2^(j+1) V + (S - 2^j V), two operations a
// coordinate.  Else the sum in the vertex's larger coordinate (at least
// cos(pi/4) of its unit length) is on the integer pipe too: three FP64
// operations a symbol, the point's coordinates turned to the vertex's order.
template <bool HALF, typename Sym>
__device__ __forceinline__ double2 encode_anchored(const Sym *s, int m, const EncTable<HALF, Sym> &tab,
                                                   const EncArgs &a, const RatioMul &mul)
{
    const unsigned N = static_cast<unsigned>(a.N);
    double x = 0.0, y = 0.0;
    bool bad = false;
    int k = 0;
    if (m >= a.pre_k) {
        unsigned at = 0;
        for (; k < a.pre_k; ++k) {
            const unsigned c = s[k];
            bad |= c >= N;
            at = at * N + c;
        }
        if (!bad) {
            const double2 p = __ldg(&a.pre[at]);
            x = p.x;
            y = p.y;
        }
    }
    if (HALF) {
        const double up = __longlong_as_double(static_cast<long long>(1023 + k) << 52);
        x = __dmul_rn(x, up);
        y = __dmul_rn(y, up);
    }
    unsigned turned = 0;
    for (; k < m; ++k) {
        unsigned c = s[k];
        bad |= c >= N;
        c = min(c, N - 1);
        if (HALF) {
            const double2 v = tab.v[k * N + c], w = tab.v[(k + 1) * N + c];
            x = __dadd_rn(w.x, __dsub_rn(x, v.x));
            y = __dadd_rn(w.y, __dsub_rn(y, v.y));
        } else {
            const double2 v = tab.v[c];
            const unsigned f = tab.turned[c];
            const bool turn = f != turned;
            turned = f;
            const double u = turn ? y : x, w = turn ? x : y;
            x = mul.plus(v.x, __dsub_rn(u, v.x));
            y = __dadd_rn(v.y, mul(__dsub_rn(w, v.y)));
        }
    }
    if (turned) {
        const double u = x;
        x = y;
        y = u;
    }
    if (HALF) {
        const double down = __longlong_as_double(static_cast<long long>(1023 - m) << 52);
        x = __dmul_rn(x, down);
        y = __dmul_rn(y, down);
    }
    const double nan = __longlong_as_double(-1ll);
    return bad ? make_double2(nan, nan) : make_double2(x, y);
}

// The same by the plain walk after the table's symbols, for few spans: with up
// to four warps on an SM its FP64 pipe keeps up, and a binary64 operation's
// latency is less than that of its integer form.
template <typename Sym>
__device__ __forceinline__ double2 encode_few(const Sym *s, int m, const double2 *V, const EncArgs &a)
{
    const unsigned N = static_cast<unsigned>(a.N);
    double x = 0.0, y = 0.0;
    bool bad = false;
    int k = 0;
    if (a.pre_k > 2 && m >= a.pre_k) {         // one or two symbols: no slower walked than looked up
        unsigned at = 0;
        for (; k < a.pre_k; ++k) {
            const unsigned c = s[k];
            bad |= c >= N;
            at = at * N + c;
        }
        if (!bad) {
            const double2 p = __ldg(&a.pre[at]);
            x = p.x;
            y = p.y;
        }
    }
    for (; k < m; ++k) {
        unsigned c = s[k];
        bad |= c >= N;
        c = min(c, N - 1);
        const double2 v = V[c];
        x = __dadd_rn(v.x, __dmul_rn(a.r, __dsub_rn(x, v.x)));
        y = __dadd_rn(v.y, __dmul_rn(a.r, __dsub_rn(y, v.y)));
    }
    const double nan = __longlong_as_double(-1ll);
    return bad ? make_double2(nan, nan) : make_double2(x, y);
}

// Spans a block (and so an SM) up to which encode_few is used.  Streams of 40
// spans, one alone, us by it and by the integer product (and by the whole walk
// in binary64, as it once was): N = 7 8.5 / 12.5 (8.6), N = 16 6.4 / 8.4 (6.4), N = 256
// 4.4 / 5.2 (4.4); 192 and 256 spans in one block: N = 9 10.5 / 10.6, 12.5 / 10.6.
constexpr int kFewSpans = 128;

// The table of points after k symbols from the anchor: entry i's symbols are
// i's k digits to the base N, the first one most significant.
__global__ void __launch_bounds__(kThreads) k_pre_table(const double2 *__restrict__ V, int N, double r, int k,
                                                        int count, double2 *__restrict__ pre)
{
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= count)
        return;
    uint16_t s[16];
    int rest = i;
    for (int j = k - 1; j >= 0; --j) {
        s[j] = static_cast<uint16_t>(rest % N);
        rest /= N;
    }
    pre[i] = encode_span(s, k, V, N, r, 0.0, 0.0);
}

// Bulk encoding, one span per thread.  Bound by the FP64 pipe and, a quarter
// below it, by instruction issue: three binary64 operations for each symbol
// after the table's, so (6 - 2) 3 = 12 a span for N = 256 where the plain walk
// takes 36.  128 streams of 392,784 symbols: 0.226 ms; 0.593 ms by the plain
// walk, 0.397 with the table, 0.278 with the products on the integer pipe too,
// 0.234 with all but the NaN and table comparisons off the FP64 pipe.
// Persistent blocks with warp-wide staging: 0.258.  16.8 M ragged symbols of
// N = 16: 0.091 ms against 0.204.
template <bool HALF, typename Sym>
__global__ void __launch_bounds__(kThreads)
k_span_encode(const Sym *__restrict__ sym, int64_t n, int64_t sym_stride, int64_t spans, int bps,
              double2 *__restrict__ pts, int64_t pt_stride, const EncArgs a, unsigned *status)
{
    __shared__ __align__(16) uint8_t sbuf[stage_bytes<Sym>()];
    __shared__ EncTable<HALF, Sym> tab;
    const int L = a.L;
    const int64_t stream = blockIdx.x / bps;
    const int64_t s0 = static_cast<int64_t>(blockIdx.x % bps) * kThreads;
    tab.load(a);
    const int64_t b = s0 * L;
    const int64_t e = min(n, (s0 + kThreads) * L);
    const int off = stage_in(sbuf, reinterpret_cast<const uint8_t *>(sym + stream * sym_stride + b),
                             static_cast<int>(e - b) * static_cast<int>(sizeof(Sym)));
    __syncthreads();
    const int64_t s = s0 + threadIdx.x;
    if (s < spans) {
        const int m = static_cast<int>(min(static_cast<int64_t>(L), n - s * L));
        const Sym *my = reinterpret_cast<const Sym *>(sbuf + off) + threadIdx.x * L;
        const double2 p = encode_anchored<HALF>(my, m, tab, a, RatioMul(a.r));
        if (__double2hiint(p.x) == -1)   // NaN: a symbol >= N
            atomicOr(status, FKV_ST_CORRUPT);
        pts[stream * pt_stride + s] = p;
    }
}

// The same for many short streams (a decode step's append): the threads count
// through all streams' spans, so that a block, its table load and its warps
// serve up to as many spans as it has threads, and read their symbols in
// place; few spans spread over the SMs (per_block of a block's threads take
// one).  2,048 streams of 48 symbols: 4.6 us; 6.3 with 256 spans to every block,
// 10.5 with a block (and its table load) a stream.  From half a block's spans
// on, many streams lose little by a block a stream; few are shared out all the
// same (one of 1,000 spans, N = 16: 6.5 us, 8.5 by its own four blocks).
template <bool HALF, bool FEW, typename Sym>
__global__ void __launch_bounds__(kThreads)
k_span_encode_flat(const Sym *__restrict__ sym, int64_t n, int64_t sym_stride, unsigned spans, unsigned total,
                   unsigned per_block, fkvd::FastDiv div_spans, double2 *__restrict__ pts, int64_t pt_stride,
                   const EncArgs a, unsigned *status)
{
    __shared__ typename std::conditional<FEW, PlainTable<Sym>, EncTable<HALF, Sym>>::type tab;
    tab.load(a);
    __syncthreads();
    const unsigned t = blockIdx.x * per_block + threadIdx.x;
    if (threadIdx.x >= per_block || t >= total)
        return;
    const unsigned stream = div_spans.div(t), s = t - stream * spans;
    const int64_t b = static_cast<int64_t>(s) * a.L;
    const int m = static_cast<int>(min(static_cast<int64_t>(a.L), n - b));
    const Sym *my = sym + stream * sym_stride + b;
    double2 p;
    if constexpr (FEW)
        p = encode_few(my, m, tab.v, a);
    else
        p = encode_anchored<HALF>(my, m, tab, a, RatioMul(a.r));
    if (__double2hiint(p.x) == -1)   // NaN: a symbol >= N
        atomicOr(status, FKV_ST_CORRUPT);
    pts[stream * pt_stride + s] = p;
}

// ------------------------------------------------------------- decoding
// (arithmetic in decode_core.cuh: exact Q1.62 walk, no division)

__host__ __device__ inline int tables_bytes(int N, int L)
{
    return (fkvdec::smem_bytes(N, L) + 15) & ~15;
}

// A persistent block's chunk (stream, span block), chunk = stream * bps +
// block, stepped gridDim.x chunks at a time without a division per step: the
// whole streams and remaining blocks of one step are worked out once.
struct ChunkWalk {
    int64_t stream, sb;
    unsigned dq, dr, bps;
    __device__ explicit ChunkWalk(int bps_) : bps(static_cast<unsigned>(bps_))
    {
        stream = blockIdx.x / bps;
        sb = blockIdx.x - static_cast<unsigned>(stream) * bps;
        dq = gridDim.x / bps;
        dr = gridDim.x - dq * bps;
    }
    __device__ void next()
    {
        sb += dr;
        stream += dq;
        if (sb >= bps) {
            sb -= bps;
            ++stream;
        }
    }
};

// Persistent: a block loads the decoder tables once and walks chunks of
// dec_threads spans (chunk = stream * bps + span block), blockIdx.x,
// + gridDim.x, ...; each thread stores its span's symbols directly, so the
// chunks need no block barrier.
template <typename Sym, fkvdec::Cell CELL>
__global__ void __launch_bounds__(dec_threads<Sym>())
k_span_decode(const double2 *__restrict__ pts, int64_t n, int64_t pt_stride, int64_t spans, int bps,
              int64_t n_chunks, Sym *__restrict__ sym, int64_t sym_stride, const fkv_decconst *__restrict__ dc,
              const longlong2 *__restrict__ T, int N, int L, unsigned *status)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    const fkvdec::Tables t = fkvdec::load(dc, T, N, L, dsm);
    __syncthreads();
    constexpr int TPB = dec_threads<Sym>();
    ChunkWalk w(bps);
    auto point = [&](const ChunkWalk &c, bool more) {     // this thread's point of a chunk, loaded a chunk ahead
        const int64_t s = c.sb * TPB + threadIdx.x;
        return more && s < spans ? __ldg(&pts[c.stream * pt_stride + s]) : make_double2(0.0, 0.0);
    };
    double2 p = point(w, blockIdx.x < n_chunks);
    for (int64_t ck = blockIdx.x; ck < n_chunks; ck += gridDim.x) {
        const int64_t s = w.sb * TPB + threadIdx.x;
        Sym *dst = sym + w.stream * sym_stride + s * L;
        w.next();
        const double2 pn = point(w, ck + gridDim.x < n_chunks);
        if (s < spans) {
            const int m = static_cast<int>(min(static_cast<int64_t>(L), n - s * L));
            dst += m - 1;
            if (!fkvdec::decode_point<CELL>(t, p, m, __ldg(&dc->alim[m]), [&] {
                    return [=](int j, int c) { dst[-j] = static_cast<Sym>(c); };
                }))
                atomicOr(status, FKV_ST_CORRUPT);
        }
        p = pn;
    }
}

// Decode 256 spans of one stream (chunk `ck` of the n_streams * bps chunks)
// into sbuf (one span per thread, symbol i of the chunk at sbuf[i]).
template <fkvdec::Cell CELL, typename Sym>
__device__ __forceinline__ void decode_chunk(const fkvdec::Tables &t, const double2 *__restrict__ pts, int64_t n,
                                             int64_t pt_stride, int64_t spans, int64_t stream, int64_t s0,
                                             Sym *sbuf, const fkv_decconst *__restrict__ dc, int L,
                                             unsigned *status)
{
    const int64_t s = s0 + threadIdx.x;
    if (s < spans) {
        const int m = static_cast<int>(min(static_cast<int64_t>(L), n - s * L));
        Sym *my = sbuf + threadIdx.x * L + m - 1;
        if (!fkvdec::decode_point<CELL>(t, pts[stream * pt_stride + s], m, __ldg(&dc->alim[m]), [&] {
                return [=](int j, int c) { my[-j] = static_cast<Sym>(c); };
            }))
            atomicOr(status, FKV_ST_CORRUPT);
    }
}

// The stream decode for long spans (more than 8 symbols): a chunk's symbols
// are staged in shared memory and written out with aligned 16-byte stores,
// since a thread's own span would otherwise be a run of scattered byte
// stores.  Persistent: chunk = stream * bps + span block, blockIdx.x,
// + gridDim.x, ...
template <typename Sym, fkvdec::Cell CELL>
__global__ void __launch_bounds__(dec_threads<Sym>())
k_span_decode_staged(const double2 *__restrict__ pts, int64_t n, int64_t pt_stride, int64_t spans, int bps,
              int64_t n_chunks, Sym *__restrict__ sym, int64_t sym_stride, const fkv_decconst *__restrict__ dc,
              const longlong2 *__restrict__ T, int N, int L, unsigned *status)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    const fkvdec::Tables t = fkvdec::load(dc, T, N, L, dsm);
    uint8_t *sbuf = dsm + tables_bytes(N, L);
    __syncthreads();
    constexpr int TPB = dec_threads<Sym>();
    ChunkWalk w(bps);
    for (int64_t ck = blockIdx.x; ck < n_chunks; ck += gridDim.x, w.next()) {
        const int64_t stream = w.stream;
        const int64_t s0 = w.sb * TPB;
        const int64_t b = s0 * L;
        const int64_t e = min(n, (s0 + TPB) * L);
        uint8_t *dst = reinterpret_cast<uint8_t *>(sym + stream * sym_stride + b);
        const int off = static_cast<int>(reinterpret_cast<uintptr_t>(dst) & 15);
        decode_chunk<CELL>(t, pts, n, pt_stride, spans, stream, s0, reinterpret_cast<Sym *>(sbuf + off), dc, L, status);
        __syncthreads();
        stage_out(dst, sbuf, static_cast<int>(e - b) * static_cast<int>(sizeof(Sym)), off);
        __syncthreads();
    }
}

// The same decode for a whole archive of token records, written out in the
// planar layout the archive gather reads: per stream, the H key planes
// (n_rec x S_K indices each, one plane per head) and then the H value planes
// (n_rec x S_V).  A block first tabulates, for each of the R symbols of a
// record, its offset inside its record's first plane row; a thread then places
// each symbol of its span as the walk yields it, last to first, at that
// offset plus record x stages, stepping back one symbol of the record (and a
// record at its start) per symbol.  Positions inside a stream are 32-bit (the
// launcher keeps a stream below 2^31 symbols) and the span's last record comes
// from a multiply-high division.  Codebooks come with N = 256 or 1024: sectors.
template <typename Sym>
__global__ void __launch_bounds__(dec_threads<Sym>())
k_span_decode_planar(const double2 *__restrict__ pts, unsigned n_rec, int64_t pt_stride, unsigned spans, int bps,
                     unsigned n_chunks, Sym *__restrict__ out, int H, int SK, int SV, fkvd::FastDiv div_r,
                     const fkv_decconst *__restrict__ dc, const longlong2 *__restrict__ T, int N, int L,
                     unsigned *status)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    const fkvdec::Tables t = fkvdec::load(dc, T, N, L, dsm);
    const int R = H * (SK + SV);
    const int nk = H * SK;
    const unsigned n = n_rec * static_cast<unsigned>(R);
    constexpr int TPB = dec_threads<Sym>();
    // symbol o of a record: plane offset (K planes, then V planes) + stage
    unsigned *poff = reinterpret_cast<unsigned *>(dsm + tables_bytes(N, L));
    for (int o = threadIdx.x; o < R; o += TPB) {
        const bool v = o >= nk;
        const int S = v ? SV : SK, oo = v ? o - nk : o;
        const int h = oo / S;
        poff[o] = (v ? static_cast<unsigned>(nk) * n_rec : 0u) + static_cast<unsigned>(h) * n_rec * S + (oo - h * S);
    }
    __syncthreads();
    const long long lim_full = __ldg(&dc->alim[L]);
    ChunkWalk w(bps);
    auto point = [&](const ChunkWalk &c, bool more) {     // this thread's point of a chunk, loaded a chunk ahead
        const unsigned s = static_cast<unsigned>(c.sb) * TPB + threadIdx.x;
        return more && s < spans ? __ldg(&pts[c.stream * pt_stride + s]) : make_double2(0.0, 0.0);
    };
    double2 p = point(w, blockIdx.x < n_chunks);
    for (unsigned ck = blockIdx.x; ck < n_chunks; ck += gridDim.x) {
        const unsigned s = static_cast<unsigned>(w.sb) * TPB + threadIdx.x;
        Sym *base = out + w.stream * static_cast<int64_t>(n);
        w.next();
        const double2 pn = point(w, ck + gridDim.x < n_chunks);
        if (s < spans) {
            const unsigned first = s * static_cast<unsigned>(L);
            const int m = n - first < static_cast<unsigned>(L) ? static_cast<int>(n - first) : L;
            const unsigned q = first + m - 1;             // the span's last symbol
            const unsigned rec = div_r.div(q);
            const int o = static_cast<int>(q - rec * static_cast<unsigned>(R));
            if (!fkvdec::decode_point<fkvdec::kSectors>(t, p, m, m == L ? lim_full : __ldg(&dc->alim[m]), [&] {
                    return [=, o = o, rec = rec](int, int c) mutable {
                        const unsigned S = o < nk ? SK : SV;
                        base[poff[o] + rec * S] = static_cast<Sym>(c);
                        if (o == 0) {
                            o = R;
                            --rec;
                        }
                        --o;
                    };
                }))
                atomicOr(status, FKV_ST_CORRUPT);
        }
        p = pn;
    }
}

// Sec. 5 retrieval in place.  Persistent blocks scan their share of the
// stored points against the query's point (the query encoded from the
// origin by the Sec. 1 map, bit for bit as the encoder would): a point of a
// span of at least l symbols inside the 2 r^l ball is a candidate, and a
// candidate is walked back l steps by the exact decoder; it matches when
// those symbols are the query.  Matches are appended (stream, span) in any
// order; counts[0] counts matches (all of them, even past cap), counts[1]
// candidates.  GB300's FP64 pipe would bound a binary64 distance test of every
// point, so each point first passes an integer box test: the ball's bounding
// box, rounded outward, in an order-preserving integer image of binary64; only
// points inside the box take the binary64 test.  Four points per thread are
// in flight at once.
struct SuffixQuery {
    uint16_t sym[kMaxSpan];
    int len;
};

// Whether the last symbols of the span stored as p are the query: step j of
// the walk recovers the query's symbol len - 1 - j.  One cell test is inlined
// (64 to 128 registers); with all three behind a call, the scan's own registers
// spilled, and next to the tables of N = 1024 the spills missed L1: 10 M points
// 56 us, 72 by the call.
template <fkvdec::Cell CELL>
__device__ __forceinline__ bool ends_in(const fkvdec::Tables &t, double2 p, const SuffixQuery &qy)
{
    long long X = fkvdec::to_q62(p.x), Y = fkvdec::to_q62(p.y);
    bool eq = true;
    fkvdec::walk<CELL, 1>(t, X, Y, qy.len, [&](int j, int c) { eq = eq && c == qy.sym[qy.len - 1 - j]; });
    return eq;
}

template <fkvdec::Cell CELL>
__global__ void __launch_bounds__(kThreads)
k_suffix_search(const double2 *__restrict__ pts, int64_t n_streams, int64_t n, int64_t pt_stride, int64_t spans,
                const __grid_constant__ SuffixQuery qy, double thr, double thr2, const double2 *__restrict__ V, double r,
                const fkv_decconst *__restrict__ dc, const longlong2 *__restrict__ T, int N, int L,
                long long *__restrict__ out, long long cap, unsigned long long *__restrict__ counts)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    __shared__ double2 q_s;
    __shared__ long long box_s[4];
    const fkvdec::Tables t = fkvdec::load(dc, T, N, L, dsm);
    // order-preserving integer image of a binary64 value (signed compare)
    auto okey = [](long long b) { return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll); };
    if (threadIdx.x == 0) {
        const double2 qq = encode_span(qy.sym, qy.len, V, N, r, 0.0, 0.0);
        q_s = qq;
        const double tb = __dmul_ru(thr, 1.0 + 0x1p-40);           // the box contains the ball
        box_s[0] = okey(__double_as_longlong(__dsub_rd(qq.x, tb)));
        box_s[1] = okey(__double_as_longlong(__dadd_ru(qq.x, tb)));
        box_s[2] = okey(__double_as_longlong(__dsub_rd(qq.y, tb)));
        box_s[3] = okey(__double_as_longlong(__dadd_ru(qq.y, tb)));
    }
    __syncthreads();
    const double2 q = q_s;
    const long long bx0 = box_s[0], bx1 = box_s[1], by0 = box_s[2], by1 = box_s[3];
    const longlong2 *pk = reinterpret_cast<const longlong2 *>(pts);
    const int l = qy.len;
    // this block's contiguous share of the n_streams * spans points, walked
    // kThreads apart per thread without division
    const int64_t total = n_streams * spans;
    const int64_t hi = total * (blockIdx.x + 1) / gridDim.x;
    int64_t g = total * blockIdx.x / gridDim.x + threadIdx.x;
    int64_t stream = g / spans, u = g - stream * spans;
    const int64_t step_s = kThreads / spans, step_u = kThreads - step_s * spans;
    constexpr int kU = 4;
    while (g < hi) {
        longlong2 pb[kU];
        int64_t su[kU], uu[kU];
        bool live[kU];
#pragma unroll
        for (int i = 0; i < kU; ++i) {
            live[i] = g < hi;
            su[i] = stream;
            uu[i] = u;
            if (live[i])
                pb[i] = pk[stream * pt_stride + u];
            g += kThreads;
            u += step_u;
            stream += step_s;
            if (u >= spans) {
                u -= spans;
                ++stream;
            }
        }
#pragma unroll
        for (int i = 0; i < kU; ++i) {
            if (!live[i])
                break;
            const int m = static_cast<int>(min(static_cast<int64_t>(L), n - uu[i] * L));
            const long long kx = okey(pb[i].x), ky = okey(pb[i].y);
            if (m >= l && kx >= bx0 && kx <= bx1 && ky >= by0 && ky <= by1) {
                const double2 p = make_double2(__longlong_as_double(pb[i].x), __longlong_as_double(pb[i].y));
                const double dx = __dsub_rn(p.x, q.x), dy = __dsub_rn(p.y, q.y);
                const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
                if (d2 <= thr2) {
                    atomicAdd(&counts[1], 1ull);
                    if (ends_in<CELL>(t, p, qy)) {
                        const unsigned long long slot = atomicAdd(&counts[0], 1ull);
                        if (static_cast<long long>(slot) < cap) {
                            out[2 * slot] = su[i];
                            out[2 * slot + 1] = uu[i];
                        }
                    }
                }
            }
        }
    }
}

// Sec. 2 random access: one request per thread, decoding only its span down
// to the requested offset.  Persistent: a block loads the decoder tables once
// and takes requests blockIdx.x * TPB + threadIdx.x, + gridDim.x * TPB, ...
template <typename Sym, fkvdec::Cell CELL>
__global__ void __launch_bounds__(dec_threads<Sym>())
k_read(const double2 *__restrict__ pts, int64_t n_streams, int64_t n, int64_t pt_stride,
       const int64_t *__restrict__ req, int64_t n_req, Sym *__restrict__ out,
       const fkv_decconst *__restrict__ dc, const longlong2 *__restrict__ T, int N, int L, unsigned *status)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    const fkvdec::Tables t = fkvdec::load(dc, T, N, L, dsm);
    __syncthreads();
    const int64_t stride = static_cast<int64_t>(gridDim.x) * dec_threads<Sym>();
    int64_t q = static_cast<int64_t>(blockIdx.x) * dec_threads<Sym>() + threadIdx.x;
    int64_t st = 0, pos = 0;
    if (q < n_req) {
        st = req[2 * q];
        pos = req[2 * q + 1];
    }
    while (q < n_req) {
        // the next request is on its way during this one's walk
        const int64_t qn = q + stride;
        int64_t stn = 0, posn = 0;
        if (qn < n_req) {
            stn = req[2 * qn];
            posn = req[2 * qn + 1];
        }
        if (st < 0 || st >= n_streams || pos < 0 || pos >= n) {
            out[q] = static_cast<Sym>(~0u);
            atomicOr(status, FKV_ST_RANGE);
        } else {
            const int64_t u = pos / L;
            const int o = static_cast<int>(pos - u * L);
            const int m = static_cast<int>(min(static_cast<int64_t>(L), n - u * L));
            const double2 p = pts[st * pt_stride + u];
            long long X = fkvdec::to_q62(p.x), Y = fkvdec::to_q62(p.y);
            int sym = 0;
            fkvdec::walk_read<CELL>(t, X, Y, m - o, [&](int j, int c) { sym = c; });
            out[q] = static_cast<Sym>(sym);
        }
        q = qn;
        st = stn;
        pos = posn;
    }
}

// Sec. 2 append: one thread per (stream, span touched by the new symbols).
// The first touched span continues from the stored tail point when the old
// length is not a multiple of L; every later span starts at the anchor.
template <typename Sym>
__global__ void __launch_bounds__(kThreads)
k_append(double2 *__restrict__ pts, int64_t n_streams, int64_t pt_stride, int64_t n_old,
         const Sym *__restrict__ sym, int64_t m, int64_t sym_stride, int64_t u_first, int64_t cnt,
         const double2 *__restrict__ V, int N, double r, int L, unsigned *status)
{
    __shared__ double2 sV[vtab_len<Sym>()];
    for (int i = threadIdx.x; i < N; i += kThreads)
        sV[i] = V[i];
    __syncthreads();
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x;
    if (t >= n_streams * cnt)
        return;
    const int64_t stream = t / cnt;
    const int64_t u = u_first + (t - stream * cnt);
    const int64_t n_new = n_old + m;
    const int64_t b = max(u * L, n_old);
    const int64_t e = min((u + 1) * L, n_new);
    double2 p = make_double2(0.0, 0.0);
    if (u * L < n_old)
        p = pts[stream * pt_stride + u];
    Sym s[kMaxSpan];
    const Sym *src = sym + stream * sym_stride + (b - n_old);
    const int len = static_cast<int>(e - b);
    for (int k = 0; k < len; ++k)
        s[k] = src[k];
    p = encode_span(s, len, sV, N, r, p.x, p.y);
    if (isnan(p.x))
        atomicOr(status, FKV_ST_CORRUPT);
    pts[stream * pt_stride + u] = p;
}

// ------------------------------------------------------------ ragged batches
// Streams of different lengths in one call (the sequences of a serving batch
// rarely share a length): stream i holds len_i = so[i + 1] - so[i] symbols at
// sym + so[i] and owns point slots [po[i], po[i + 1]) of pts, at least
// ceil(len_i / L) of them.  so and po are device arrays of n_streams + 1
// offsets.  The kernels walk the point slots [po[0], po[n_streams])
// grid-stride, one span per thread, and find a slot's stream by binary search
// over po.  A stream whose offsets are inconsistent (a negative length, fewer
// point slots than spans) is left alone and reported by the range status bit;
// the check runs once per stream, so a stream with no slots is reported too.

// The stream owning point slot g: the largest i < n_streams with po[i] <= g
// (po nondecreasing; every index read stays in [0, n_streams]).
__device__ __forceinline__ int64_t ragged_stream(const int64_t *__restrict__ po, int64_t n_streams, int64_t g)
{
    int64_t lo = 0, hi = n_streams;
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(&po[mid]) <= g)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// Length of stream i and whether its offsets hold together.
__device__ __forceinline__ bool ragged_ok(const int64_t *__restrict__ so, const int64_t *__restrict__ po, int64_t i,
                                          int L, int64_t *len)
{
    const int64_t n = __ldg(&so[i + 1]) - __ldg(&so[i]);
    const int64_t slots = __ldg(&po[i + 1]) - __ldg(&po[i]);
    *len = n;
    return n >= 0 && slots >= 0 && slots >= (n + L - 1) / L;
}

// Every thread of the grid takes part in checking the streams' offsets.
__device__ __forceinline__ void ragged_check(const int64_t *__restrict__ so, const int64_t *__restrict__ po,
                                             int64_t n_streams, int L, unsigned *status)
{
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_streams; i += stride) {
        int64_t n;
        if (!ragged_ok(so, po, i, L, &n))
            atomicOr(status, FKV_ST_RANGE);
    }
}

// At most kFewSpans slots of a ragged batch, one a thread of one block.  A call,
// for inlined it costs the bulk loop registers (1 us of 11 for 1,000 spans).
template <typename Sym>
static __device__ __noinline__ void encode_ragged_few(const Sym *__restrict__ sym, const int64_t *__restrict__ so,
                                                      int64_t n_streams, double2 *__restrict__ pts,
                                                      const int64_t *__restrict__ po, const EncArgs a, int64_t g,
                                                      unsigned *status)
{
    const int64_t i = ragged_stream(po, n_streams, g);
    int64_t n;
    if (!ragged_ok(so, po, i, a.L, &n))
        return;
    const int64_t s = g - __ldg(&po[i]);
    if (s < 0 || s * a.L >= n)
        return;
    const int m = static_cast<int>(min(static_cast<int64_t>(a.L), n - s * a.L));
    const double2 p = encode_few(sym + __ldg(&so[i]) + s * a.L, m, a.V, a);
    if (__double2hiint(p.x) == -1)
        atomicOr(status, FKV_ST_CORRUPT);
    pts[g] = p;
}

template <bool HALF, typename Sym>
__global__ void __launch_bounds__(kThreads)
k_span_encode_ragged(const Sym *__restrict__ sym, const int64_t *__restrict__ so, int64_t n_streams,
                     double2 *__restrict__ pts, const int64_t *__restrict__ po, const EncArgs a, unsigned *status)
{
    __shared__ EncTable<HALF, Sym> tab;
    const int L = a.L;
    const RatioMul mul(a.r);
    tab.load(a);
    __syncthreads();
    ragged_check(so, po, n_streams, L, status);
    const int64_t g0 = __ldg(&po[0]), g1 = __ldg(&po[n_streams]);
    if (!HALF && g1 - g0 <= kFewSpans) {
        if (blockIdx.x == 0 && threadIdx.x < g1 - g0)
            encode_ragged_few(sym, so, n_streams, pts, po, a, g0 + threadIdx.x, status);
        return;
    }
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kThreads;
    for (int64_t g = g0 + static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; g < g1; g += stride) {
        const int64_t i = ragged_stream(po, n_streams, g);
        int64_t n;
        if (!ragged_ok(so, po, i, L, &n))
            continue;
        const int64_t s = g - __ldg(&po[i]);
        if (s < 0 || s * L >= n)
            continue;                       // a slot past the stream's last span
        const int m = static_cast<int>(min(static_cast<int64_t>(L), n - s * L));
        const double2 p = encode_anchored<HALF>(sym + __ldg(&so[i]) + s * L, m, tab, a, mul);
        if (__double2hiint(p.x) == -1)
            atomicOr(status, FKV_ST_CORRUPT);
        pts[g] = p;
    }
}

// Receiver of a walk that stores m symbols from dst, last to first; WORDS: bytes
// go out as the aligned words they make up.
template <bool WORDS, typename Sym>
__device__ __forceinline__ auto span_writer(Sym *dst, int m)
{
    if constexpr (!WORDS) {
        return [=](int j, int c) { dst[m - 1 - j] = static_cast<Sym>(c); };
    } else {
        const unsigned last = static_cast<unsigned>(reinterpret_cast<uintptr_t>(dst)) + m - 1;
        return [=, acc = 0u](int j, int c) mutable {
            acc = (acc << 8) | static_cast<unsigned>(c);
            const unsigned in_word = (last - static_cast<unsigned>(j)) & 3u;
            if (in_word == 0u) {
                uint8_t *at = dst + (m - 1 - j);
                if (j >= 3) {
                    *reinterpret_cast<unsigned *>(at) = acc;
                } else {
                    for (int k = 0; k <= j; ++k)
                        at[k] = static_cast<uint8_t>(acc >> (8 * k));
                }
            } else if (j == m - 1) {
                const int cnt = min(m, 4 - static_cast<int>(in_word));
                for (int k = 0; k < cnt; ++k)
                    dst[k] = static_cast<uint8_t>(acc >> (8 * k));
            }
        };
    }
}

// WORDS: bytes as words (span_writer) in batches of more than kWordSpans spans;
// in smaller ones the stores are not what a warp waits for (8,097 spans of 44
// symbols, N = 4: 12.6 us as bytes, 14.4 as words; 26,903 of 24, N = 8: 10.5 and
// 12.6; 33,868 of 44, N = 4: 18.9 and 12.6).  A loop for each, for a branch
// inside one costs up to 3 us.
constexpr int64_t kWordSpans = 24576;

template <typename Sym, fkvdec::Cell CELL, bool WORDS>
__global__ void __launch_bounds__(dec_threads<Sym>())
k_span_decode_ragged(const double2 *__restrict__ pts, const int64_t *__restrict__ po, int64_t n_streams,
                     Sym *__restrict__ sym, const int64_t *__restrict__ so, const fkv_decconst *__restrict__ dc,
                     const longlong2 *__restrict__ T, int N, int L, unsigned *status)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    const fkvdec::Tables t = fkvdec::load(dc, T, N, L, dsm);
    __syncthreads();
    ragged_check(so, po, n_streams, L, status);
    const int64_t g0 = __ldg(&po[0]), g1 = __ldg(&po[n_streams]);
    const bool many = g1 - g0 > kWordSpans;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    auto all = [&](auto words) {
        for (int64_t g = g0 + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; g < g1; g += stride) {
            const int64_t i = ragged_stream(po, n_streams, g);
            int64_t n;
            if (!ragged_ok(so, po, i, L, &n))
                continue;
            const int64_t s = g - __ldg(&po[i]);
            if (s < 0 || s * L >= n)
                continue;
            const int m = static_cast<int>(min(static_cast<int64_t>(L), n - s * L));
            Sym *dst = sym + __ldg(&so[i]) + s * L;
            if (!fkvdec::decode_point<CELL>(t, pts[g], m, __ldg(&dc->alim[m]),
                                            [&] { return span_writer<words.value>(dst, m); }))
                atomicOr(status, FKV_ST_CORRUPT);
        }
    };
    if (WORDS && many)
        all(std::integral_constant<bool, WORDS>());
    else
        all(std::false_type());
}

// Random access into a ragged batch: request q = (stream, position), the
// position checked against that stream's own length.
template <typename Sym, fkvdec::Cell CELL>
__global__ void __launch_bounds__(dec_threads<Sym>())
k_read_ragged(const double2 *__restrict__ pts, const int64_t *__restrict__ po, const int64_t *__restrict__ so,
              int64_t n_streams, const int64_t *__restrict__ req, int64_t n_req, Sym *__restrict__ out,
              const fkv_decconst *__restrict__ dc, const longlong2 *__restrict__ T, int N, int L, unsigned *status)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    const fkvdec::Tables t = fkvdec::load(dc, T, N, L, dsm);
    __syncthreads();
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < n_req; q += stride) {
        const int64_t st = req[2 * q], pos = req[2 * q + 1];
        int64_t n = 0;
        if (st < 0 || st >= n_streams || !ragged_ok(so, po, st, L, &n) || pos < 0 || pos >= n) {
            out[q] = static_cast<Sym>(~0u);
            atomicOr(status, FKV_ST_RANGE);
            continue;
        }
        const int64_t u = pos / L;
        const int o = static_cast<int>(pos - u * L);
        const int m = static_cast<int>(min(static_cast<int64_t>(L), n - u * L));
        const double2 p = pts[__ldg(&po[st]) + u];
        long long X = fkvdec::to_q62(p.x), Y = fkvdec::to_q62(p.y);
        int c = 0;
        fkvdec::walk_read<CELL>(t, X, Y, m - o, [&](int, int cc) { c = cc; });
        out[q] = static_cast<Sym>(c);
    }
}

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// ------------------------------------------------------------- lossy archive
// Sec. 4: a span's stored point truncated to B bits per coordinate, the
// B-bit two's complement code k = floor(x 2^(B-1)); the spans of a stream
// older than its last keep_exact are kept as codes, packed into uint32 words
// (span u's x code at stream bit 2uB, its y code at 2uB + B, least
// significant bit first), the recent ones as exact points in a tail array.
struct LossyArgs {
    const uint32_t *codes;   // [n_streams][code_stride] words
    int64_t code_stride;
    int64_t words;           // words holding codes, per stream
    const double2 *tail;     // [n_streams][tail_stride] exact points of spans T ..
    int64_t tail_stride;
    int64_t T;               // truncated spans per stream
    int bits;
    double scale;            // 2^-(B-1)
};

// B-bit code of one coordinate: floor(x 2^(B-1)).  From the binary64 fields
// with integer ops (a conversion issues at the FP64 rate): x = m 2^(e - 1075),
// a right shift of m by s = 1076 - B - e, rounded up for a negative x.
__device__ __forceinline__ unsigned long long trunc_field(double x, double up, int bits)
{
    const long long b = __double_as_longlong(x);
    const int e = static_cast<int>((b >> 52) & 0x7FF);
    const unsigned long long mask = (1ull << bits) - 1;
    if (e == 0 || e > 1023)                      // zero, subnormal, |x| >= 2 or not finite
        return static_cast<unsigned long long>(floor_fp64(mul_fp64(x, up))) & mask;
    const unsigned long long m = (static_cast<unsigned long long>(b) & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int s = min(1076 - bits - e, 63);      // >= 0
    if (b < 0)
        return (0ull - ((m + ((1ull << s) - 1)) >> s)) & mask;
    return (m >> s) & mask;
}

// Warp per group of 32 spans of one stream: the group's 64 codes fill exactly
// 2B words (the group starts at stream bit 64 B g, a word boundary).  A lane
// puts its span's two codes, 2B bits that touch at most five words, into the
// warp's words in shared memory (neighbours share words, so by atomic OR), and
// the warp writes those out.  1.14 M spans at 24 bits:
// 10.4 us (15.2 with the words gathered by shuffles).
__global__ void __launch_bounds__(kThreads)
k_truncate(const double *__restrict__ pts, int64_t pt_stride, int64_t n_streams, int64_t T, int bits,
           uint32_t *__restrict__ codes, int64_t code_stride, int64_t words)
{
    __shared__ uint32_t wbuf[kThreads / 32][2 * 53 + 4];
    const double up = static_cast<double>(1ull << (bits - 1));
    const int lane = threadIdx.x & 31;
    uint32_t *w = wbuf[threadIdx.x >> 5];
    const int64_t gps = (T + 31) >> 5;                       // groups per stream
    const int64_t n_groups = n_streams * gps;
    const int64_t nw = static_cast<int64_t>(gridDim.x) * (kThreads / 32);
    const int wpg = 2 * bits;                                // words per group
    for (int j = lane; j < wpg + 4; j += 32)
        w[j] = 0;
    __syncwarp();
    for (int64_t g = (static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x) >> 5; g < n_groups; g += nw) {
        const int64_t stream = g / gps, grp = g - stream * gps;
        const int64_t u = grp * 32 + lane;
        if (u < T) {
            const double2 p = __ldg(&reinterpret_cast<const double2 *>(pts)[stream * pt_stride + u]);
            const unsigned long long fx = trunc_field(p.x, up, bits), fy = trunc_field(p.y, up, bits);
            // the 2B bits from bit 2B lane on, as words of 32
            const int at = wpg * lane, sh = at & 31;
            const unsigned long long lo = fx | (fy << bits), hi = bits < 64 - bits ? 0ull : fy >> (64 - bits);
            uint32_t v[5];
            v[0] = static_cast<uint32_t>(lo << sh);
            v[1] = __funnelshift_l(static_cast<uint32_t>(lo), static_cast<uint32_t>(lo >> 32), sh);
            v[2] = __funnelshift_l(static_cast<uint32_t>(lo >> 32), static_cast<uint32_t>(hi), sh);
            v[3] = __funnelshift_l(static_cast<uint32_t>(hi), static_cast<uint32_t>(hi >> 32), sh);
            v[4] = __funnelshift_l(static_cast<uint32_t>(hi >> 32), 0u, sh);
            const int nv = (sh + wpg + 31) >> 5;
#pragma unroll
            for (int i = 0; i < 5; ++i)
                if (i < nv)
                    atomicOr(&w[(at >> 5) + i], v[i]);
        }
        __syncwarp();
        const int64_t w0 = grp * wpg;
        const int nwg = static_cast<int>(min(static_cast<int64_t>(wpg), words - w0));
        for (int j = lane; j < wpg; j += 32) {
            if (j < nwg)
                codes[stream * code_stride + w0 + j] = w[j];
            w[j] = 0;
        }
        __syncwarp();
    }
}

// The B-bit field at stream bit `pos`, sign-extended.
__device__ __forceinline__ long long read_field(const uint32_t *w, int64_t words, int64_t pos, int bits)
{
    const int64_t q = pos >> 5;
    const int off = static_cast<int>(pos & 31);
    unsigned long long v = __ldg(w + q);
    if (q + 1 < words)
        v |= static_cast<unsigned long long>(__ldg(w + q + 1)) << 32;
    v >>= off;
    if (off + bits > 64 && q + 2 < words)
        v |= static_cast<unsigned long long>(__ldg(w + q + 2)) << (64 - off);
    const int sh = 64 - bits;
    return static_cast<long long>(v << sh) >> sh;
}

// k 2^-(bits - 1) for a bits-bit code k: below 53 bits, k added to the integer
// pattern of 1.5 2^52 and that number subtracted again is k exactly, and the
// scaling is the exponent's.
__device__ __forceinline__ double code_value(long long k, int bits, double scale)
{
    if (bits > 52)
        return __dmul_rn(static_cast<double>(k), scale);
    const double v = __dsub_rn(__longlong_as_double(k + 0x4338000000000000ll), 0x1.8p52);
    const int hi = __double2hiint(v);
    return __hiloint2double(k != 0 ? hi - ((bits - 1) << 20) : 0, __double2loint(v));
}

// The point a lossy archive keeps for span u of a stream.
__device__ __forceinline__ double2 lossy_point(const LossyArgs &a, int64_t stream, int64_t u)
{
    if (u >= a.T)
        return a.tail[stream * a.tail_stride + (u - a.T)];
    const uint32_t *w = a.codes + stream * a.code_stride;
    const int64_t pos = 2 * u * a.bits;
    const long long kx = read_field(w, a.words, pos, a.bits);
    const long long ky = read_field(w, a.words, pos + a.bits, a.bits);
    return make_double2(code_value(kx, a.bits, a.scale), code_value(ky, a.bits, a.scale));
}

// Squared distance to a vertex as the paper's binary64 arithmetic forms it
// (two products and a sum, no FMA).
__device__ __forceinline__ double dist2(double2 v, double x, double y)
{
    const double dx = __dsub_rn(x, v.x), dy = __dsub_rn(y, v.y);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}

// What the lossy walks use of a context.
struct LossyWalk {
    const double2 *V;
    int N, L;
    double w, r;             // 1 - r and r
    unsigned long long inv;  // floor(2^127 / (r's mantissa at the top of 64 bits)); 0 for r a power of two
    int er;                  // r's exponent field
    const int2 *bound;       // (cos, -sin) 2^30 of boundary g + 1/2 at [g + N / 2 + 1], g = -N/2 - 1 .. N/2
    float sect_a[5];         // arctangent polynomial in sector widths
};

static __device__ __noinline__ double div_fp64(double a, double b) { return __ddiv_rn(a, b); }

// a / r rounded to nearest even, as __ddiv_rn(a, r), on the integer pipe: the
// mantissa of a (at the top of 64 bits) times inv is the quotient's upper 64
// bits, low by less than two units (inv is rounded down, and the product's
// upper word again), and rounds at its 53rd bit.  A quotient of two 53-bit
// numbers is no midpoint (r not a power of two).  So with the dropped bits of h
// at one half or above the quotient rounds up, at one half less two units or
// below it rounds down, and one unit below one half it may be on either side:
// those (1 in 1024), far-out exponents and r a power of two take the IEEE
// division.
__device__ __forceinline__ double div_ratio(const LossyWalk &q, double a)
{
    const unsigned hi = static_cast<unsigned>(__double2hiint(a)), lo = static_cast<unsigned>(__double2loint(a));
    const int e = static_cast<int>((hi >> 20) & 0x7FFu);
    const unsigned long long m = (static_cast<unsigned long long>(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) |
                                 (lo << 11);
    const unsigned long long h = __umul64hi(m, q.inv);
    const int top = static_cast<int>(h >> 63);
    const int drop = 10 + top;
    const unsigned half = 512u << top;
    const unsigned rest = static_cast<unsigned>(h) & (2u * half - 1u);
    if (static_cast<unsigned>(e - 512) >= 1000u || rest == half - 1u || q.inv == 0)
        return div_fp64(a, q.r);
    const unsigned long long n = (h + half) >> drop;
    const unsigned th = static_cast<unsigned>(n >> 32) + (static_cast<unsigned>(1021 + top + e - q.er) << 20);
    return __hiloint2double(static_cast<int>(th | (hi & 0x80000000u)), static_cast<int>(static_cast<unsigned>(n)));
}

// Sec. 1 cell test in binary64 for a point that need not be a code point:
// the vertex of least binary64 squared distance, lowest index on a tie.  The
// nearest vertex is the angularly nearest.  For a larger coordinate in
// [2^-14, 2^16) the fp32 angle names the pair of neighbouring sectors (any
// error below half a sector will do) and the sign of the cross product with
// their common boundary, on 31-bit images of the point and the boundary, picks
// one of them.  The images are off by at most one unit (the point, truncated)
// and half a unit (the boundary) a coordinate, so the product by less than
// (sqrt 2 + 2) 2^30.  At 2^34 and above its sign is sure, and the direction at
// least 12.5 2^30 / 2^61.5 = 4.1e-9 rad off the boundary: the two squared
// distances differ by 4 |p| sin(pi/N) 4.1e-9, above their rounding,
// (|p| + 1)^2 3.4e-16 (at N = 1024 by a factor of 9 at |p| = 2^-14, 1.6 at
// 2^16.5 and 10^4 at 1).  Nearer the boundary, and for |p|^2 up to 2^60, the
// three vertices around the angle are scored: every other vertex is farther by
// at least 2|p|(cos(pi/N) - cos(3 pi/N)) (7.5e-5 |p| at N = 1024), so the
// choice equals a full scan's.  Other points (tiny, huge, not finite) take the
// full scan.
// The angle alone with a margin for the polynomial's 1.2e-5 rad, as in the
// planar decoder, left 3 warps in 4 a lane to score: a code point's offset
// from its vertex is r times a point near the unit circle, so its place across
// the sector crowds at the boundaries.  k_lossy_decode on 96 streams of 71,136
// symbols (N = 256, 24 bits): 53 us, 105 with the margin.  (The planar
// decoder settles its near cases with four integer products; there the cross
// product costs more than it saves, 0.460 against 0.456 ms for encoding and
// decoding 50.3 M symbols.)
static __device__ __noinline__ int nearest64_scored(const double2 *sV, int N, double x, double y)
{
    const double rr = x * x + y * y;
    if (rr >= 0x1p-40 && rr <= 0x1p60) {
        const float a = atan2f(static_cast<float>(y), static_cast<float>(x)) *
                        (static_cast<float>(N) * 0.15915494309189535f);
        int c0 = static_cast<int>(rintf(a));
        c0 = c0 < 0 ? c0 + N : (c0 >= N ? c0 - N : c0);
        int best = -1;
        double bd = 0.0;
#pragma unroll
        for (int k = -1; k <= 1; ++k) {
            int c = c0 + k;
            c = c < 0 ? c + N : (c >= N ? c - N : c);
            const double d = dist2(sV[c], x, y);
            if (best < 0 || d < bd || (d == bd && c < best)) {
                bd = d;
                best = c;
            }
        }
        return best;
    }
    int best = 0;
    double bd = INFINITY;
    for (int c = 0; c < N; ++c) {
        const double d = dist2(sV[c], x, y);
        if (d < bd) {
            bd = d;
            best = c;
        }
    }
    return best;
}

// The 31 upper bits of a binary64 mantissa, shifted down to exponent field e.
__device__ __forceinline__ int image31(double v, int e)
{
    const int hi = __double2hiint(v);
    const int ev = (hi >> 20) & 0x7FF;
    const unsigned m = 0x40000000u | ((static_cast<unsigned>(hi) & 0xFFFFFu) << 10) |
                       (static_cast<unsigned>(__double2loint(v)) >> 22);
    const int r = static_cast<int>(m >> min(e - ev, 31));
    return hi < 0 ? -r : r;
}

__device__ __forceinline__ int nearest64(const LossyWalk &q, const int2 *bound, const double2 *sV, double x, double y)
{
    // exponent field of the larger coordinate, in [2^-14, 2^16)
    const int big = max(__double2hiint(x) & 0x7FFFFFFF, __double2hiint(y) & 0x7FFFFFFF) >> 20;
    if (static_cast<unsigned>(big - 1009) < 30u) {
        const int hx = image31(x, big), hy = image31(y, big);
        const float a = fkvdec::sector_angle(q.N, q.sect_a, __int2float_rn(hx), __int2float_rn(hy), 1.0f);
        const int lower = __float_as_int(__fadd_rd(a, 12582912.0f)) - 0x4B400000;   // floor, -N/2 - 1 .. N/2
        const int2 b = bound[lower + (q.N / 2 + 1)];
        const int s =
            static_cast<int>((static_cast<long long>(b.x) * hy + static_cast<long long>(b.y) * hx) >> 32);
        const int c = lower + (s > 0 ? 1 : 0);
        if (static_cast<unsigned>(s + 4) > 7u)
            return c < 0 ? c + q.N : c;
    }
    return nearest64_scored(sV, q.N, x, y);
}

// Vertices V(c) at sV[c], their multiples (1 - r) V(c) at sV[N + c], the
// sector boundaries behind them (lossy_table_bytes in all).
__host__ __device__ inline int lossy_table_bytes(int N) { return (N * 32 + (N + 2) * 8 + 15) & ~15; }

__device__ __forceinline__ const int2 *load_lossy(double2 *sV, const LossyWalk &q)
{
    int2 *bound = reinterpret_cast<int2 *>(sV + 2 * q.N);
    for (int i = threadIdx.x; i < q.N + 2; i += blockDim.x)
        bound[i] = q.bound[i];
    for (int i = threadIdx.x; i < q.N; i += blockDim.x) {
        const double2 v = q.V[i];
        sV[i] = v;
        sV[q.N + i] = make_double2(__dmul_rn(q.w, v.x), __dmul_rn(q.w, v.y));
    }
    return bound;
}

// Backward walk from (x, y) in the paper's arithmetic: the cell, then
// p <- (p - w V(c)) / r with w = 1 - r (binary64 product, difference and
// IEEE division).  emit(j, c) receives the symbol of step j.  Two binary64
// operations a symbol, the differences; three scored distances, the products
// and two divisions on the FP64 pipe took about 40.  96 streams of 71,136
// symbols (N = 256, 24 bits): 0.053 ms, 0.586 ms before.
template <class Emit>
__device__ __forceinline__ void walk64(const LossyWalk &q, const int2 *bound, const double2 *sV, double x,
                                       double y, int steps, Emit emit)
{
    for (int j = 0; j < steps; ++j) {
        const int c = nearest64(q, bound, sV, x, y);
        emit(j, c);
        const double2 v = sV[q.N + c];
        x = div_ratio(q, __dsub_rn(x, v.x));
        y = div_ratio(q, __dsub_rn(y, v.y));
    }
}

// Staging of one warp's 32 spans, 16-byte aligned, with the realignment slack.
template <typename Sym>
__host__ __device__ inline int warp_stage_bytes(int L)
{
    return (32 * L * static_cast<int>(sizeof(Sym)) + 32 + 15) & ~15;
}

// Bulk decode of a lossy archive: persistent blocks walk chunks of 256 spans
// (one per thread); each warp writes its 32 spans' symbols through its own
// piece of shared memory, so that no warp waits for another's walk.
template <typename Sym>
__global__ void __launch_bounds__(kThreads)
k_lossy_decode(const LossyArgs a, int64_t n, int64_t spans, int bps, int64_t n_chunks, Sym *__restrict__ sym,
               int64_t sym_stride, const LossyWalk q)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    double2 *sV = reinterpret_cast<double2 *>(dsm);
    const int L = q.L, lane = threadIdx.x & 31;
    uint8_t *sbuf = dsm + lossy_table_bytes(q.N) + (threadIdx.x >> 5) * warp_stage_bytes<Sym>(L);
    const int2 *bound = load_lossy(sV, q);
    __syncthreads();
    ChunkWalk cw(bps);
    for (int64_t ck = blockIdx.x; ck < n_chunks; ck += gridDim.x, cw.next()) {
        const int64_t stream = cw.stream;
        const int64_t s0 = cw.sb * kThreads + (threadIdx.x & ~31);     // the warp's first span
        if (s0 >= spans)
            continue;
        const int64_t b = s0 * L;
        const int64_t e = min(n, (s0 + 32) * L);
        uint8_t *dst = reinterpret_cast<uint8_t *>(sym + stream * sym_stride + b);
        const int off = static_cast<int>(reinterpret_cast<uintptr_t>(dst) & 15);
        const int64_t s = s0 + lane;
        if (s < spans) {
            const int m = static_cast<int>(min(static_cast<int64_t>(L), n - s * L));
            const double2 p = lossy_point(a, stream, s);
            Sym *my = reinterpret_cast<Sym *>(sbuf + off) + lane * L + m - 1;
            walk64(q, bound, sV, p.x, p.y, m, [&](int j, int c) { my[-j] = static_cast<Sym>(c); });
        }
        __syncwarp();
        stage_out_warp(dst, sbuf, static_cast<int>(e - b) * static_cast<int>(sizeof(Sym)), off);
        __syncwarp();
    }
}

// Random reads from a lossy archive: one request per thread.
template <typename Sym>
__global__ void __launch_bounds__(kThreads)
k_lossy_read(const LossyArgs a, int64_t n_streams, int64_t n, const int64_t *__restrict__ req, int64_t n_req,
             Sym *__restrict__ out, const LossyWalk q, unsigned *status)
{
    extern __shared__ __align__(16) uint8_t dsm[];
    double2 *sV = reinterpret_cast<double2 *>(dsm);
    const int L = q.L;
    const int2 *bound = load_lossy(sV, q);
    __syncthreads();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; i < n_req;
         i += static_cast<int64_t>(gridDim.x) * kThreads) {
        const int64_t st = req[2 * i], pos = req[2 * i + 1];
        if (st < 0 || st >= n_streams || pos < 0 || pos >= n) {
            out[i] = static_cast<Sym>(~0u);
            atomicOr(status, FKV_ST_RANGE);
            continue;
        }
        const int64_t u = pos / L;
        const int o = static_cast<int>(pos - u * L);
        const int m = static_cast<int>(min(static_cast<int64_t>(L), n - u * L));
        const double2 p = lossy_point(a, st, u);
        int c = 0;
        walk64(q, bound, sV, p.x, p.y, m - o, [&](int j, int cc) { c = cc; });
        out[i] = static_cast<Sym>(c);
    }
}

}  // namespace

// Symbol width of a context: 1 byte for N <= 256, else 2.
inline bool wide(const fkv_ctx *c) { return c->N > 256; }

int codec_smem_bytes(int N, int L)
{
    return tables_bytes(N, L) + (N > 256 ? dec_stage_bytes<uint16_t>(L) : dec_stage_bytes<uint8_t>(L));
}

static EncArgs enc_args(const fkv_ctx *c)
{
    return EncArgs{c->d_V, c->d_pre, c->N, c->L, c->pre_k, c->r};
}

// The table's symbols: as many as give at most 2^16 points (1 MB, which L2
// holds), no more than a span.
int pre_table_symbols(int N, int L, int *count)
{
    int k = 0, n = 1;
    while (k < L && n <= (1 << 16) / N) {
        n *= N;
        ++k;
    }
    *count = n;
    return k;
}

cudaError_t launch_pre_table(const fkv_ctx *c, cudaStream_t st)
{
    int count = 0;
    const int k = pre_table_symbols(c->N, c->L, &count);
    k_pre_table<<<(count + kThreads - 1) / kThreads, kThreads, 0, st>>>(c->d_V, c->N, c->r, k, count, c->d_pre);
    return cudaGetLastError();
}

template <typename Sym>
cudaError_t span_encode_t(const fkv_ctx *c, const Sym *sym, int64_t n_streams, int64_t n, int64_t sym_stride,
                          double *pts, int64_t pt_stride, cudaStream_t st)
{
    const int64_t spans = cdiv(n, c->L);
    const int64_t bps = cdiv(spans, kThreads);
    const int64_t blocks = n_streams * bps;
    if (blocks == 0)
        return cudaSuccess;
    if (blocks > 0x7FFFFFFF)
        return cudaErrorInvalidConfiguration;
    // streams of at most half a block's spans share blocks, and so do all while
    // they are few
    if (n_streams * spans <= (spans <= kThreads / 2 ? 0x7FFFFFFF : kFewSpans * c->sms)) {
        const unsigned total = static_cast<unsigned>(n_streams * spans);
        // an SM's share of the spans in whole warps, a block's threads at most
        const unsigned share = (total / c->sms + 32) & ~31u, per = share < kThreads ? share : kThreads;
        const auto flat = c->r == 0.5 ? k_span_encode_flat<true, false, Sym>
                          : per <= kFewSpans ? k_span_encode_flat<false, true, Sym>
                                             : k_span_encode_flat<false, false, Sym>;
        flat<<<(total + per - 1) / per, kThreads, 0, st>>>(
            sym, n, sym_stride, static_cast<unsigned>(spans), total, per,
            fkvd::FastDiv::make(static_cast<unsigned>(spans)), reinterpret_cast<double2 *>(pts), pt_stride,
            enc_args(c), c->d_status);
        return cudaGetLastError();
    }
    const auto kern = c->r == 0.5 ? k_span_encode<true, Sym> : k_span_encode<false, Sym>;
    kern<<<static_cast<unsigned>(blocks), kThreads, 0, st>>>(sym, n, sym_stride, spans, static_cast<int>(bps),
                                                             reinterpret_cast<double2 *>(pts), pt_stride, enc_args(c),
                                                             c->d_status);
    return cudaGetLastError();
}

cudaError_t launch_span_encode(const fkv_ctx *c, const void *sym, int64_t n_streams, int64_t n,
                               int64_t sym_stride, double *pts, int64_t pt_stride, cudaStream_t st)
{
    if (wide(c))
        return span_encode_t(c, static_cast<const uint16_t *>(sym), n_streams, n, sym_stride, pts, pt_stride, st);
    return span_encode_t(c, static_cast<const uint8_t *>(sym), n_streams, n, sym_stride, pts, pt_stride, st);
}

// Persistent decode grid: as many blocks of `threads` as fit on the GPU at
// once, at most one per chunk.
cudaError_t decode_grid(const fkv_ctx *c, const void *kern, int smem, int64_t n_chunks, unsigned *grid,
                        int threads = kThreads)
{
    int per_sm = 0;
    const cudaError_t e = kernel_use(c, kern, threads, smem, &per_sm);
    if (e != cudaSuccess)
        return e;
    int64_t g = static_cast<int64_t>(c->sms) * (per_sm > 0 ? per_sm : 1);
    if (g > n_chunks)
        g = n_chunks;
    *grid = static_cast<unsigned>(g);
    return cudaSuccess;
}

template <typename Sym>
cudaError_t span_decode_t(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n, int64_t pt_stride,
                          Sym *sym, int64_t sym_stride, cudaStream_t st)
{
    constexpr int TPB = dec_threads<Sym>();
    const int64_t spans = cdiv(n, c->L);
    const int64_t bps = cdiv(spans, TPB);
    const int64_t n_chunks = n_streams * bps;
    if (n_chunks == 0)
        return cudaSuccess;
    if (bps > 0x7FFFFFFF)
        return cudaErrorInvalidConfiguration;
    // spans of up to 8 symbols: each thread stores its own; longer ones: staged
    const bool direct = c->L <= 8;
    auto kern = direct ? k_span_decode<Sym, fkvdec::kSectors> : k_span_decode_staged<Sym, fkvdec::kSectors>;
    if constexpr (sizeof(Sym) == 1) {
        if (c->N == 4)
            kern = direct ? k_span_decode<Sym, fkvdec::kAxes> : k_span_decode_staged<Sym, fkvdec::kAxes>;
        else if (c->N <= 8)
            kern = direct ? k_span_decode<Sym, fkvdec::kScores> : k_span_decode_staged<Sym, fkvdec::kScores>;
    }
    const int smem = tables_bytes(c->N, c->L) + (direct ? 0 : dec_stage_bytes<Sym>(c->L));
    unsigned grid = 0;
    cudaError_t e = decode_grid(c, reinterpret_cast<const void *>(kern), smem, n_chunks, &grid, TPB);
    if (e != cudaSuccess)
        return e;
    kern<<<grid, TPB, smem, st>>>(reinterpret_cast<const double2 *>(pts), n, pt_stride, spans, static_cast<int>(bps),
                                  n_chunks, sym, sym_stride, c->d_dec, c->d_T, c->N, c->L, c->d_status);
    return cudaGetLastError();
}

cudaError_t launch_span_decode(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n,
                               int64_t pt_stride, void *sym, int64_t sym_stride, cudaStream_t st)
{
    if (wide(c))
        return span_decode_t(c, pts, n_streams, n, pt_stride, static_cast<uint16_t *>(sym), sym_stride, st);
    return span_decode_t(c, pts, n_streams, n, pt_stride, static_cast<uint8_t *>(sym), sym_stride, st);
}

template <typename Sym>
cudaError_t span_decode_planar_t(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n_rec,
                                 int64_t pt_stride, Sym *out, cudaStream_t st)
{
    const int SK = c->cb[0].stages, SV = c->cb[1].stages;
    const int R = c->H * (SK + SV);
    const int64_t n = n_rec * R;
    constexpr int TPB = dec_threads<Sym>();
    const int64_t spans = cdiv(n, c->L);
    const int64_t bps = cdiv(spans, TPB);
    const int64_t n_chunks = n_streams * bps;
    if (n_chunks == 0)
        return cudaSuccess;
    // 32-bit positions inside a stream, and chunk numbers
    if (n > 0x7FFFFFFF || n_chunks > 0x7FFFFFFF)
        return cudaErrorInvalidConfiguration;
    const int smem = tables_bytes(c->N, c->L) + R * static_cast<int>(sizeof(unsigned));
    unsigned grid = 0;
    cudaError_t e = decode_grid(c, reinterpret_cast<const void *>(k_span_decode_planar<Sym>), smem, n_chunks, &grid, TPB);
    if (e != cudaSuccess)
        return e;
    k_span_decode_planar<Sym><<<grid, TPB, smem, st>>>(
        reinterpret_cast<const double2 *>(pts), static_cast<unsigned>(n_rec), pt_stride,
        static_cast<unsigned>(spans), static_cast<int>(bps), static_cast<unsigned>(n_chunks), out, c->H, SK, SV,
        fkvd::FastDiv::make(static_cast<unsigned>(R)), c->d_dec, c->d_T, c->N, c->L, c->d_status);
    return cudaGetLastError();
}

cudaError_t launch_span_decode_planar(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n_rec,
                                      int64_t pt_stride, void *out, cudaStream_t st)
{
    if (wide(c))
        return span_decode_planar_t(c, pts, n_streams, n_rec, pt_stride, static_cast<uint16_t *>(out), st);
    return span_decode_planar_t(c, pts, n_streams, n_rec, pt_stride, static_cast<uint8_t *>(out), st);
}

cudaError_t launch_suffix_search(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n,
                                 int64_t pt_stride, const uint16_t *query, int qlen, int64_t *out, int64_t cap,
                                 int64_t *counts, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(counts, 0, 2 * sizeof(int64_t), st);
    if (e != cudaSuccess)
        return e;
    const int64_t spans = cdiv(n, c->L);
    if (n_streams * spans == 0)
        return cudaSuccess;
    SuffixQuery qy;
    for (int i = 0; i < kMaxSpan; ++i)
        qy.sym[i] = i < qlen ? query[i] : 0;
    qy.len = qlen;
    // (2 r^l)^2 with r^l by l successive multiplications (the Sec. 5 ball)
    double rl = 1.0;
    for (int i = 0; i < qlen; ++i)
        rl = rl * c->r;
    const double t = 2.0 * rl;
    const double thr2 = t * t;
    const int smem = tables_bytes(c->N, c->L);
    unsigned grid = 0;
    const auto kern = c->N > 8    ? k_suffix_search<fkvdec::kSectors>
                      : c->N == 4 ? k_suffix_search<fkvdec::kAxes>
                                  : k_suffix_search<fkvdec::kScores>;
    e = decode_grid(c, reinterpret_cast<const void *>(kern), smem, cdiv(n_streams * spans, kThreads), &grid);
    if (e != cudaSuccess)
        return e;
    kern<<<grid, kThreads, smem, st>>>(reinterpret_cast<const double2 *>(pts), n_streams, n, pt_stride, spans, qy, t,
                                       thr2, c->d_V, c->r, c->d_dec, c->d_T, c->N, c->L,
                                       reinterpret_cast<long long *>(out), cap,
                                       reinterpret_cast<unsigned long long *>(counts));
    return cudaGetLastError();
}

template <typename Sym>
cudaError_t read_t(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n, int64_t pt_stride,
                   const int64_t *req, int64_t n_req, Sym *out, cudaStream_t st)
{
    constexpr int TPB = dec_threads<Sym>();
    const int64_t blocks = cdiv(n_req, TPB);
    if (blocks == 0)
        return cudaSuccess;
    auto kern = k_read<Sym, fkvdec::kSectors>;
    if constexpr (sizeof(Sym) == 1) {
        if (c->N <= 8)
            kern = c->N == 4 ? k_read<Sym, fkvdec::kAxes> : k_read<Sym, fkvdec::kScores>;
    }
    const int smem = tables_bytes(c->N, c->L);
    unsigned grid = 0;
    cudaError_t e = decode_grid(c, reinterpret_cast<const void *>(kern), smem, blocks, &grid, TPB);
    if (e != cudaSuccess)
        return e;
    kern<<<grid, TPB, smem, st>>>(
        reinterpret_cast<const double2 *>(pts), n_streams, n, pt_stride, req, n_req, out, c->d_dec, c->d_T,
        c->N, c->L, c->d_status);
    return cudaGetLastError();
}

cudaError_t launch_read(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n,
                        int64_t pt_stride, const int64_t *req, int64_t n_req, void *out,
                        cudaStream_t st)
{
    if (wide(c))
        return read_t(c, pts, n_streams, n, pt_stride, req, n_req, static_cast<uint16_t *>(out), st);
    return read_t(c, pts, n_streams, n, pt_stride, req, n_req, static_cast<uint8_t *>(out), st);
}

template <typename Sym>
cudaError_t append_t(const fkv_ctx *c, double *pts, int64_t n_streams, int64_t pt_stride, int64_t n_old,
                     const Sym *sym, int64_t m, int64_t sym_stride, cudaStream_t st)
{
    if (m <= 0 || n_streams <= 0)
        return cudaSuccess;
    const int L = c->L;
    int64_t head = 0;   // new symbols that finish the stored partial span
    if (n_old % L) {
        head = min(m, L - n_old % L);
        const int64_t blocks = cdiv(n_streams, kThreads);
        if (blocks > 0x7FFFFFFF)
            return cudaErrorInvalidConfiguration;
        k_append<Sym><<<static_cast<unsigned>(blocks), kThreads, 0, st>>>(
            reinterpret_cast<double2 *>(pts), n_streams, pt_stride, n_old, sym, head, sym_stride, n_old / L, 1,
            c->d_V, c->N, c->r, L, c->d_status);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess)
            return e;
    }
    if (m == head)
        return cudaSuccess;
    // every later span starts at the anchor: the bulk span encoder on the
    // remaining symbols, writing from span (n_old + head) / L on
    return span_encode_t(c, sym + head, n_streams, m - head, sym_stride, pts + 2 * ((n_old + head) / L),
                         pt_stride, st);
}

cudaError_t launch_append(const fkv_ctx *c, double *pts, int64_t n_streams, int64_t pt_stride,
                          int64_t n_old, const void *sym, int64_t m, int64_t sym_stride,
                          cudaStream_t st)
{
    if (wide(c))
        return append_t(c, pts, n_streams, pt_stride, n_old, static_cast<const uint16_t *>(sym), m, sym_stride,
                        st);
    return append_t(c, pts, n_streams, pt_stride, n_old, static_cast<const uint8_t *>(sym), m, sym_stride, st);
}

// ------------------------------------------------------------ lossy launches
namespace {

LossyArgs lossy_args(const fkv_ctx *c, const uint32_t *codes, int64_t code_stride, const double *tail,
                     int64_t tail_stride, int64_t n, int bits, int64_t keep_exact)
{
    LossyArgs a;
    const int64_t spans = cdiv(n, c->L);
    a.T = spans > keep_exact ? spans - keep_exact : 0;
    a.codes = codes;
    a.code_stride = code_stride;
    a.words = cdiv(2 * a.T * bits, 32);
    a.tail = reinterpret_cast<const double2 *>(tail);
    a.tail_stride = tail_stride;
    a.bits = bits;
    a.scale = ldexp(1.0, -(bits - 1));
    return a;
}

LossyWalk lossy_walk(const fkv_ctx *c)
{
    LossyWalk q;
    q.V = c->d_V;
    q.N = c->N;
    q.L = c->L;
    q.w = 1.0 - c->r;
    q.r = c->r;
    uint64_t b;
    memcpy(&b, &c->r, sizeof(b));
    const uint64_t m = (b << 11) | (1ull << 63);
    q.inv = m == 1ull << 63 ? 0ull : static_cast<unsigned long long>((static_cast<unsigned __int128>(1) << 127) / m);
    q.er = static_cast<int>(b >> 52);
    memcpy(q.sect_a, c->sect_a, sizeof(q.sect_a));
    q.bound = c->d_dec->bound;
    return q;
}

template <typename Sym>
cudaError_t lossy_decode_t(const fkv_ctx *c, const LossyArgs &a, int64_t n_streams, int64_t n, Sym *sym,
                           int64_t sym_stride, cudaStream_t st)
{
    const int64_t spans = cdiv(n, c->L);
    const int64_t bps = cdiv(spans, kThreads);
    const int64_t n_chunks = n_streams * bps;
    if (n_chunks == 0)
        return cudaSuccess;
    if (bps > 0x7FFFFFFF)
        return cudaErrorInvalidConfiguration;
    const int smem = lossy_table_bytes(c->N) + kThreads / 32 * warp_stage_bytes<Sym>(c->L);
    unsigned grid = 0;
    cudaError_t e = decode_grid(c, reinterpret_cast<const void *>(k_lossy_decode<Sym>), smem, n_chunks, &grid);
    if (e != cudaSuccess)
        return e;
    k_lossy_decode<Sym><<<grid, kThreads, smem, st>>>(a, n, spans, static_cast<int>(bps), n_chunks, sym, sym_stride,
                                                      lossy_walk(c));
    return cudaGetLastError();
}

template <typename Sym>
cudaError_t lossy_read_t(const fkv_ctx *c, const LossyArgs &a, int64_t n_streams, int64_t n, const int64_t *req,
                         int64_t n_req, Sym *out, cudaStream_t st)
{
    const int64_t blocks = cdiv(n_req, kThreads);
    if (blocks == 0)
        return cudaSuccess;
    const int smem = lossy_table_bytes(c->N);
    unsigned grid = 0;
    cudaError_t e = decode_grid(c, reinterpret_cast<const void *>(k_lossy_read<Sym>), smem, blocks, &grid);
    if (e != cudaSuccess)
        return e;
    k_lossy_read<Sym><<<grid, kThreads, smem, st>>>(a, n_streams, n, req, n_req, out, lossy_walk(c),
                                                    c->d_status);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_truncate(const fkv_ctx *c, const double *pts, int64_t n_streams, int64_t n, int64_t pt_stride,
                            int bits, int64_t keep_exact, uint32_t *codes, int64_t code_stride, double *tail,
                            int64_t tail_stride, cudaStream_t st)
{
    const int64_t spans = cdiv(n, c->L);
    const int64_t T = spans > keep_exact ? spans - keep_exact : 0;
    const int64_t words = cdiv(2 * T * bits, 32);
    if (n_streams > 0 && words > 0) {
        const int64_t blocks = min(cdiv(n_streams * cdiv(T, 32), kThreads / 32), static_cast<int64_t>(c->sms) * 8);
        k_truncate<<<static_cast<unsigned>(blocks), kThreads, 0, st>>>(pts, pt_stride, n_streams, T, bits, codes,
                                                                        code_stride, words);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess)
            return e;
    }
    if (tail && n_streams > 0 && spans > T)
        return cudaMemcpy2DAsync(tail, tail_stride * 16, pts + 2 * T, pt_stride * 16, (spans - T) * 16, n_streams,
                                 cudaMemcpyDeviceToDevice, st);
    return cudaSuccess;
}

cudaError_t launch_lossy_decode(const fkv_ctx *c, const uint32_t *codes, int64_t code_stride, const double *tail,
                                int64_t tail_stride, int64_t n_streams, int64_t n, int bits, int64_t keep_exact,
                                void *sym, int64_t sym_stride, cudaStream_t st)
{
    const LossyArgs a = lossy_args(c, codes, code_stride, tail, tail_stride, n, bits, keep_exact);
    if (wide(c))
        return lossy_decode_t(c, a, n_streams, n, static_cast<uint16_t *>(sym), sym_stride, st);
    return lossy_decode_t(c, a, n_streams, n, static_cast<uint8_t *>(sym), sym_stride, st);
}

cudaError_t launch_lossy_read(const fkv_ctx *c, const uint32_t *codes, int64_t code_stride, const double *tail,
                              int64_t tail_stride, int64_t n_streams, int64_t n, int bits, int64_t keep_exact,
                              const int64_t *req, int64_t n_req, void *out, cudaStream_t st)
{
    const LossyArgs a = lossy_args(c, codes, code_stride, tail, tail_stride, n, bits, keep_exact);
    if (wide(c))
        return lossy_read_t(c, a, n_streams, n, req, n_req, static_cast<uint16_t *>(out), st);
    return lossy_read_t(c, a, n_streams, n, req, n_req, static_cast<uint8_t *>(out), st);
}


// ------------------------------------------------------------ ragged launches
namespace {

// Persistent grid for the ragged kernels: the slot count lives on the device,
// so the grid is sized to fill the GPU and the kernels stride over the slots.
template <typename Sym>
cudaError_t ragged_decoder_grid(const fkv_ctx *c, const void *kern, int smem, unsigned *grid)
{
    return decode_grid(c, kern, smem, 1ll << 40, grid, dec_threads<Sym>());
}

template <typename Sym>
cudaError_t encode_ragged_t(const fkv_ctx *c, const Sym *sym, const int64_t *so, int64_t n_streams, double *pts,
                            const int64_t *po, cudaStream_t st)
{
    const auto kern = c->r == 0.5 ? k_span_encode_ragged<true, Sym> : k_span_encode_ragged<false, Sym>;
    unsigned grid = 0;
    cudaError_t e = decode_grid(c, reinterpret_cast<const void *>(kern), 0, 1ll << 40, &grid);
    if (e != cudaSuccess)
        return e;
    kern<<<grid, kThreads, 0, st>>>(sym, so, n_streams, reinterpret_cast<double2 *>(pts), po, enc_args(c),
                                    c->d_status);
    return cudaGetLastError();
}

template <typename Sym>
cudaError_t decode_ragged_t(const fkv_ctx *c, const double *pts, const int64_t *po, int64_t n_streams, Sym *sym,
                            const int64_t *so, cudaStream_t st)
{
    auto kern = k_span_decode_ragged<Sym, fkvdec::kSectors, false>;
    if constexpr (sizeof(Sym) == 1) {
        // words pay from longer spans on (the walk bounds the shorter ones).  64
        // streams of about 262,144 symbols as bytes and as words: sectors (N = 9)
        // 55.1 / 57.2 us at 14 symbols a span, 58.4 / 46.1 at 16, 74.2 / 49.4 at 22;
        // axes 37.1 / 43.4 at 16, 43.0 / 41.2 at 18, 83.9 / 33.0 at 44; scores 78.8 /
        // 82.2 (N = 5) and 86.6 / 92.4 (N = 8) at 20, 77.3 / 69.8 and 83.8 / 85.5 at 24
        const bool words = c->L >= (c->N == 4 ? 18 : c->N <= 8 ? 24 : 16);
        if (c->N == 4)
            kern = words ? k_span_decode_ragged<Sym, fkvdec::kAxes, true>
                         : k_span_decode_ragged<Sym, fkvdec::kAxes, false>;
        else if (c->N <= 8)
            kern = words ? k_span_decode_ragged<Sym, fkvdec::kScores, true>
                         : k_span_decode_ragged<Sym, fkvdec::kScores, false>;
        else if (words)
            kern = k_span_decode_ragged<Sym, fkvdec::kSectors, true>;
    }
    const int smem = tables_bytes(c->N, c->L);
    unsigned grid = 0;
    cudaError_t e = ragged_decoder_grid<Sym>(c, reinterpret_cast<const void *>(kern), smem, &grid);
    if (e != cudaSuccess)
        return e;
    kern<<<grid, dec_threads<Sym>(), smem, st>>>(reinterpret_cast<const double2 *>(pts), po, n_streams, sym, so,
                                                 c->d_dec, c->d_T, c->N, c->L, c->d_status);
    return cudaGetLastError();
}

template <typename Sym>
cudaError_t read_ragged_t(const fkv_ctx *c, const double *pts, const int64_t *po, const int64_t *so,
                          int64_t n_streams, const int64_t *req, int64_t n_req, Sym *out, cudaStream_t st)
{
    auto kern = k_read_ragged<Sym, fkvdec::kSectors>;
    if constexpr (sizeof(Sym) == 1) {
        if (c->N <= 8)
            kern = c->N == 4 ? k_read_ragged<Sym, fkvdec::kAxes> : k_read_ragged<Sym, fkvdec::kScores>;
    }
    const int smem = tables_bytes(c->N, c->L);
    unsigned grid = 0;
    cudaError_t e = ragged_decoder_grid<Sym>(c, reinterpret_cast<const void *>(kern), smem, &grid);
    if (e != cudaSuccess)
        return e;
    const int64_t need = cdiv(n_req, dec_threads<Sym>());
    if (static_cast<int64_t>(grid) > need)
        grid = static_cast<unsigned>(need);
    kern<<<grid, dec_threads<Sym>(), smem, st>>>(reinterpret_cast<const double2 *>(pts), po, so, n_streams, req, n_req,
                                                 out, c->d_dec, c->d_T, c->N, c->L, c->d_status);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_span_encode_ragged(const fkv_ctx *c, const void *sym, const int64_t *so, int64_t n_streams,
                                      double *pts, const int64_t *po, cudaStream_t st)
{
    if (wide(c))
        return encode_ragged_t(c, static_cast<const uint16_t *>(sym), so, n_streams, pts, po, st);
    return encode_ragged_t(c, static_cast<const uint8_t *>(sym), so, n_streams, pts, po, st);
}

cudaError_t launch_span_decode_ragged(const fkv_ctx *c, const double *pts, const int64_t *po, int64_t n_streams,
                                      void *sym, const int64_t *so, cudaStream_t st)
{
    if (wide(c))
        return decode_ragged_t(c, pts, po, n_streams, static_cast<uint16_t *>(sym), so, st);
    return decode_ragged_t(c, pts, po, n_streams, static_cast<uint8_t *>(sym), so, st);
}

cudaError_t launch_read_ragged(const fkv_ctx *c, const double *pts, const int64_t *po, const int64_t *so,
                               int64_t n_streams, const int64_t *req, int64_t n_req, void *out, cudaStream_t st)
{
    if (wide(c))
        return read_ragged_t(c, pts, po, so, n_streams, req, n_req, static_cast<uint16_t *>(out), st);
    return read_ragged_t(c, pts, po, so, n_streams, req, n_req, static_cast<uint8_t *>(out), st);
}

// ------------------------------------------------------------ FP64 probe
// Binary64 add/mul throughput with independent chains: every thread runs
// kChains chains of x <- x * a, x <- x + b (round to nearest, no FMA: the
// encoder's operation mix), whose fixed point b / (1 - a) keeps the values
// bounded.  The chains' sum is written only when it equals an impossible
// value, so the work stays live without a store per thread.
namespace {
constexpr int kFp64Chains = 8;
__device__ double g_fp64_sink;

__global__ void __launch_bounds__(256) k_fp64_rate(int iters, double a, double b)
{
    double x[kFp64Chains];
#pragma unroll
    for (int i = 0; i < kFp64Chains; ++i)
        x[i] = 1.0 + 1e-3 * i + 1e-7 * threadIdx.x;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < kFp64Chains; ++i) {
            x[i] = __dmul_rn(x[i], a);
            x[i] = __dadd_rn(x[i], b);
        }
    }
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < kFp64Chains; ++i)
        s += x[i];
    if (s == -1.0)
        g_fp64_sink = s;
}
}  // namespace

cudaError_t measure_fp64_rate(int device, cudaStream_t st, double *ops_per_s)
{
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess)
        return e;
    const int blocks = sms * 4, iters = 4096;
    cudaEvent_t t0, t1;
    if ((e = cudaEventCreate(&t0)) != cudaSuccess)
        return e;
    if ((e = cudaEventCreate(&t1)) != cudaSuccess) {
        cudaEventDestroy(t0);
        return e;
    }
    float best = 0.0f;
    for (int rep = 0; rep < 4 && e == cudaSuccess; ++rep) {   // the first launch warms up
        cudaEventRecord(t0, st);
        k_fp64_rate<<<blocks, 256, 0, st>>>(iters, 0.99999999, 1e-8);
        cudaEventRecord(t1, st);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaEventSynchronize(t1);
        float ms = 0.0f;
        if (e == cudaSuccess)
            e = cudaEventElapsedTime(&ms, t0, t1);
        if (e == cudaSuccess && rep > 0 && (best == 0.0f || ms < best))
            best = ms;
    }
    cudaEventDestroy(t0);
    cudaEventDestroy(t1);
    if (e != cudaSuccess)
        return e;
    *ops_per_s = 2.0 * kFp64Chains * static_cast<double>(iters) * blocks * 256 / (best * 1e-3);
    return cudaSuccess;
}
