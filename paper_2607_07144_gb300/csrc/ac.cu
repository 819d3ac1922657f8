// Probability-weighted maps (Sec. 6 eq. (1)): the arithmetic-coding form of
// the iterated map, in which symbol c shrinks the interval [lo, hi] to its
// sub-interval of width p(c) at offset F(c).  Decoding is sequential within a
// stream, so the GPU codes independent streams side by side and each stream
// is bound by the latency of its serial chain, interval to interval.  The
// kernels keep on that chain only what the next interval needs.
//
// Integer form (32-bit interval, 64-bit products): with w = hi - lo + 1 and T
// the count total, lo' = lo + floor(w cum(c) / T), hi' = lo + floor(w (cum(c) +
// cnt(c)) / T) - 1; a settled half emits its bit (and the pending opposite
// bits), a middle-half straddle adds a pending bit, and the interval doubles.
// Counts start at 1 and, adaptively, the coded symbol's count grows by one
// (add-one prequential model); otherwise p(c) = 1/N throughout, which is the
// uniform code of Sec. 1.  Bits are written most significant first.
//
// The renormalisation runs in two counted shifts instead of a bit loop: the n
// leading bits in which lo and hi agree leave together, and then lo = 0..,
// hi = 1.. and the e positions after the top bit that are 1 in lo and 0 in hi
// are the middle-half straddles (after either run the interval straddles the
// middle, so no third run follows).
//
// Measured at 96 streams of 17,784 symbols (N = 256, adaptive, one GB300):
// encode 1.38 ms (160 cycles a symbol; 19.8 ms with divisions, bit loops and
// the model on the chain), decode 3.96 ms (450 cycles; 26.9 ms; 4.37 with the
// code words and reciprocals by shuffle and the bits in two branches).  Testing
// a lane's eight symbols at once instead of by halves takes fewer dependent
// steps but more instructions, and one warp issues too few: 4.85 ms.
#include "fkv_internal.h"

namespace {

constexpr uint32_t kQtr = 0x40000000u;

// (hi:lo) << min(n, 32), upper word.
__device__ __forceinline__ uint32_t shl_in(uint32_t hi, uint32_t lo, int n)
{
    return __funnelshift_lc(lo, hi, n);
}

// Middle-half straddles of an interval with lo = 0.., hi = 1..: the positions
// after the top bit, from the left, that hold 1 in lo and 0 in hi (at most 31).
__device__ __forceinline__ int straddles(uint32_t lo, uint32_t hi)
{
    return __clz(static_cast<int>(((~lo | hi) << 1) | 1u));
}

// ceil(2^64 cum / T) for 0 <= cum < T < 2^31, given M = floor((2^64 - 1) / T):
// two 32-bit digits, each a multiply-high estimate that is at most one low.
__device__ __forceinline__ unsigned long long scaled_up(uint32_t cum, uint32_t T, unsigned long long M)
{
    unsigned long long a = static_cast<unsigned long long>(cum) << 32;
    uint32_t q1 = static_cast<uint32_t>(__umul64hi(a, M));
    uint32_t r = static_cast<uint32_t>(a) - q1 * T;
    if (r >= T) {
        r -= T;
        ++q1;
    }
    a = static_cast<unsigned long long>(r) << 32;
    uint32_t q0 = static_cast<uint32_t>(__umul64hi(a, M));
    r = static_cast<uint32_t>(a) - q0 * T;
    if (r >= T) {
        r -= T;
        ++q0;
    }
    return ((static_cast<unsigned long long>(q1) << 32) | q0) + (r != 0 ? 1ull : 0ull);
}

// floor((d + 1) F / 2^64): with F = ceil(2^64 cum / T) it is exactly
// floor((d + 1) cum / T), since the excess is below 2^-32 and the quotient's
// fraction is a multiple of 1 / T > 2^-32 away from the next integer.
__device__ __forceinline__ uint32_t scale_by(uint32_t d, unsigned long long F)
{
    const uint32_t fl = static_cast<uint32_t>(F), fh = static_cast<uint32_t>(F >> 32);
    const unsigned long long low = static_cast<unsigned long long>(d) * fl + fl;
    const unsigned long long t = static_cast<unsigned long long>(d) * fh + (static_cast<unsigned long long>(fh) + (low >> 32));
    return static_cast<uint32_t>(t >> 32);
}

// Encoder: one block of three warps per stream, passing batches of 32 symbols
// on through shared memory.  The symbols are known, so the model runs ahead of
// the interval: warp 0 works out each symbol's cumulative counts, one symbol
// per lane (a prefix table as of the batch's start, corrected by the batch's
// own earlier symbols), and from them the fractions ceil(2^64 cum / T), whose
// product with the interval's width needs no division.  Lane 0 of warp 1 walks
// the interval, the serial chain, and leaves each symbol's settled bits and
// straddles to lane 0 of warp 2, which packs them.  The upper fraction of a
// symbol whose interval reaches the top is all ones, which scale_by turns into
// w - 1.
template <typename Sym, int CPL>
__global__ void __launch_bounds__(96)
k_ac_encode(const Sym *__restrict__ sym, int64_t n, int64_t sym_stride, int N, int adaptive,
            uint32_t *__restrict__ words, int64_t word_stride, int64_t *__restrict__ nbits, unsigned *status)
{
    __shared__ ulonglong2 frac[2][32];
    __shared__ uint2 settled[2][32];             // the settled interval's lower end; settled bits | straddles << 8
    __shared__ uint32_t last_lo;
    __shared__ __align__(16) uint32_t cnt[32 * CPL], below[32 * CPL];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t stream = blockIdx.x;
    const Sym *src = sym + stream * sym_stride;
    const int64_t batches = (n + 31) >> 5;
    auto batch_len = [&](int64_t b) { return static_cast<int>(min(static_cast<int64_t>(32), n - 32 * b)); };
    // model (warp 0)
    bool bad = false;
    uint32_t next = 0;
    // interval (lane 0 of warp 1)
    uint32_t lo = 0, hi = 0xFFFFFFFFu;
    // packer (lane 0 of warp 2)
    uint32_t *out = words + stream * word_stride;
    int64_t follow = 0, wi = 0;
    unsigned long long acc = 0;
    int an = 0;                                  // bits in acc, below 32 between symbols
    auto put = [&](uint32_t v, int len) {        // len <= 32 bits
        acc = (acc << len) | v;
        an += len;
        if (an >= 32) {
            an -= 32;
            if (wi < word_stride)
                out[wi] = static_cast<uint32_t>(acc >> an);
            ++wi;
        }
    };
    auto put_settled = [&](uint32_t b) {         // a settled bit and the pending opposite ones
        put(b, 1);
        while (follow > 0) {
            const int len = follow < 31 ? static_cast<int>(follow) : 31;
            put(b ? 0u : (1u << len) - 1u, len);
            follow -= len;
        }
    };
    if (warp == 0) {
        for (int i = lane; i < 32 * CPL; i += 32) {
            cnt[i] = i < N ? 1u : 0u;
            below[i] = min(i, N);
        }
        next = lane < n ? src[lane] : 0u;
        __syncwarp();
    }
    for (int64_t b = 0; b < batches + 2; ++b) {
        if (warp == 0 && b < batches) {
            const int64_t k = 32 * b + lane;
            uint32_t c = next;
            next = k + 32 < n ? src[k + 32] : 0u;
            if (c >= static_cast<uint32_t>(N)) {   // not a symbol: coded as N - 1, reported
                bad = true;
                c = N - 1;
            }
            uint32_t cum = c, f = 1, T = N;
            if (adaptive) {
                cum = below[c];
                f = cnt[c];
                T = static_cast<uint32_t>(N + k);
#pragma unroll
                for (int j = 0; j < 31; ++j) {
                    const uint32_t cj = __shfl_sync(0xFFFFFFFFu, c, j);
                    cum += j < lane && cj < c ? 1u : 0u;
                    f += j < lane && cj == c ? 1u : 0u;
                }
            }
            const unsigned long long M = 0xFFFFFFFFFFFFFFFFull / T;
            ulonglong2 v;
            v.x = scaled_up(cum, T, M);
            v.y = cum + f == T ? 0xFFFFFFFFFFFFFFFFull : scaled_up(cum + f, T, M);
            frac[b & 1][lane] = v;
            if (adaptive) {
                __syncwarp();
                if (k < n)
                    atomicAdd(&cnt[c], 1u);
                __syncwarp();
                uint32_t own[CPL], sum = 0;
#pragma unroll
                for (int j = 0; j < CPL; j += 4) {
                    const uint4 q = *reinterpret_cast<const uint4 *>(&cnt[lane * CPL + j]);
                    own[j] = sum;
                    own[j + 1] = own[j] + q.x;
                    own[j + 2] = own[j + 1] + q.y;
                    own[j + 3] = own[j + 2] + q.z;
                    sum = own[j + 3] + q.w;
                }
                uint32_t incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    incl += lane >= o ? t : 0u;
                }
                const uint32_t base = incl - sum;
#pragma unroll
                for (int j = 0; j < CPL; j += 4)
                    *reinterpret_cast<uint4 *>(&below[lane * CPL + j]) =
                        make_uint4(base + own[j], base + own[j + 1], base + own[j + 2], base + own[j + 3]);
                __syncwarp();
            }
        } else if (threadIdx.x == 32 && b >= 1 && b <= batches) {
            const ulonglong2 *fr = frac[(b - 1) & 1];
            uint2 *to = settled[(b - 1) & 1];
            const int m = batch_len(b - 1);
            ulonglong2 F = fr[0];
#pragma unroll 4
            for (int k = 0; k < m; ++k) {
                const ulonglong2 Fn = fr[(k + 1) & 31];
                const uint32_t d = hi - lo;
                const uint32_t l2 = lo + scale_by(d, F.x);
                const uint32_t h2 = lo + scale_by(d, F.y) - (F.y == 0xFFFFFFFFFFFFFFFFull ? 0u : 1u);
                F = Fn;
                const int s = __clz(static_cast<int>(l2 ^ h2));        // settled bits
                lo = shl_in(l2, 0u, s);
                hi = shl_in(h2, 0xFFFFFFFFu, s);
                const int e = straddles(lo, hi);
                lo = (lo << e) & 0x7FFFFFFFu;
                hi = shl_in(hi, 0xFFFFFFFFu, e) | 0x80000000u;
                to[k] = make_uint2(l2, static_cast<uint32_t>(s | (e << 8)));
            }
            last_lo = lo;
        } else if (threadIdx.x == 64 && b >= 2) {
            const uint2 *from = settled[b & 1];
            const int m = batch_len(b - 2);
            for (int k = 0; k < m; ++k) {
                const uint2 q = from[k];
                const int s = static_cast<int>(q.y & 0xFFu);
                if (s > 0) {
                    // the first settled bit, the pending opposite bits, the other settled
                    // bits: 1 0..0 or 0 1..1 is 2^follow - 1 + bit
                    const uint32_t bit = q.x >> 31;
                    const uint32_t rest = (q.x & 0x7FFFFFFFu) >> (32 - s);
                    if (follow + s <= 32) {
                        const uint32_t lead = (1u << static_cast<int>(follow)) - 1u + bit;
                        put((lead << (s - 1)) | rest, static_cast<int>(follow) + s);
                        follow = 0;
                    } else {
                        put_settled(bit);
                        put(rest, s - 1);
                    }
                }
                follow += q.y >> 8;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 64) {
        ++follow;
        put_settled(n > 0 && last_lo >= kQtr ? 1u : 0u);
        if (an > 0 && wi < word_stride)
            out[wi] = static_cast<uint32_t>(acc << (32 - an));        // the last, partial word
        const int64_t nb = wi * 32 + an;
        const bool overflow = nb > word_stride * 32;
        nbits[stream] = overflow ? -1 : nb;
        if (overflow)
            atomicOr(status, FKV_ST_CORRUPT);
    }
    if (bad)
        atomicOr(status, FKV_ST_CORRUPT);
}

// Decoder: one warp per stream, the cumulative counts of CPL symbols (and of
// the next lane's first) in each lane's registers.  The symbol is the last one
// with floor(w cum / T) <= val - lo, which is w cum <= (val - lo + 1) T - 1
// without a division: every lane tests its first symbol (the owner is the last
// lane that passes) and, at the same time, searches its own symbols by halves
// and works out the interval of the one it finds (the quotients by T from
// reciprocals prepared 32 symbols at a time); the owner's interval and symbol
// then come by shuffle.  The bits to come sit in a 64-bit window refilled
// without a branch from 64 code words in shared memory, of which 32 symbols
// use at most 32 (SMALL: N + n < 2^28, so that a symbol settles fewer than 32
// bits: an interval of 2^30 or more leaves at least 4, which doubles at most
// 30 times).  Larger counts take a symbol's bits in two steps.
template <typename Sym, int CPL, bool SMALL>
__global__ void __launch_bounds__(32)
k_ac_decode(const uint32_t *__restrict__ words, int64_t word_stride, const int64_t *__restrict__ nbits, int64_t n,
            int N, int adaptive, Sym *__restrict__ sym, int64_t sym_stride, unsigned *status)
{
    constexpr unsigned kAll = 0xFFFFFFFFu;
    constexpr int kWords = SMALL ? 64 : 128;      // a batch of 32 symbols uses at most half
    __shared__ uint32_t code[kWords];
    __shared__ unsigned long long recip[32];
    const int lane = threadIdx.x;
    const int64_t stream = blockIdx.x;
    const uint32_t *in = words + stream * word_stride;
    Sym *dst = sym + stream * sym_stride;
    int64_t nb = nbits[stream];
    if (nb < 0 || nb > word_stride * 32) {        // not a code this call can read
        if (lane == 0)
            atomicOr(status, FKV_ST_CORRUPT);
        nb = 0;
    }
    // word q of the code, the bits past the code's end read as zero
    auto word_at = [&](int64_t q) -> uint32_t {
        const int64_t left = nb - 32 * q;
        if (left <= 0)
            return 0u;
        const uint32_t w = __ldg(in + q);
        return left >= 32 ? w : w & (0xFFFFFFFFu << (32 - static_cast<int>(left)));
    };
    // code[] holds words base .. base + kWords - 1 (word q at q mod kWords), the
    // 32 after them are on their way in `ahead`
    for (int i = lane; i < kWords; i += 32)
        code[i] = word_at(i);
    int64_t wq = kWords + lane;
    uint32_t ahead = word_at(wq);
    __syncwarp();
    uint32_t cum[CPL + 1];                        // counts below symbols lane CPL + j
#pragma unroll
    for (int j = 0; j <= CPL; ++j)
        cum[j] = min(lane * CPL + j, N);
    uint32_t lo = 0, hi = 0xFFFFFFFFu, val = code[0];
    unsigned long long win = static_cast<unsigned long long>(code[1]) << 32;   // bits to come
    int have = 32;                                // of them valid, from the top: at least 32 between uses
    unsigned taken = 2;                           // words already in the window
    unsigned loaded = kWords;                     // words that code[] has held
    auto use = [&](int len) {                     // drop len <= 32 bits
        const uint32_t w = code[taken & (kWords - 1)];
        win <<= len;
        have -= len;
        const bool refill = have < 32;
        win |= refill ? static_cast<unsigned long long>(w) << (32 - have) : 0ull;
        have += refill ? 32 : 0;
        taken += refill ? 1u : 0u;
    };
    uint32_t T = N;
    unsigned long long M = 0xFFFFFFFFFFFFFFFFull / T;
    for (int64_t k0 = 0; k0 < n; k0 += 32) {
        const int len = static_cast<int>(min(static_cast<int64_t>(32), n - k0));
        __syncwarp();
        if (adaptive)
            recip[lane] = 0xFFFFFFFFFFFFFFFFull / (T + lane);
        // keep half of code[] ahead of the window
        while (loaded - taken <= kWords - 32) {
            code[(loaded + lane) & (kWords - 1)] = ahead;
            loaded += 32;
            wq += 32;
            ahead = word_at(wq);
        }
        __syncwarp();
        uint32_t pending = 0;
        for (int k = 0; k < len; ++k) {
            if (adaptive)
                M = recip[k];
            const uint32_t d = hi - lo, v = val - lo;
            const unsigned long long R = static_cast<unsigned long long>(v) * T + (T - 1);
            auto passes = [&](uint32_t x) { return static_cast<unsigned long long>(d) * x + x <= R; };
            const unsigned has = __ballot_sync(kAll, passes(cum[0]));
            const int o = 31 - __clz(static_cast<int>(has));   // lane 0 always passes: its count is 0
            uint32_t w[CPL + 1];
#pragma unroll
            for (int j = 0; j <= CPL; ++j)
                w[j] = cum[j];
            int off = 0;
#pragma unroll
            for (int h = CPL / 2; h >= 1; h >>= 1) {
                const bool up = passes(w[h]);
                off += up ? h : 0;
#pragma unroll
                for (int j = 0; j <= h; ++j)
                    w[j] = up ? w[j + h] : w[j];
            }
            // floor((d + 1) x / T): the estimate is at most one low
            auto quot = [&](uint32_t x) {
                const unsigned long long p = static_cast<unsigned long long>(d) * x + x;
                const uint32_t q = static_cast<uint32_t>(__umul64hi(p, M));
                const uint32_t r = static_cast<uint32_t>(p) - q * T;
                return q + (r >= T ? 1u : 0u);
            };
            uint32_t l2 = lo + quot(w[0]), h2 = lo + quot(w[1]) - 1u;
            l2 = __shfl_sync(kAll, l2, o);
            h2 = __shfl_sync(kAll, h2, o);
            const int c = __shfl_sync(kAll, min(lane * CPL + off, N - 1), o);
            pending = lane == k ? static_cast<uint32_t>(c) : pending;
            const int s = __clz(static_cast<int>(l2 ^ h2));
            lo = shl_in(l2, 0u, s);
            hi = shl_in(h2, 0xFFFFFFFFu, s);
            const int e = straddles(lo, hi);
            lo = (lo << e) & 0x7FFFFFFFu;
            hi = shl_in(hi, 0xFFFFFFFFu, e) | 0x80000000u;
            if (SMALL) {
                val = shl_in(val, static_cast<uint32_t>(win >> 32), s + e);
                use(s + e);
            } else {
                val = shl_in(val, static_cast<uint32_t>(win >> 32), s);
                use(s);
                val = shl_in(val, static_cast<uint32_t>(win >> 32), e);
                use(e);
            }
            val ^= e > 0 ? 0x80000000u : 0u;
            if (adaptive) {
                const int t = c - lane * CPL;
#pragma unroll
                for (int j = 0; j <= CPL; ++j)
                    cum[j] += j > t ? 1u : 0u;
                ++T;
            }
        }
        if (lane < len)                           // 32 symbols per store
            dst[k0 + lane] = static_cast<Sym>(pending);
    }
}

// Symbols per lane: N <= 256 comes as uint8, up to 1024 as uint16.
template <typename Sym>
constexpr int kPerLane = sizeof(Sym) == 1 ? 8 : 32;

template <typename Sym>
cudaError_t ac_encode_t(const fkv_ctx *c, const Sym *sym, int64_t n_streams, int64_t n, int64_t sym_stride,
                        int adaptive, uint32_t *words, int64_t word_stride, int64_t *nbits, cudaStream_t st)
{
    if (n_streams > 0x7FFFFFFF)
        return cudaErrorInvalidConfiguration;
    k_ac_encode<Sym, kPerLane<Sym>><<<static_cast<unsigned>(n_streams), 96, 0, st>>>(
        sym, n, sym_stride, c->N, adaptive, words, word_stride, nbits, c->d_status);
    return cudaGetLastError();
}

template <typename Sym>
cudaError_t ac_decode_t(const fkv_ctx *c, const uint32_t *words, int64_t word_stride, const int64_t *nbits,
                        int64_t n_streams, int64_t n, int adaptive, Sym *sym, int64_t sym_stride, cudaStream_t st)
{
    if (n_streams > 0x7FFFFFFF)
        return cudaErrorInvalidConfiguration;
    const auto kern = n + c->N < (int64_t(1) << 28) ? k_ac_decode<Sym, kPerLane<Sym>, true>
                                                    : k_ac_decode<Sym, kPerLane<Sym>, false>;
    kern<<<static_cast<unsigned>(n_streams), 32, 0, st>>>(words, word_stride, nbits, n, c->N, adaptive, sym, sym_stride,
                                                          c->d_status);
    return cudaGetLastError();
}

}  // namespace

int64_t ac_capacity_words(int N, int64_t n)
{
    int per = 1;
    while ((int64_t(1) << per) < N + n)
        ++per;
    return (n * (per + 1) + 2 + 31) / 32 + 1;
}

cudaError_t launch_ac_encode(const fkv_ctx *c, const void *sym, int64_t n_streams, int64_t n, int64_t sym_stride,
                             int adaptive, uint32_t *words, int64_t word_stride, int64_t *nbits, cudaStream_t st)
{
    if (n_streams <= 0)
        return cudaSuccess;
    if (c->N > 256)
        return ac_encode_t(c, static_cast<const uint16_t *>(sym), n_streams, n, sym_stride, adaptive, words,
                           word_stride, nbits, st);
    return ac_encode_t(c, static_cast<const uint8_t *>(sym), n_streams, n, sym_stride, adaptive, words, word_stride,
                       nbits, st);
}

cudaError_t launch_ac_decode(const fkv_ctx *c, const uint32_t *words, int64_t word_stride, const int64_t *nbits,
                             int64_t n_streams, int64_t n, int adaptive, void *sym, int64_t sym_stride, cudaStream_t st)
{
    if (n_streams <= 0 || n <= 0)
        return cudaSuccess;
    if (c->N > 256)
        return ac_decode_t(c, words, word_stride, nbits, n_streams, n, adaptive, static_cast<uint16_t *>(sym),
                           sym_stride, st);
    return ac_decode_t(c, words, word_stride, nbits, n_streams, n, adaptive, static_cast<uint8_t *>(sym), sym_stride,
                       st);
}
