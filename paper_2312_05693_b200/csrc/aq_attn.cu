// Log2 quantization of the softmax output (paper Eq. 3, Sec. 5.1) and the attention-times-value
// product on its codes, where every product is a shift of the int8 value code.
#include <cooperative_groups.h>
#include <cuda.h>

#include "aq_attn_parts.cuh"
#include "aq_common.cuh"
#include "aq_quant_math.cuh"

namespace cg = cooperative_groups;

namespace aq {

namespace {

constexpr int kLog2Ctas = 4;                            // CTAs of 256 threads per SM, all resident at once (codes)
constexpr int kLog2MaxThreads = 512;                    // the maximum: clusters of eight CTAs, two CTAs per SM, all resident at once
constexpr int kLog2InFlight = 8;                        // 16-byte loads a thread has in flight

// ---- layer-wide max |x| as an fp16 bit pattern (NaN ignored, Inf counts as 65504) -------------
// 16-byte loads where the pointer allows; what they leave (the ragged tail, or all of an array that lies elsewhere) goes round
// the threads one by one.
// Every cluster leaves its word in the control block; the first CTA sets the status word up.
__global__ void __cluster_dims__(kRangeCtas, 1, 1) __launch_bounds__(kLog2MaxThreads, 2)
log2_absmax_kernel(const __half* __restrict__ x, long long count, Control* __restrict__ ctl) {
    cluster_started_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");      // launched while the kernel ahead drains
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->status = 0;
    unsigned int b = 0;
    auto take = [&](unsigned int hb) {
        hb &= 0x7FFFu;
        if (hb > 0x7C00u) return;
        if (hb == 0x7C00u) hb = 0x7BFFu;
        b = max(b, hb);
    };
    const bool vec = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
    const long long nvec = vec ? count / 8 : 0;
    const uint4* xv = reinterpret_cast<const uint4*>(x);
    // two values per instruction: the half2 maximum returns the other operand when one is NaN, so NaN
    // never enters; Inf does and is replaced by the largest finite value below
    __half2 m2 = __float2half2_rn(0.0f);
    const long long stride = (long long)gridDim.x * blockDim.x, at = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    auto take8 = [&](const uint4& d) {
        const uint32_t w[4] = {d.x & 0x7FFF7FFFu, d.y & 0x7FFF7FFFu, d.z & 0x7FFF7FFFu, d.w & 0x7FFF7FFFu};
#pragma unroll
        for (int t = 0; t < 4; ++t) m2 = __hmax2(m2, *reinterpret_cast<const __half2*>(&w[t]));
    };
    // whole batches without a test in them, then the rest (one load at a time with its own test: 72 us instead of 45)
    const uint4* p = xv + at;
    long long left = nvec - at;                             // vectors from p to the end
    for (; left > (kLog2InFlight - 1) * stride; left -= kLog2InFlight * stride, p += kLog2InFlight * stride) {
        uint4 d[kLog2InFlight];
#pragma unroll
        for (int k = 0; k < kLog2InFlight; ++k) d[k] = __ldg(p + k * stride);
#pragma unroll
        for (int k = 0; k < kLog2InFlight; ++k) take8(d[k]);
    }
    for (; left > 0; left -= stride, p += stride) take8(__ldg(p));
    {
        const uint32_t mw = *reinterpret_cast<const uint32_t*>(&m2);
        take(mw & 0xFFFFu);
        take(mw >> 16);
    }
    for (long long i = nvec * 8 + at; i < count; i += stride) take(__half_as_ushort(x[i]));
    __shared__ unsigned int peers[kRangeCtas];
    cluster_started_wait();
    leave_range<false, kLog2MaxThreads>(ctl, b, 0u, peers, cg::this_cluster().map_shared_rank(&peers[cg::this_cluster().block_rank()], 0));
}

// A positive fp16 bit pattern as mant * 2^expo with 1024 <= mant < 2048.
__device__ __forceinline__ void half_parts(unsigned int hb, int& mant, int& expo) {
    const int ex = (int)(hb >> 10), fr = (int)(hb & 0x3FFu);
    if (ex > 0) { mant = 1024 + fr; expo = ex - 25; }
    else {                                         // subnormal: fr * 2^-24, fr > 0
        const int sh = __clz(fr) - 21;             // brings the leading one to bit 10
        mant = fr << sh;
        expo = -24 - sh;
    }
}

// Eq. 3: k = clip(round(-log2(|x| / max)), 0, kmax), stored as Sign(x) * (k + 1), 0 for zero / NaN.
// The rounding is decided with integers: -log2(r) = (Eb - Ea) + log2(mb / ma), and log2(mb / ma) passes
// +-1/2 exactly when mb^2 passes 2 ma^2 or ma^2 / 2 (mantissas are 11-bit integers).
// The two mantissa thresholds of the rounding rule for a given maximum mantissa mb (1024..2047):
// t_up = largest ma with 2 ma^2 <= mb^2 (below or at it k rounds up), t_down = smallest ma with
// ma^2 > 2 mb^2 (from it on k rounds down).
__device__ __forceinline__ void log2_thresholds(int mb, int& t_up, int& t_down) {
    int a = (int)(sqrtf(0.5f * (float)mb * (float)mb));
    while (2 * (a + 1) * (a + 1) <= mb * mb) ++a;
    while (2 * a * a > mb * mb) --a;
    t_up = a;
    int b = (int)(sqrtf(2.0f * (float)mb * (float)mb));
    while (b * b > 2 * mb * mb) --b;
    while ((b + 1) * (b + 1) <= 2 * mb * mb) ++b;
    t_down = b + 1;
}

__device__ __forceinline__ int log2_code(unsigned int raw, unsigned int mb_bits, int eb, int t_up, int t_down, int kmax) {
    unsigned int hb = raw & 0x7FFFu;
    const bool none = hb == 0 || hb > 0x7C00u || mb_bits == 0;      // zero, NaN, or an all-zero layer
    hb = min(hb, 0x7BFFu);                                           // Inf counts as the largest finite value
    // Without branches (softmax outputs mix normal and subnormal values inside every warp): the exact
    // conversion to binary32 normalises subnormals, |x| = (1024 + top ten fraction bits) * 2^(E - 10).
    const unsigned int fb = __float_as_uint(__half2float(__ushort_as_half((unsigned short)hb)));
    const int ma = 1024 + (int)((fb >> 13) & 0x3FFu);
    const int ea = (int)(fb >> 23) - 137;
    int k = eb - ea + (ma <= t_up ? 1 : 0) - (ma >= t_down ? 1 : 0);
    k = min(max(k, 0), kmax) + 1;
    return none ? 0 : ((raw & 0x8000u) ? -k : k);
}

// codes -> weights: c > 0 -> 128 >> (c - 1); 0 -> 0; a negative code is not representable here:
// it is recorded in the status word (11) and treated as 0.
__device__ __forceinline__ uint32_t log2_factors4(uint32_t c4, bool& bad) {
    uint32_t o = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int c = (int)(int8_t)((c4 >> (8 * t)) & 0xFFu);
        bad |= c < 0;
        o |= (c > 0 ? (128u >> (c - 1)) : 0u) << (8 * t);
    }
    return o;
}

// 4-bit codes in half2 arithmetic. k does not increase with |x|, so k = #{ j in 1..7 : |x| < B_j } with B_j the
// smallest half whose k is below j. By the integer rule above, k <= j - 1 needs, at exponent Eb - j, a mantissa
// from t_down on, and at exponent Eb - j + 1 a mantissa above t_up; one exponent lower nothing qualifies, one
// higher everything does. So B_j = t_down * 2^(Eb - j) when t_down is a mantissa (<= 2047), else
// (t_up + 1) * 2^(Eb - j + 1), rounded up to a half where it falls between subnormals (the inputs are halves,
// so that keeps the comparison's outcome). Seven compares and adds for two elements replace the exponent and
// mantissa arithmetic per element.
struct Log2Fast {
    __half2 bound[7];
};
__device__ __forceinline__ Log2Fast log2_fast_bounds(int mb, int eb, int t_up, int t_down) {
    Log2Fast f;
#pragma unroll
    for (int j = 1; j <= 7; ++j) {
        const float b = t_down <= 2047 ? ldexpf((float)t_down, eb - j) : ldexpf((float)max(t_up + 1, 1024), eb - j + 1);
        f.bound[j - 1] = __half2half2(__float2half_ru(b));
    }
    (void)mb;
    return f;
}
// Two halves -> (k + 1) * valid as halves (codes), or 2^(7 - k) * valid (factors); valid = 0 for zero and NaN.
template <bool FACTORS>
__device__ __forceinline__ __half2 log2_fast2(__half2 x2, const Log2Fast& f) {
    const __half2 mag = __habs2(x2);
    const __half2 valid = __hgt2(mag, __float2half2_rn(0.0f));                // 1 or 0; NaN compares false
    const __half2 ax = __hmin2(mag, __float2half2_rn(65504.0f));              // Inf counts as the largest finite value (a NaN lane becomes 65504 here and is dropped by valid)
    __half2 r = __float2half2_rn(FACTORS ? 128.0f : 1.0f);
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        const __half2 below = __hlt2(ax, f.bound[j]);                         // 1 or 0
        if (FACTORS) r = __hfma2(below, __float2half2_rn(-(float)(64 >> j)), r);   // 128 - 64 - 32 - ... = 2^(7 - k)
        else r = __hadd2(r, below);
    }
    return __hmul2(r, valid);
}

// Byte factors of eight values where all bounds are normal halves: one mantissa, exponents one apart, so as integers B_j = B_1 - 1024 (j - 1)
// and k = min((B_1 + 1023 - |x|) >> 10, 7) on the bit patterns, two to a register. Four k's select four bytes of the eight factors in one
// byte permute; zeros, NaNs and negative inputs (recorded) give 0. cap: B_1 + 1023 in both halves. NEAR: the largest remainders (of 1024) of
// the values with k < 7, the lanes apart: a B_1 larger by d, d < 1024, changes the factors where the remainder is 1024 - d or more, and no others;
// least: the least distance from cap so far (0: a value of cap or more, negative or NaN).
template <bool NEAR>
__device__ __forceinline__ uint2 log2_factors8(const uint4& d, uint32_t cap, uint32_t& near, uint32_t& least, bool& bad) {
    const uint32_t w[4] = {d.x, d.y, d.z, d.w};
    uint32_t below[4], some[4], sel[2];
    near = 0u;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        some[t] = __hgt2_mask(*reinterpret_cast<const __half2*>(&w[t]), __float2half2_rn(0.0f));
        const uint32_t all = cap - __vminu2(w[t], cap);
        if (NEAR) least = __vminu2(least, all);
        below[t] = __vminu2(all, 0x1C001C00u);                // 7 * 1024: k = 7, remainder 0
        if (NEAR) near = __vmaxu2(near, below[t] & 0x03FF03FFu);
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {                             // k of four values in four nibbles
        const uint32_t k = ((below[2 * t] >> 10) & 0x00070007u) | ((below[2 * t + 1] >> 2) & 0x07000700u);
        sel[t] = k | (k >> 12);
    }
    if ((w[0] | w[1] | w[2] | w[3]) & 0x80008000u) {
#pragma unroll
        for (int t = 0; t < 4; ++t)
            bad |= __hlt2_mask(*reinterpret_cast<const __half2*>(&w[t]), __float2half2_rn(0.0f)) != 0u;
    }
    return make_uint2(__byte_perm(0x10204080u, 0x01020408u, sel[0] & 0x7777u) & __byte_perm(some[0], some[1], 0x6420),
                      __byte_perm(0x10204080u, 0x01020408u, sel[1] & 0x7777u) & __byte_perm(some[2], some[3], 0x6420));
}
// B_1 of a maximum, or 0 where not all bounds are normal halves (see log2_fast_bounds: the same, as a bit pattern).
__device__ __forceinline__ unsigned int log2_first_bound(unsigned int max_bits) {
    if (max_bits == 0u) return 0u;
    int mb, eb, t_up, t_down;
    half_parts(max_bits, mb, eb);
    log2_thresholds(mb, t_up, t_down);
    const int bits = t_down <= 2047 ? ((eb + 24) << 10) + t_down - 1024 : ((eb + 25) << 10) + max(t_up + 1, 1024) - 1024;
    return bits >= 0x1C00 ? (unsigned int)bits : 0u;         // B_7 = B_1 / 64
}
__device__ __forceinline__ uint8_t log2_factor(unsigned int raw, unsigned int mb_bits, int eb, int t_up, int t_down, bool& bad) {
    const int c = log2_code(raw, mb_bits, eb, t_up, t_down, 7);
    bad |= c < 0;
    return (uint8_t)(c > 0 ? 128u >> (c - 1) : 0u);
}

// ---- byte factors in one pass over x -----------------------------------------------------------
// The maximum is known only when all of x has been read, but nearly all factors are settled before: by a maximum that is a little too small
// a factor comes out wrong only where the value lies just under a bound, and values from 2^-6.5 of the maximum down have the
// last factor whatever it is. So a cooperative grid reads x once, writes the factors by the largest maximum seen so far, and notes in shared
// memory the vectors of eight that a maximum up to the lead further would change; when all is read the grid meets, and
// the noted vectors are written again by the true maximum. The lead reaches to a maximum of 1, so that no softmax output goes
// beyond it; were a maximum beyond it to come all the same, the batches that it found written are written again.
// That pays where a sample, taken before, shows that 1 is near and that few vectors will be noted; elsewhere (softmax of small differences)
// the grid reads x for its maximum alone and again, from its end, for the factors, as the two kernels do that this replaces for arrays
// larger than the L2 keeps. Rules of kLead, kOnceShare: a noted vector costs a scattered read and a partial write, 28 heads of 2048 x 2048 some
// 20 us for every hundredth of the vectors while the maximum stays where it is (117 us with half an octave to 1 and 15 notes in 1000 vectors, 92.3 in two
// kernels, 77 without notes); one that rises soon costs less (2.5 standard deviations of scores, 278 steps and 14 in 1000: 83). The
// decision is one for the grid: where some CTAs read twice and others wrote, all waited for the slower ones (126 us).
// Bound by memory: 2 bytes in, 1 out per value, at 5.6 TB/s between the meetings (32 x 2048 x 2048).
constexpr int kOnceThreads = 1024, kOnceNotes = 10240;
constexpr unsigned int kLead = 300;                     // of 1024 steps to twice the bound
constexpr int kOnceShare = 64;                          // one vector in so many may be noted
// Bytes of x, read last, that the L2 is to keep for the second reading: what comes before is marked as first to go (28 / 32 / 56 heads read
// twice without the marks 96.7 / 111.1 / -, with them and 116 MB 92.0 / 104.6 / 181.9, 97 MB 91.9 / 104.5 / 180.9, 78 MB 91.1 / 104.1 / 179.9).
constexpr long long kOnceKeep = 78ll << 20;
constexpr unsigned int kBoundOfOne = 0x39A9u;           // B_1 where the maximum is 1: 1449 * 2^-11, 1449 the least whole number above 1024 sqrt(2)
constexpr int kOnceChanges = 8;

// The factors of a thread's vectors from v downwards (see log2_codes_kernel); whether a negative value was met.
__device__ __forceinline__ bool log2_write_again(const uint4* xv, uint2* out, long long v, long long stride, uint32_t cap) {
    bool bad = false;
    uint32_t near, least = 0u;
    const uint4* src = xv + v;
    uint2* dst = out + v;
    for (; v >= (kLog2InFlight - 1) * stride; v -= kLog2InFlight * stride, src -= kLog2InFlight * stride, dst -= kLog2InFlight * stride) {
        uint4 d[kLog2InFlight];
#pragma unroll
        for (int k = 0; k < kLog2InFlight; ++k) d[k] = __ldg(src - k * stride);
#pragma unroll
        for (int k = 0; k < kLog2InFlight; ++k) __stcs(dst - k * stride, log2_factors8<false>(d[k], cap, near, least, bad));
    }
    for (; v >= 0; v -= stride, src -= stride, dst -= stride) __stcs(dst, log2_factors8<false>(__ldg(src), cap, near, least, bad));
    return bad;
}

// The same where not all bounds are normal halves, by comparisons with each (see log2_codes_kernel).
__device__ __forceinline__ bool log2_write_by_bounds(const uint4* xv, uint2* out, long long v, long long nvec, long long stride, unsigned int mb_bits, int mb, int eb,
                                                     int t_up, int t_down) {
    if (mb_bits == 0u) {
        for (; v < nvec; v += stride) __stcs(out + v, make_uint2(0u, 0u));
        return false;
    }
    const Log2Fast fast = log2_fast_bounds(mb, eb, t_up, t_down);
    bool bad = false;
#pragma unroll 4
    for (; v < nvec; v += stride) {
        const uint4 d = __ldg(xv + v);
        const uint32_t w[4] = {d.x, d.y, d.z, d.w};
        uint32_t m[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const __half2 x2 = *reinterpret_cast<const __half2*>(&w[t]);
            __half2 r = log2_fast2<true>(x2, fast);
            const __half2 neg = __hlt2(x2, __float2half2_rn(0.0f));
            bad |= (*reinterpret_cast<const uint32_t*>(&neg) != 0u);
            r = __hadd2(__hfma2(neg, __hneg2(r), r), __float2half2_rn(1024.0f));
            m[t] = *reinterpret_cast<uint32_t*>(&r);
        }
        __stcs(out + v, make_uint2(__byte_perm(m[0], m[1], 0x6420), __byte_perm(m[2], m[3], 0x6420)));
    }
    return bad;
}

__global__ void __launch_bounds__(kOnceThreads, 1)
log2_factors_once_kernel(const __half* __restrict__ x, long long count, Control* __restrict__ ctl, uint8_t* __restrict__ factors,
                         uint32_t* __restrict__ max_bits_out) {
    __shared__ uint32_t notes[kOnceNotes];
    __shared__ unsigned int noted, note_rate, warp_max[kOnceThreads / 32];
    // per warp: from which of its batches on its factors stood for which B_1 (a new entry where its maximum changed)
    __shared__ unsigned short covers[kOnceThreads / 32][kOnceChanges];
    __shared__ uint32_t from_batch[kOnceThreads / 32][kOnceChanges];
    cg::grid_group grid = cg::this_grid();
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const long long nvec = count / 8, stride = (long long)gridDim.x * kOnceThreads, at = (long long)blockIdx.x * kOnceThreads + threadIdx.x;
    const uint4* const xv = reinterpret_cast<const uint4*>(x);
    uint2* const out = reinterpret_cast<uint2*>(factors);
    volatile unsigned int* const running = &ctl->absmax_bits;
    __half2 m2 = __float2half2_rn(0.0f);                 // NaN operands are dropped
    auto largest = [&](const uint4& d) {
        const uint32_t w[4] = {d.x & 0x7FFF7FFFu, d.y & 0x7FFF7FFFu, d.z & 0x7FFF7FFFu, d.w & 0x7FFF7FFFu};
#pragma unroll
        for (int t = 0; t < 4; ++t) m2 = __hmax2(m2, *reinterpret_cast<const __half2*>(&w[t]));
    };
    auto load = [&](uint4 (&d)[kLog2InFlight], const uint4* src, bool whole) {
#pragma unroll
        for (int k = 0; k < kLog2InFlight; ++k) {
            d[k] = make_uint4(0u, 0u, 0u, 0u);
            if (whole || src + k * stride < xv + nvec) d[k] = __ldg(src + k * stride);
        }
    };
    // of this thread's values so far; Inf counts as the largest finite value
    auto max_bits = [&] {
        const unsigned int b = max((unsigned int)__half_as_ushort(__low2half(m2)), (unsigned int)__half_as_ushort(__high2half(m2)));
        return min(b, 0x7BFFu);
    };
    // a first maximum: from the first batches of as many CTAs as the control block has words for, and from vectors spread over all of x
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->status = 0;
        *running = 0u;
    }
    // of each warp; the vectors of all but its last one are all there
    const uint32_t batches = (uint32_t)((nvec + kLog2InFlight * stride - 1) / (kLog2InFlight * stride));
    if (threadIdx.x == 0) {
        noted = 0u;
        note_rate = 2 * kOnceNotes / batches;            // twice the notes that would fit at an even rate, per batch
    }
    const unsigned int words = min(gridDim.x, (unsigned int)Control::kRangeWords);
    if (blockIdx.x < words) {
        // (a warp's side by side; they also tell how many vectors have values in the range of the factors below 1)
        const uint4 probe = __ldg(xv + (long long)(blockIdx.x * (kOnceThreads / 32) + warp) * (nvec / (words * (kOnceThreads / 32))) + lane);
#pragma unroll
        for (int k = 0; k < kLog2InFlight; ++k)
            if (at + k * stride < nvec) largest(__ldg(xv + at + k * stride));
        largest(probe);
        const unsigned int b = __reduce_max_sync(0xFFFFFFFFu, max_bits());
        if (lane == 0) warp_max[warp] = b;
        uint32_t near, least = 0u;
        bool negative = false;
        (void)log2_factors8<true>(probe, (kBoundOfOne + 1023u) * 0x00010001u, near, least, negative);
        const unsigned int hits = (unsigned int)__syncthreads_count(near != 0u);
        if (threadIdx.x < 32) {
            const unsigned int c = __reduce_max_sync(0xFFFFFFFFu, lane < kOnceThreads / 32 ? warp_max[lane] : 0u);
            if (lane == 0) ctl->range[blockIdx.x] = c | (hits << 16);
        }
    }
    grid.sync();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned int word = lane < (int)words ? ((volatile unsigned int*)ctl->range)[lane] : 0u;
    unsigned int known = __reduce_max_sync(0xFFFFFFFFu, word & 0xFFFFu), used = ~0u;
    uint32_t cap = 0u, edge = 0u;                        // edge: remainders from 1024 - lead on reach bit 15 when it is added
    unsigned int bound = 0u;
    int changes = 0;
    bool bad = false, all_again = false;
    auto take_bound = [&](uint32_t batch) {
        used = known;
        bound = log2_first_bound(used);
        cap = (bound + 1023u) * 0x00010001u;
        // a softmax output is 1 at most
        const unsigned int lead = used <= 0x3C00u ? min(kBoundOfOne - bound, kLead) : 64u;
        edge = (0x8000u - 1024u + lead) * 0x00010001u;
        // (with no place left the last entry stands for fewer batches than it could)
        const int place = min(changes, kOnceChanges - 1);
        if (lane == 0) {
            covers[warp][place] = (unsigned short)(bound + lead);
            from_batch[warp][place] = batch;
        }
        changes = place + 1;
    };
    take_bound(0u);
    const long long hits = __reduce_add_sync(0xFFFFFFFFu, word >> 16), to_one = (long long)kBoundOfOne - bound;
    // of the vectors in that range to_one / 1024 are noted, remainders being as good as even; half the room for notes is to spare
    const bool twice = bound == 0u || to_one < 0 || to_one > kLead || hits * to_one * kOnceShare > (long long)words * kOnceThreads * 1024 ||
                       hits * to_one * nvec > (long long)words * kOnceThreads * 1024 * (kOnceNotes / 2) * gridDim.x;
    const uint4* p = xv + at;
    uint2* dst = out + at;
    if (twice) {
        all_again = true;
        uint64_t pass;
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pass));
        const long long keep = kOnceKeep / (long long)(kLog2InFlight * stride * sizeof(uint4));
        uint32_t batch = 0;
        for (; batch + 1 + keep < batches; ++batch, p += kLog2InFlight * stride) {
            uint4 d[kLog2InFlight];
#pragma unroll
            for (int k = 0; k < kLog2InFlight; ++k)
                asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                             : "=r"(d[k].x), "=r"(d[k].y), "=r"(d[k].z), "=r"(d[k].w) : "l"(p + k * stride), "l"(pass));
#pragma unroll
            for (int k = 0; k < kLog2InFlight; ++k) largest(d[k]);
        }
        for (; batch < batches; ++batch, p += kLog2InFlight * stride) {
            uint4 d[kLog2InFlight];
            load(d, p, batch + 1 < batches);
#pragma unroll
            for (int k = 0; k < kLog2InFlight; ++k) largest(d[k]);
        }
    }
    for (uint32_t batch = twice ? batches : 0; batch < batches; ++batch, p += kLog2InFlight * stride, dst += kLog2InFlight * stride) {
        uint4 d[kLog2InFlight];
        const bool whole = batch + 1 < batches;
        load(d, p, whole);
        // for the next batch, one lane's for all: others write it meanwhile, and the warp's bound and notes have to agree
        const unsigned int next = __shfl_sync(0xFFFFFFFFu, *running, 0);
        if (known != used) take_bound(batch);
        if (all_again) {
#pragma unroll
            for (int k = 0; k < kLog2InFlight; ++k) largest(d[k]);
        } else {
            uint32_t least = cap;
#pragma unroll
            for (int k = 0; k < kLog2InFlight; ++k) {
                uint32_t near;
                const uint2 f = log2_factors8<true>(d[k], cap, near, least, bad);
                if (whole || p + k * stride < xv + nvec) {
                    __stcs(dst + k * stride, f);
                    if ((near + edge) & 0x80008000u) {
                        const unsigned int n = atomicAdd(&noted, 1u);
                        if (n < (unsigned int)kOnceNotes) notes[n] = (uint32_t)(p - xv + k * stride);
                        all_again |= n >= min((unsigned int)kOnceNotes, note_rate * (batch + 1));
                    }
                }
            }
            // (where cap lies above infinity a NaN may be what comes nearest to it: the values themselves then)
            if (__vminu2(least, 0x00010001u) != 0x00010001u || cap > 0x7C007C00u) {
#pragma unroll
                for (int k = 0; k < kLog2InFlight; ++k) largest(d[k]);
            } else {
                const uint32_t most = cap - least;
                m2 = __hmax2(m2, *reinterpret_cast<const __half2*>(&most));
            }
        }
        all_again = __any_sync(0xFFFFFFFFu, all_again);
        known = max(known, next);
        const unsigned int own = __reduce_max_sync(0xFFFFFFFFu, max_bits());
        if (own > known) {
            if (lane == 0) atomicMax(&ctl->absmax_bits, own);
            known = own;
        }
    }
    // the ragged tail's maximum
    for (long long i = nvec * 8 + at; i < count; i += stride) {
        const unsigned int hb = __half_as_ushort(x[i]) & 0x7FFFu;
        if (hb <= 0x7C00u) known = max(known, min(hb, 0x7BFFu));
    }
    __syncwarp();
    {
        const unsigned int b = __reduce_max_sync(0xFFFFFFFFu, max(known, max_bits()));
        if (lane == 0) warp_max[warp] = b;
        __syncthreads();
        if (threadIdx.x < 32) {
            const unsigned int c = __reduce_max_sync(0xFFFFFFFFu, lane < kOnceThreads / 32 ? warp_max[lane] : 0u);
            if (lane == 0 && c > *running) atomicMax(&ctl->absmax_bits, c);
        }
    }
    grid.sync();
    const unsigned int mb_bits = *running, final_bound = log2_first_bound(mb_bits);
    if (blockIdx.x == 0 && threadIdx.x == 0 && max_bits_out) *max_bits_out = mb_bits;
    const uint32_t final_cap = (final_bound + 1023u) * 0x00010001u;
    int mb = 1024, eb = 0, t_up = 0, t_down = 0;
    if (mb_bits) half_parts(mb_bits, mb, eb);
    log2_thresholds(mb, t_up, t_down);
    uint32_t near, least = 0u;
    // the batches up to the first change whose factors stand for the true bound
    const bool again = __any_sync(0xFFFFFFFFu, all_again || final_bound == 0u);
    long long redo = again ? batches : 0;
    if (!again && changes > 0) {
        int c = 0;
        while (c < changes && covers[warp][c] < final_bound) ++c;
        redo = c == changes ? batches : from_batch[warp][c];
    }
    if (final_bound) {
        const long long end = min(nvec, redo * kLog2InFlight * stride + at);
        if (end > at) bad |= log2_write_again(xv, out, at + (end - 1 - at) / stride * stride, stride, final_cap);
    } else {
        bad |= log2_write_by_bounds(xv, out, at, nvec, stride, mb_bits, mb, eb, t_up, t_down);
    }
    // (another warp's vectors may be among these, written by it above as well: the same factors)
    if (final_bound)
        for (unsigned int n = threadIdx.x; n < min(noted, (unsigned int)kOnceNotes); n += kOnceThreads)
            out[notes[n]] = log2_factors8<false>(__ldg(xv + notes[n]), final_cap, near, least, bad);
    for (long long i = nvec * 8 + at; i < count; i += stride)
        factors[i] = log2_factor(__half_as_ushort(x[i]), mb_bits, eb, t_up, t_down, bad);
    if (bad) atomicCAS(&ctl->status, 0u, 11u);
}

__global__ void __launch_bounds__(256, kLog2Ctas)
log2_codes_kernel(const __half* __restrict__ x, long long count, int bits, int words, Control* __restrict__ ctl,
                  int8_t* __restrict__ codes, uint32_t* __restrict__ max_bits_out, int as_factors) {
    // as_factors (4-bit codes of a non-negative input): instead of the code c the byte 2^(kmax - k) = 128 >> (c - 1)
    // is written (0 for a zero), the form the tensor-core product takes; a negative value is reported (status 11)
    asm volatile("griddepcontrol.wait;" ::: "memory");      // launched while the maximum's kernel drains
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool bad = false;
    const unsigned int mb_bits = met_range(ctl, words);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->absmax_bits = mb_bits;
        if (max_bits_out) *max_bits_out = mb_bits;
    }
    const int kmax = (1 << (bits - 1)) - 1;
    int mb = 1024, eb = 0, t_up = 0, t_down = 0;
    if (mb_bits) half_parts(mb_bits, mb, eb);
    log2_thresholds(mb, t_up, t_down);
    const bool vec = (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && (reinterpret_cast<uintptr_t>(codes) & 7u) == 0;
    const long long nvec = vec ? count / 8 : 0;
    const uint4* xv = reinterpret_cast<const uint4*>(x);
    if (bits == 4 && mb_bits != 0) {
        const Log2Fast fast = log2_fast_bounds(mb, eb, t_up, t_down);
        const unsigned int b1 = __half_as_ushort(__low2half(fast.bound[0]));
        if (as_factors && (unsigned int)__half_as_ushort(__low2half(fast.bound[6])) >= 0x0400u) {
            // x is walked backwards, since its end is what the maximum's kernel has left in the L2 (57 MB of 268 MB hit there), with
            // stores marked as not used again (loads marked so cost 10 us). Both kernels on 32 x 2048 x 2048: 145.6 -> 107.3 us (45 us at
            // 5.9 TB/s and 66 us at 4.8 TB/s of HBM traffic, reads and writes mixed); on 4 heads, 33 MB, 28.8 -> 19.2 us.
            const uint32_t cap = (b1 + 1023u) * 0x00010001u;
            const long long stride = (long long)gridDim.x * blockDim.x;
            auto factors = [&](const uint4& d) {
                uint32_t near, least = 0u;
                return log2_factors8<false>(d, cap, near, least, bad);
            };
            long long v = nvec - 1 - ((long long)blockIdx.x * blockDim.x + threadIdx.x);       // this thread's vector, downwards
            const uint4* src = xv + v;
            uint2* dst = reinterpret_cast<uint2*>(codes) + v;
            for (; v >= (kLog2InFlight - 1) * stride; v -= kLog2InFlight * stride, src -= kLog2InFlight * stride, dst -= kLog2InFlight * stride) {
                uint4 d[kLog2InFlight];
#pragma unroll
                for (int k = 0; k < kLog2InFlight; ++k) d[k] = __ldg(src - k * stride);
#pragma unroll
                for (int k = 0; k < kLog2InFlight; ++k) __stcs(dst - k * stride, factors(d[k]));
            }
            for (; v >= 0; v -= stride, src -= stride, dst -= stride) __stcs(dst, factors(__ldg(src)));
        } else
#pragma unroll 4
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += (long long)gridDim.x * blockDim.x) {
            const uint4 d = __ldg(xv + i);
            const uint32_t w[4] = {d.x, d.y, d.z, d.w};
            uint32_t m[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const __half2 x2 = *reinterpret_cast<const __half2*>(&w[t]);
                __half2 r;
                if (as_factors) {
                    r = log2_fast2<true>(x2, fast);
                    // a negative input has no factor: recorded, its byte is 0
                    const __half2 neg = __hlt2(x2, __float2half2_rn(0.0f));
                    bad |= (*reinterpret_cast<const uint32_t*>(&neg) != 0u);
                    r = __hfma2(neg, __hneg2(r), r);                                    // r * (1 - neg)
                    r = __hadd2(r, __float2half2_rn(1024.0f));                           // the integer sits in the low bits
                } else {
                    r = log2_fast2<false>(x2, fast);
                    uint32_t rb = *reinterpret_cast<uint32_t*>(&r) | (w[t] & 0x80008000u);   // Sign(x) * (k + 1)
                    r = __hadd2(*reinterpret_cast<__half2*>(&rb), __float2half2_rn(1536.0f));   // two's complement in the low byte
                }
                m[t] = *reinterpret_cast<uint32_t*>(&r);
            }
            *reinterpret_cast<uint2*>(codes + 8 * i) = make_uint2(__byte_perm(m[0], m[1], 0x6420), __byte_perm(m[2], m[3], 0x6420));
        }
    } else
#pragma unroll 4
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += (long long)gridDim.x * blockDim.x) {
        const uint4 d = __ldg(xv + i);
        const uint32_t w[4] = {d.x, d.y, d.z, d.w};
        uint32_t out[2] = {0u, 0u};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t c0 = (uint32_t)log2_code(w[t] & 0xFFFFu, mb_bits, eb, t_up, t_down, kmax) & 0xFFu;
            const uint32_t c1 = (uint32_t)log2_code(w[t] >> 16, mb_bits, eb, t_up, t_down, kmax) & 0xFFu;
            out[t >> 1] |= (c0 | (c1 << 8)) << (16 * (t & 1));
        }
        if (as_factors) { out[0] = log2_factors4(out[0], bad); out[1] = log2_factors4(out[1], bad); }
        *reinterpret_cast<uint2*>(codes + 8 * i) = make_uint2(out[0], out[1]);
    }
    for (long long i = nvec * 8 + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
        const int c = log2_code(__half_as_ushort(x[i]), mb_bits, eb, t_up, t_down, kmax);
        bad |= as_factors && c < 0;
        codes[i] = as_factors ? (int8_t)(uint8_t)(c > 0 ? (128u >> (c - 1)) : 0u) : (int8_t)c;
    }
    if (bad) atomicCAS(&ctl->status, 0u, 11u);
}

// ---- attention x value on the codes -----------------------------------------------------------
// A CTA of 256 threads takes `rows` consecutive query rows of one head and all D value columns; a
// thread owns one row and four consecutive columns (one 4-byte load of value codes per j) and adds
// each value code shifted left by kmax - k_j, negated for negative probabilities, skipped for zeros.
__global__ void __launch_bounds__(256)
attn_v_log2_kernel(const int8_t* __restrict__ pcodes, const uint32_t* __restrict__ max_bits,
                   const int8_t* __restrict__ vq, const int32_t* __restrict__ e_v, int M, int J, int D, int bits,
                   int rows, __half* __restrict__ y, int32_t* __restrict__ acc_dump) {
    const int quads = D / 4;
    const int r = threadIdx.x / quads, dq = threadIdx.x % quads;
    const int h = blockIdx.y;
    const int m = blockIdx.x * rows + r;
    if (r >= rows || m >= M) return;
    const int kmax = (1 << (bits - 1)) - 1;
    const int8_t* prow = pcodes + ((size_t)h * M + m) * J;
    const char4* vcol = reinterpret_cast<const char4*>(vq + (size_t)h * J * D) + dq;
    int a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll 4
    for (int j = 0; j < J; ++j) {
        const int c = prow[j];
        if (c == 0) continue;
        const char4 v = __ldg(vcol + (size_t)j * quads);
        const int sh = kmax + 1 - abs(c);
        const int sg = c > 0 ? 1 : -1;
        a0 += (sg * (int)v.x) << sh;
        a1 += (sg * (int)v.y) << sh;
        a2 += (sg * (int)v.z) << sh;
        a3 += (sg * (int)v.w) << sh;
    }
    const float pmax = __half2float(__ushort_as_half((unsigned short)(*max_bits & 0xFFFFu)));
    const float scale = pmax * __int_as_float((127 + *e_v - kmax) << 23);
    const size_t o = ((size_t)h * M + m) * D + 4 * dq;
    y[o + 0] = __float2half_rn(scale * (float)a0);
    y[o + 1] = __float2half_rn(scale * (float)a1);
    y[o + 2] = __float2half_rn(scale * (float)a2);
    y[o + 3] = __float2half_rn(scale * (float)a3);
    if (acc_dump) { acc_dump[o] = a0; acc_dump[o + 1] = a1; acc_dump[o + 2] = a2; acc_dump[o + 3] = a3; }
}

// ---- the same product on the tensor cores (non-negative P, i.e. a softmax output) --------------
// With P >= 0 the factor 2^(kmax - k) is an unsigned byte (1..128), so the product is a plain
// u8 x s8 -> s32 contraction over the key index j: acc[m][d] = sum_j w[m][j] * v[d][j], with both
// operands stored j-major. tcgen05.mma kind::i8 reads both from shared memory (128-byte swizzle,
// staged by TMA); the accumulator [128 query rows x D] lives in tensor memory.

// The first kernel of a call (launched while the kernel ahead drains) sets the control block up.
__device__ __forceinline__ void begin_attn_call(Control* ctl) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) ctl->status = 0;
}

// [H][J][D] int8 -> [H][D][J] int8 through a 32 x 32 shared-memory tile.
__global__ void __launch_bounds__(256)
transpose_i8_kernel(const int8_t* __restrict__ in, int J, int D, int8_t* __restrict__ out, Control* __restrict__ ctl) {
    begin_attn_call(ctl);
    __shared__ int8_t tile[32][33];
    const int h = blockIdx.z, j0 = blockIdx.x * 32, d0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;          // 32 x 8
    for (int r = ty; r < 32; r += 8) {
        const int j = j0 + r, d = d0 + tx;
        tile[r][tx] = (j < J && d < D) ? in[((size_t)h * J + j) * D + d] : (int8_t)0;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int d = d0 + r, j = j0 + tx;
        if (d < D && j < J) out[((size_t)h * D + d) * J + j] = tile[tx][r];
    }
}

// The same through a 64 x 64 tile with 4-byte accesses on both sides (D and J multiples of 4, 4-byte aligned
// buffers): a warp reads and writes 64-byte row pieces as words instead of 32 single bytes.
__global__ void __launch_bounds__(256)
transpose_i8_words_kernel(const int8_t* __restrict__ in, int J, int D, int8_t* __restrict__ out, Control* __restrict__ ctl) {
    begin_attn_call(ctl);
    __shared__ __align__(4) int8_t tile[64][68];                      // [j][d], rows padded to 68 bytes
    const int h = blockIdx.z, j0 = blockIdx.x * 64, d0 = blockIdx.y * 64;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int idx = (int)threadIdx.x + 256 * k, r = idx >> 4, c = 4 * (idx & 15);
        const int j = j0 + r, d = d0 + c;
        uint32_t w = 0u;
        if (j < J && d < D) w = *reinterpret_cast<const uint32_t*>(in + ((size_t)h * J + j) * D + d);
        *reinterpret_cast<uint32_t*>(&tile[r][c]) = w;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int idx = (int)threadIdx.x + 256 * k, r = idx >> 4, c = 4 * (idx & 15);      // output row d0 + r, columns j0 + c..
        const int d = d0 + r, j = j0 + c;
        if (d < D && j < J) {
            const uint32_t w = (uint32_t)(uint8_t)tile[c][r] | ((uint32_t)(uint8_t)tile[c + 1][r] << 8) |
                               ((uint32_t)(uint8_t)tile[c + 2][r] << 16) | ((uint32_t)(uint8_t)tile[c + 3][r] << 24);
            *reinterpret_cast<uint32_t*>(out + ((size_t)h * D + d) * J + j) = w;
        }
    }
}

constexpr int kTcStages = 4;
// warp 0: TMA, warp 1: MMA + TMEM owner, then EW epilogue warps (4, or 8: two per quarter of the tensor-memory lanes,
// each taking half of the columns, for products with one k step per tile, where the epilogue sets the pace)
constexpr int kConvWarps = 8;                        // warps that turn codes into byte factors (CONVERT)
constexpr int tc_threads(int ew, bool convert = false) { return (2 + ew + (convert ? kConvWarps : 0)) * 32; }
constexpr unsigned long long kTcWaitCycles = 4000000000ull;

// One thread of a converged warp: the compiler then knows that a copy or an MMA has one set of operands (see elect_one in aq_tc.cuh).
__device__ __forceinline__ bool a_elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ uint32_t a_smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool a_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(a_smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait; false when the limit ran out or another role gave up.
__device__ __forceinline__ bool a_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag) {
    if (a_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    uint32_t spins = 0;
    while (!a_try_wait(bar, parity)) {
        if ((++spins & 0x3FFu) == 0) {
            if (*abort_flag) return false;
            if ((unsigned long long)(clock64() - t0) > kTcWaitCycles) { *abort_flag = 12u; return false; }
        }
    }
    return true;
}
// K-major tile with 128-byte rows written by TMA with the 128-byte swizzle (see aq_gemm_tensor.cu).
__device__ __forceinline__ uint64_t a_desc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

template <int DN, int RT, int EW>
struct AttnSmem {
    alignas(1024) uint8_t a[kTcStages][RT * 128 * 128];   // weights tile: RT x 128 query rows x 128 j
    alignas(1024) uint8_t b[kTcStages][DN * 128];    // value tile: DN columns x 128 j
    // Output staging: each epilogue warp owns two boxes of 32 rows x 64 halves (128-byte rows, written
    // with the 128-byte swizzle of the store's tensor map), for alternate 64-column chunks.
    alignas(1024) uint8_t ystage[EW][2][32 * 128];
    alignas(8) uint64_t full[kTcStages];
    uint64_t empty[kTcStages];
    uint64_t conv[kTcStages];                        // CONVERT: the A tile of the stage holds byte factors -> MMA
    uint64_t acc_full[2];                            // MMA -> epilogue, one per accumulator stage
    uint64_t acc_empty[2];                           // epilogue (4 warps) -> MMA
    uint32_t tmem_base;
    volatile uint32_t abort_flag;
};

// Batched int8 contraction y[h][m][n] = scale * sum_k A[h*M + m][k] * B[h*NB + n][k] (both operands
// k-major). A work item is (128 rows of A, head) and all tiles of DN rows of B for those rows, or one of `parts` runs
// of those tiles (see attn_parts). The grid is persistent: CTA c takes the items c, c + gridDim.x, ..., and the ring of operand stages and the two
// accumulator stages in tensor memory run on across items, so the producer fetches the next item's tiles
// while the epilogue of the last tile of this one still writes (a CTA's 16 k steps of one item alone were
// mostly fill and drain). With RT = 2 an item is 256 rows of A, two accumulators of 128 rows that share
// every tile of B: what limits this kernel is the L2 -> SM path, and the B tile is then fetched once for
// twice the rows. A is unsigned or signed bytes, B signed. CONVERT: A arrives as 4-bit log2 codes (c = k + 1,
// 0 for a zero) and kConvWarps more warps turn every landed A tile into byte factors 128 >> k in place before the
// MMA reads it, so that attention x value needs no conversion pass over the probabilities in memory.
// scale = (max_bits ? the half in its low 16 bits : 1) * 2^(*e1 + (e2 ? *e2 : 0) + e_off).
// Used for attention x value (A = byte factors of the log2 codes, B = transposed value codes, k = key
// index) and for the query x key product (A, B = int8 codes, k = head dimension).
template <int DN, bool A_SIGNED, int RT = 1, int EW = 4, bool CONVERT = false>
__global__ void __launch_bounds__(tc_threads(EW, CONVERT), 1)
attn_v_tc_kernel(const __grid_constant__ CUtensorMap a_map, const __grid_constant__ CUtensorMap b_map,
                 const __grid_constant__ CUtensorMap y_map, const uint32_t* __restrict__ max_bits, const int32_t* __restrict__ e1, const int32_t* __restrict__ e2,
                 int e_off, int H, int M, int J /* length of k */, int NB, int parts, int clear_status, __half* __restrict__ y,
                 Control* __restrict__ ctl) {
    extern __shared__ uint8_t attn_smem_raw[];
    using Smem = AttnSmem<DN, RT, EW>;
    static_assert(EW == 4 || (EW == 8 && DN % 64 == 0), "epilogue warps: one or two per lane quarter");
    constexpr int kColsPerWarp = DN / (EW / 4);                          // columns an epilogue warp drains
    static_assert(2 * RT * DN <= 512, "two accumulator stages of RT x DN columns in tensor memory");
    constexpr int kRows = RT * 128;                                       // rows of A per item
    Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(attn_smem_raw) + 1023) & ~(uintptr_t)1023);
    // Elected issuing threads pay everywhere but where codes are converted for items of 128 rows: there the paced issue of
    // `lane == 0` leaves the converting warps more of the shared-memory pipe (40 heads, 1000 x 1008 32.5 -> 31.1 us, 12 heads,
    // 2000 x 2000 38.4 -> 35.8; items of 256 rows the other way round, 40 heads, 2048 x 1008 46.1 elected, 47.1 paced).
    constexpr bool kElect = !CONVERT || RT > 1;
    const int warp = kElect ? __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0) : (int)threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int MT = (M + kRows - 1) / kRows;                               // row tiles per head
    const int items = MT * H * parts;                                     // work items, see below
    const int JB = (J + 127) / 128;
    const int NT = (NB + DN - 1) / DN;                                    // tiles of B rows
    const int tiles_per_part = (NT + parts - 1) / parts;
    // item w: head, first row, and the tiles [nt0, nt1) of B rows
    auto item_at = [&](int w, int& h, int& m0, int& nt0, int& nt1) {
        const int rows = parts > 1 ? w / parts : w;
        nt0 = (w - rows * parts) * tiles_per_part;
        nt1 = min(NT, nt0 + tiles_per_part);
        h = rows / MT;
        m0 = (rows - h * MT) * kRows;
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < kTcStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(a_smem_u32(&sm.full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(a_smem_u32(&sm.empty[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a_smem_u32(&sm.conv[s])), "r"(kConvWarps) : "memory");
        }
        for (int a = 0; a < 2; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(a_smem_u32(&sm.acc_full[a])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a_smem_u32(&sm.acc_empty[a])), "r"(EW) : "memory");
        }
        sm.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(a_smem_u32(&sm.tmem_base)), "r"((uint32_t)(2 * RT * DN)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = sm.tmem_base;
    volatile uint32_t* abort_flag = &sm.abort_flag;
    // Set up while the kernel ahead drains; nothing is read or written before it has completed. The launch behind this one is not
    // allowed early: its waiting CTAs on the SMs cost this kernel more than the launch gap (scores, byte factors and attention x
    // value of 32 heads, 2048 x 2048: 216.1 us with plain launches, 217.5 with early ones behind this kernel, 198.7 as it is).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (clear_status && blockIdx.x == 0 && threadIdx.x == 0) ctl->status = 0;

    if (warp == 0) {
        if (kElect ? a_elect_one() : lane == 0) {
            int it = 0;                                                   // stages filled so far, over all items
            bool ok = true;
            for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
              int h, m0, nt0, nt1;
              item_at(w, h, m0, nt0, nt1);
              for (int nt = nt0; nt < nt1 && ok; ++nt)
              for (int jb = 0; jb < JB; ++jb, ++it) {
                const int n0 = nt * DN;
                const int s = it % kTcStages;
                if (!a_wait(&sm.empty[s], ((it / kTcStages) & 1) ^ 1, abort_flag)) { ok = false; break; }
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                             ::"r"(a_smem_u32(&sm.full[s])), "r"((uint32_t)((kRows + DN) * 128)) : "memory");
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                    ::"r"(a_smem_u32(sm.a[s])), "l"(&a_map), "r"(jb * 128), "r"(h * M + m0), "r"(a_smem_u32(&sm.full[s]))
                    : "memory");
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                    ::"r"(a_smem_u32(sm.b[s])), "l"(&b_map), "r"(jb * 128), "r"(h * NB + n0), "r"(a_smem_u32(&sm.full[s]))
                    : "memory");
              }
            }
        }
    } else if (warp == 1) {
        if (kElect ? a_elect_one() : lane == 0) {
            // D = s32 (2 at bits 4-5), A unsigned 8-bit (0 at bits 7-9), B signed 8-bit (1 at bits 10-12),
            // both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28
            constexpr uint32_t idesc = (2u << 4) | ((A_SIGNED ? 1u : 0u) << 7) | (1u << 10) | ((uint32_t)(DN >> 3) << 17) |
                                       ((uint32_t)(128 >> 4) << 24);
            bool ok = true;
            int it = 0, tc = 0;                                           // stages and tiles consumed so far, over all items
            for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
            int h, m0, nt0, nt1;
            item_at(w, h, m0, nt0, nt1);
            for (int nt = nt0; nt < nt1 && ok; ++nt, ++tc) {
              const int a = tc & 1;
              ok = a_wait(&sm.acc_empty[a], ((tc >> 1) & 1) ^ 1, abort_flag);      // the epilogue has drained this stage
              if (!ok) break;
              for (int jb = 0; jb < JB && ok; ++jb, ++it) {
                const int s = it % kTcStages;
                ok = a_wait(CONVERT ? &sm.conv[s] : &sm.full[s], (it / kTcStages) & 1, abort_flag);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t adesc = a_desc_sw128(a_smem_u32(sm.a[s]));
                const uint64_t bdesc = a_desc_sw128(a_smem_u32(sm.b[s]));
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    // the r-th 128 rows of the A tile start 16 KB (1024 in descriptor units of 16 bytes) further on
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const uint32_t accumulate = (jb == 0 && t == 0) ? 0u : 1u;
                        asm volatile(
                            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                            ::"r"(tmem + (uint32_t)((a * RT + r) * DN)), "l"(adesc + (uint64_t)(1024 * r + 2 * t)),
                              "l"(bdesc + (uint64_t)(2 * t)), "r"(idesc), "r"(accumulate)
                            : "memory");
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(a_smem_u32(&sm.empty[s])) : "memory");
              }
              if (ok)
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(a_smem_u32(&sm.acc_full[a])) : "memory");
            }
            }
        }
    } else if (CONVERT && warp >= 2 + EW) {
        // ---- codes -> byte factors, in place, on every A tile that has landed (the map is bytewise, so the
        // tile's swizzle does not matter). Per 32-bit word: a byte permute looks the factors of codes 1..7 up
        // by the codes' low three bits, code 8 (k = 7) is added as 1, codes above 8 and negative codes give 0,
        // and a negative code is recorded (status 11) as the conversion pass does.
        const int cw = warp - (2 + EW);                                       // 0..kConvWarps-1
        bool bad = false;
        int it = 0;
        bool ok = true;
        for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
            int h, m0, nt0, nt1;
            item_at(w, h, m0, nt0, nt1);
            for (int i = 0; i < (nt1 - nt0) * JB && ok; ++i, ++it) {
                const int s = it % kTcStages;
                ok = __all_sync(0xFFFFFFFFu, a_wait(&sm.full[s], (it / kTcStages) & 1, abort_flag) ? 1 : 0) != 0;
                if (!ok) break;
                uint4* tile = reinterpret_cast<uint4*>(sm.a[s]);
#pragma unroll 4
                for (int v = cw * 32 + lane; v < kRows * 128 / 16; v += kConvWarps * 32) {
                    uint4 c = tile[v];
                    uint32_t* cwds = reinterpret_cast<uint32_t*>(&c);
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const uint32_t x = cwds[t];
                        const uint32_t neg = x & 0x80808080u;
                        const uint32_t x7 = x & 0x7F7F7F7Fu;
                        const uint32_t big = (x7 + 0x77777777u) & 0x80808080u;          // bytes from 9 up
                        const uint32_t low = x & 0x07070707u;
                        const uint32_t sel = __byte_perm(low | (low >> 4), 0u, 0x4420);   // four 3-bit indices as nibbles
                        uint32_t r = __byte_perm(0x20408000u, 0x02040810u, sel);          // index 0..7 -> 0, 128, 64, ..., 2
                        r |= (x7 >> 3) & 0x01010101u;                                     // code 8 -> 1 (9..15 are cleared below)
                        const uint32_t kill = ((neg | big) >> 7) * 0xFFu;
                        cwds[t] = r & ~kill;
                        bad |= neg != 0u;
                    }
                    tile[v] = c;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes before the tensor core's reads
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a_smem_u32(&sm.conv[s])) : "memory");
            }
        }
        if (bad) atomicCAS(&ctl->status, 0u, 11u);
    } else {
        const int quarter = warp & 3;                                     // TMEM lanes this warp may read
        const float pmax = max_bits ? __half2float(__ushort_as_half((unsigned short)(*max_bits & 0xFFFFu))) : 1.0f;
        const float scale = pmax * __int_as_float((127 + *e1 + (e2 ? *e2 : 0) + e_off) << 23);
        int tc = 0;                                                       // tiles drained so far, over all items
        int next_box = 0;
        bool alive = true;
        for (int w = blockIdx.x; w < items && alive; w += gridDim.x) {
          int h, m0_item, nt0, nt1;
          item_at(w, h, m0_item, nt0, nt1);
          for (int nt = nt0; nt < nt1; ++nt, ++tc) {
            const int a = tc & 1, n0 = nt * DN;
            if (!(__all_sync(0xFFFFFFFFu, a_wait(&sm.acc_full[a], (tc >> 1) & 1, abort_flag) ? 1 : 0) != 0)) { alive = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int ew = warp - 2;
#pragma unroll 1
            for (int r = 0; r < RT; ++r) {
            const int m0 = m0_item + r * 128, m = m0 + quarter * 32 + lane;          // this accumulator's 128 rows
#pragma unroll 1
            for (int c0 = ((warp - 2) >> 2) * kColsPerWarp; c0 < (((warp - 2) >> 2) + 1) * kColsPerWarp; c0 += 32) {
                uint32_t v[32];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                    "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                    "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                      "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                      "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                    : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((a * RT + r) * DN + c0))
                    : "memory");
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                // 32 columns of this thread's row -> 64 bytes of its 128-byte staging row; 16-byte chunk j of
                // row r sits at chunk position j ^ (r & 7), as the store's tensor map expects
                const int row0 = m0 + quarter * 32;
                if (row0 + 32 > M) {
                    // a box of 32 rows would run into the next head's rows: this warp stores its rows itself
                    if (m < M) {
                        __half* yrow = y + ((size_t)h * M + m) * NB + n0;
#pragma unroll
                        for (int q8 = 0; q8 < 4; ++q8) {
                            if (n0 + c0 + 8 * q8 >= NB) break;               // NB is a multiple of 8
                            __half2 o[4];
#pragma unroll
                            for (int t = 0; t < 4; ++t)
                                o[t] = __floats2half2_rn(scale * (float)(int)v[8 * q8 + 2 * t], scale * (float)(int)v[8 * q8 + 2 * t + 1]);
                            *reinterpret_cast<uint4*>(yrow + c0 + 8 * q8) = *reinterpret_cast<uint4*>(o);
                        }
                    }
                    continue;
                }
                // (a warp that drains one box per tile takes its two in turn, from store to store)
                const int box = kColsPerWarp > 64 ? (c0 >> 6) & 1 : next_box, half_of_box = (c0 >> 5) & 1;
                uint8_t* srow = sm.ystage[ew][box] + lane * 128;
                if (half_of_box == 0) {
                    // the box is about to be rewritten: the store that used it last must have read it (with two
                    // boxes in rotation one younger store may still be pending)
                    if (lane == 0) {
                        asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    }
                    __syncwarp();
                }
#pragma unroll
                for (int q8 = 0; q8 < 4; ++q8) {
                    __half2 o[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        o[t] = __floats2half2_rn(scale * (float)(int)v[8 * q8 + 2 * t], scale * (float)(int)v[8 * q8 + 2 * t + 1]);
                    const int chunk = half_of_box * 4 + q8;
                    *reinterpret_cast<uint4*>(srow + ((chunk ^ (lane & 7)) << 4)) = *reinterpret_cast<uint4*>(o);
                }
                if (half_of_box == 1 || c0 + 32 >= DN) {   // (a warp's column range ends on a box boundary or at DN)
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    const int col = n0 + (c0 & ~63);
                    if (lane == 0 && col < NB) {
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                                     ::"l"(&y_map), "r"(col), "r"(h * M + row0), "r"(a_smem_u32(sm.ystage[ew][box])) : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                    if (col < NB) next_box ^= 1;
                }
            }
            }
            // this warp's part of the accumulator stage is in registers / written: hand the stage back
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a_smem_u32(&sm.acc_empty[a])) : "memory");
          }
        }
    }
    if (warp >= 2 && warp < 2 + EW && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // staging rows live until read
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (sm.abort_flag) {
        for (int i = 0; i < 64; ++i) __nanosleep(1000);                   // let copies in flight land
        if (threadIdx.x == 0) atomicCAS(&ctl->status, 0u, sm.abort_flag);
    }
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * RT * DN)) : "memory");
}

typedef CUresult (*AttnEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

template <int DN, bool A_SIGNED, int RT = 1, int EW = 4, bool CONVERT = false>
cudaError_t launch_attn_tc(const void* w, const int8_t* vt, const uint32_t* max_bits, const int32_t* e1, const int32_t* e2,
                           int e_off, int H, int M, int J, int NB, __half* y, Control* ctl, const DeviceInfo& dev,
                           cudaStream_t stream, bool first_of_call = false) {
    using Smem = AttnSmem<DN, RT, EW>;
    const size_t smem_bytes = sizeof(Smem) + 1024;
    static SmemOptIn opt_in;
    if (const cudaError_t e = opt_in.ensure(attn_v_tc_kernel<DN, A_SIGNED, RT, EW, CONVERT>, dev.device, smem_bytes); e != cudaSuccess)
        return e;
    CUtensorMap amap, bmap;
    const cuuint32_t estr[2] = {1u, 1u};
    const cuuint64_t strides[1] = {(cuuint64_t)J};
    const cuuint64_t adims[2] = {(cuuint64_t)J, (cuuint64_t)H * M};
    const cuuint32_t abox[2] = {128u, (cuuint32_t)(RT * 128)};
    const cuuint64_t bdims[2] = {(cuuint64_t)J, (cuuint64_t)H * NB};
    const cuuint32_t bbox[2] = {128u, (cuuint32_t)DN};
    AttnEncodeFn enc = reinterpret_cast<AttnEncodeFn>(dev.encode_tiled);
    if (enc(&amap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(w), adims, strides, abox, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    if (enc(&bmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t*>(vt), bdims, strides, bbox, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    // outputs: [H*M rows][NB] halves, stored in boxes of 64 columns x 32 rows with the 128-byte swizzle
    CUtensorMap ymap;
    const cuuint64_t ydims[2] = {(cuuint64_t)NB, (cuuint64_t)H * M};
    const cuuint64_t ystrides[1] = {(cuuint64_t)NB * 2};
    const cuuint32_t ybox[2] = {64u, 32u};
    if (enc(&ymap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, y, ydims, ystrides, ybox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    const long row_items = (long)((M + RT * 128 - 1) / (RT * 128)) * H;
    const int parts = attn_parts(row_items, (NB + DN - 1) / DN, dev.sm_count);
    const long items = row_items * parts;
    return launch_overlapped_smem(attn_v_tc_kernel<DN, A_SIGNED, RT, EW, CONVERT>, dim3((unsigned int)(items < dev.sm_count ? items : dev.sm_count)),
                             tc_threads(EW, CONVERT), stream, smem_bytes, amap, bmap, ymap, max_bits, e1, e2, e_off, H, M, J, NB, parts,
                             first_of_call ? 1 : 0, y, ctl);
}

}  // namespace

size_t attn_tc_scratch_bytes(int H, int M, int J, int D) {
    (void)M;
    return ((size_t)H * D * J + 255) / 256 * 256;
}

// scratch: the transposed value codes, H*D*J bytes.
// p_is_factors: pcodes already holds the byte factors (written by the log2 kernel); otherwise the product kernel
// converts the codes tile by tile in shared memory.
cudaError_t launch_attn_v_log2_tc(const int8_t* pcodes, const uint32_t* max_bits, const int8_t* vq, const int32_t* e_v,
                                  int H, int M, int J, int D, __half* y, Control* ctl, void* scratch,
                                  const DeviceInfo& dev, cudaStream_t stream, bool p_is_factors) {
    int8_t* vt = static_cast<int8_t*>(scratch);
    cudaError_t e = cudaSuccess;
    // codes or byte factors: the product kernel reads either
    const uint8_t* w = reinterpret_cast<const uint8_t*>(pcodes);
    if (J % 4 == 0 && D % 4 == 0 && (reinterpret_cast<uintptr_t>(vq) & 3u) == 0 && (reinterpret_cast<uintptr_t>(vt) & 3u) == 0)
        e = launch_overlapped(transpose_i8_words_kernel, dim3((J + 63) / 64, (D + 63) / 64, H), 256, stream, vq, J, D, vt, ctl);
    else
        e = launch_overlapped(transpose_i8_kernel, dim3((J + 31) / 32, (D + 31) / 32, H), 256, stream, vq, J, D, vt, ctl);
    if (e != cudaSuccess) return e;
    const bool wide_items = M % 256 == 0;       // items of 256 query rows share every value tile; whole items only
    if (p_is_factors)
        return D == 64 ? launch_attn_tc<64, false>(w, vt, max_bits, e_v, nullptr, -7, H, M, J, D, y, ctl, dev, stream)
               : wide_items ? launch_attn_tc<128, false, 2>(w, vt, max_bits, e_v, nullptr, -7, H, M, J, D, y, ctl, dev, stream)
                            : launch_attn_tc<128, false>(w, vt, max_bits, e_v, nullptr, -7, H, M, J, D, y, ctl, dev, stream);
    return D == 64 ? launch_attn_tc<64, false, 1, 4, true>(w, vt, max_bits, e_v, nullptr, -7, H, M, J, D, y, ctl, dev, stream)
           : wide_items ? launch_attn_tc<128, false, 2, 4, true>(w, vt, max_bits, e_v, nullptr, -7, H, M, J, D, y, ctl, dev, stream)
                        : launch_attn_tc<128, false, 1, 4, true>(w, vt, max_bits, e_v, nullptr, -7, H, M, J, D, y, ctl, dev, stream);
}

// Query x key: s[h][m][j] = 2^(e_q + e_k) * sum_d q[h][m][d] * k[h][j][d], int8 codes, D = 128.
cudaError_t launch_attn_qk_tc(const int8_t* qc, const int32_t* e_q, const int8_t* kc, const int32_t* e_k, int H, int M,
                              int J, int D, __half* s_out, Control* ctl, const DeviceInfo& dev, cudaStream_t stream) {
    // one k step per tile (k = D = 128): the epilogue, 64 KB of scores per tile and row block, sets the pace
    return launch_attn_tc<128, true, 1, 8>(qc, kc, nullptr, e_q, e_k, 0, H, M, D, J, s_out, ctl, dev, stream, true);
}

// Values from which one kernel makes the byte factors: 235 MB of them, nearly twice what the L2 holds. us in two kernels / one, graph replay, softmax
// outputs of normal scores with a deviation of 3 (x read once): 56 x 2048 x 2048 values 188.8 / 133.0, 32 x 2048 x 2048 106.2 / 82.6, 28 x 2048 x 2048
// 92.4 / 76.4, 24 x 2048 x 2048 77.3 / 67.6, 40 x 1500 x 1024 47.1 / 49.4, 16 x 1024 x 2048 24.0 / 32.6; of 1 (read twice): 188.6 / 183.5, 106.3 /
// 104.1, 92.2 / 91.4, 77.3 / 78.3, 47.0 / 49.3, 23.9 / 28.1. The grid's two meetings and a launch that overlaps nothing cost some 10 us, and in smaller
// arrays more of the second reading comes from the L2: the line lies where neither kind loses.
constexpr long long kOnceCount = 14ll << 23;

cudaError_t launch_log2_quantize(const __half* x, long long count, int bits, Control* ctl, int8_t* codes,
                                 uint32_t* max_bits_out, const DeviceInfo& dev, cudaStream_t stream, bool as_factors) {
    if (as_factors && count >= kOnceCount && count < (1ll << 35) && (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && (reinterpret_cast<uintptr_t>(codes) & 7u) == 0) {
        // all CTAs at once: one an SM
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(dev.sm_count);
        cfg.blockDim = dim3(kOnceThreads);
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, log2_factors_once_kernel, x, count, ctl, reinterpret_cast<uint8_t*>(codes), max_bits_out);
        if (e != cudaErrorCooperativeLaunchTooLarge) return e;
        (void)cudaGetLastError();                        // a part of the GPU only: in two kernels
    }
    // as many clusters as the control block has words for (232 CTAs: two per SM of most), fewer for small arrays
    long long clusters = (count / 8 + kRangeCtas * kLog2MaxThreads - 1) / (kRangeCtas * kLog2MaxThreads);
    if (clusters > Control::kRangeWords) clusters = Control::kRangeWords;
    if (clusters < 1) clusters = 1;
    const cudaError_t e = launch_overlapped(log2_absmax_kernel, dim3((unsigned int)clusters * kRangeCtas), kLog2MaxThreads, stream, x, count, ctl);
    if (e != cudaSuccess) return e;
    long long blocks = (count / 8 + 255) / 256;
    const long long cap = (long long)dev.sm_count * kLog2Ctas;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return launch_overlapped(log2_codes_kernel, dim3((unsigned int)blocks), 256, stream, x, count, bits, (int)clusters, ctl, codes, max_bits_out,
                             as_factors ? 1 : 0);
}

cudaError_t launch_attn_v_log2(const int8_t* pcodes, const uint32_t* max_bits, const int8_t* vq, const int32_t* e_v,
                               int H, int M, int J, int D, int bits, __half* y, int32_t* acc_dump, cudaStream_t stream) {
    const int quads = D / 4;
    const int rows = 256 / quads;                  // D <= 1024 and D % 4 == 0 are checked by the caller
    dim3 grid((M + rows - 1) / rows, H);
    attn_v_log2_kernel<<<grid, 256, 0, stream>>>(pcodes, max_bits, vq, e_v, M, J, D, bits, rows, y, acc_dump);
    return cudaGetLastError();
}

}  // namespace aq
