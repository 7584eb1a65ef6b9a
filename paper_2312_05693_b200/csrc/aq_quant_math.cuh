// The arithmetic of the activation quantizer (Eq. 1, Eq. 2 / Eq. 5 with zp = 0 and a power-of-two step),
// shared by the quantize kernels and the decode kernel that quantizes its own activations.
#pragma once

#include <cooperative_groups.h>

#include "aq_common.cuh"

namespace aq {

namespace {

__device__ inline int quantize_one(float v, float inv, float lo, float hi) {
    const float t = v * inv;                 // exact: inv is a power of two
    if (t != t) return 0;                    // NaN
    return (int)fminf(fmaxf(rintf(t), lo), hi);
}

// Eight halves -> eight codes in two 32-bit words, in half2 arithmetic, for exponents whose 2^-e is a
// normal half (|e| <= 14). Every step is exact or rounds exactly like the fp32 route: the product by
// a power of two is exact unless it leaves the half range (overflow saturates to Inf and is clamped
// like any large value; results below 2^-14 round to code 0 either way); NaN is cleared to 0 by a
// lane mask; clamping to the integer bounds before rounding gives the same code as after; adding
// 1536 (ulp 1 in [1024, 2048)) rounds to the nearest integer, ties to even, and leaves the code's
// two's-complement byte in the low 8 bits of the half's bit pattern.
__device__ __forceinline__ void quantize8_half2(const uint4& d, __half2 inv2, __half2 lo2, __half2 hi2, uint32_t& w0,
                                                uint32_t& w1) {
    const __half2* h = reinterpret_cast<const __half2*>(&d);
    const __half2 bias = __floats2half2_rn(1536.0f, 1536.0f);
    uint32_t r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __half2 t = __hmul2(h[i], inv2);
        const uint32_t ok = __heq2_mask(t, t);                            // 0xFFFF per lane that is not NaN
        uint32_t tb = *reinterpret_cast<uint32_t*>(&t) & ok;
        t = *reinterpret_cast<__half2*>(&tb);
        t = __hadd2(__hmin2(__hmax2(t, lo2), hi2), bias);
        r[i] = *reinterpret_cast<uint32_t*>(&t);
    }
    w0 = __byte_perm(r[0], r[1], 0x6420);
    w1 = __byte_perm(r[2], r[3], 0x6420);
}

// 8 halves -> 8 values in fp32 arithmetic. With TRIP factors (Eq. 5 with a per-channel alpha,
// `al` = the 8 factor bytes of these channels) channel k uses the step 2^(e + alpha_k) and its code
// is stored shifted left by alpha_k, the form in which the factor enters the integer product.
__device__ __forceinline__ uint2 quantize8_fp32(const uint4& d, int e, float lo, float hi, const uint2* al) {
    const __half* h = reinterpret_cast<const __half*>(&d);
    const uint8_t* ab = reinterpret_cast<const uint8_t*>(al);
    uint32_t out[2];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        uint32_t word = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = 4 * w + b;
            const int a = al ? (int)ab[i] : 0;
            const float inv = __int_as_float((127 - e - a) << 23);           // 2^-(e + alpha)
            word |= ((uint32_t)(quantize_one(__half2float(h[i]), inv, lo, hi) << a) & 0xFFu) << (8 * b);
        }
        out[w] = word;
    }
    return make_uint2(out[0], out[1]);
}

// The half2 route with TRIP factors (4-bit codes): lane k multiplies by 2^-(e + alpha_k), built from
// the factor byte as a half bit pattern (exponent field 15 - e - alpha_k, which must be 1..30),
// clamps to [-8, 7], rounds by adding and removing 1536, multiplies by 2^alpha_k (exact, |result|
// <= 128) and adds 1536 again so that the value's two's-complement byte sits in the low 8 bits.
__device__ __forceinline__ void quantize8_half2_trip(const uint4& d, int e, const uint2& al, uint32_t& w0, uint32_t& w1) {
    const __half2* h = reinterpret_cast<const __half2*>(&d);
    const __half2 bias = __floats2half2_rn(1536.0f, 1536.0f);
    const __half2 lo2 = __floats2half2_rn(-8.0f, -8.0f), hi2 = __floats2half2_rn(7.0f, 7.0f);
    const uint32_t inv_base = (uint32_t)(15 - e) * 0x04000400u;              // both lanes: (15 - e) << 10
    const uint32_t one_base = 15u * 0x04000400u;                            // 1.0 in both lanes
    uint32_t r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t word = i < 2 ? al.x : al.y;
        const uint32_t a0 = (word >> (16 * (i & 1))) & 0xFFu, a1 = (word >> (16 * (i & 1) + 8)) & 0xFFu;
        const uint32_t apair = (a0 | (a1 << 16)) << 10;
        uint32_t ib = inv_base - apair, sb = one_base + apair;
        __half2 t = __hmul2(h[i], *reinterpret_cast<__half2*>(&ib));
        const uint32_t ok = __heq2_mask(t, t);                              // clears NaN lanes
        uint32_t tb = *reinterpret_cast<uint32_t*>(&t) & ok;
        t = *reinterpret_cast<__half2*>(&tb);
        t = __hsub2(__hadd2(__hmin2(__hmax2(t, lo2), hi2), bias), bias);    // the 4-bit code, rounded to nearest even
        t = __hadd2(__hmul2(t, *reinterpret_cast<__half2*>(&sb)), bias);
        r[i] = *reinterpret_cast<uint32_t*>(&t);
    }
    w0 = __byte_perm(r[0], r[1], 0x6420);
    w1 = __byte_perm(r[2], r[3], 0x6420);
}

// 8 halves -> 8 stored codes (q - 2^(b-1)) of the zero-point quantizer in half2 arithmetic, for
// exponents whose 2^-e is a normal half. The product by 2^-e is exact (or saturates and is clamped);
// NaN lanes are cleared to 0, which becomes the code zp; clamping rint(t) + zp to [0, qr] equals
// clamping t to [-zp, qr - zp] before rounding (integer bounds); adding 1536 rounds to nearest even;
// adding the integer zp - 2^(b-1) keeps the sum inside [1024, 2048), so the code's byte is the low
// 8 bits of the half's bit pattern.
__device__ __forceinline__ void quantize8_half2_asym(const uint4& d, __half2 inv2, __half2 lo2, __half2 hi2,
                                                     __half2 shift2, uint32_t& w0, uint32_t& w1) {
    const __half2* h = reinterpret_cast<const __half2*>(&d);
    const __half2 bias = __floats2half2_rn(1536.0f, 1536.0f);
    uint32_t r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __half2 t = __hmul2(h[i], inv2);
        const uint32_t ok = __heq2_mask(t, t);
        uint32_t tb = *reinterpret_cast<uint32_t*>(&t) & ok;
        t = *reinterpret_cast<__half2*>(&tb);
        t = __hadd2(__hadd2(__hmin2(__hmax2(t, lo2), hi2), bias), shift2);
        r[i] = *reinterpret_cast<uint32_t*>(&t);
    }
    w0 = __byte_perm(r[0], r[1], 0x6420);
    w1 = __byte_perm(r[2], r[3], 0x6420);
}
// The same in fp32 arithmetic (inv = 2^-e), for the other exponents.
__device__ __forceinline__ uint2 quantize8_fp32_asym(const uint4& d, float inv, int zp, int bits) {
    const __half* h = reinterpret_cast<const __half*>(&d);
    const float fzp = (float)zp, fqr = (float)((1 << bits) - 1);
    uint32_t out[2];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        uint32_t word = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float t = __half2float(h[4 * w + b]) * inv;                          // exact
            int code = zp;                                                             // NaN: value 0
            if (t == t) code = (int)fminf(fmaxf(rintf(t) + fzp, 0.0f), fqr);
            word |= ((uint32_t)(code - (1 << (bits - 1))) & 0xFFu) << (8 * b);
        }
        out[w] = word;
    }
    return make_uint2(out[0], out[1]);
}

// Exponent and zero point (Eq. 6, Eq. 7): e the smallest with (2^b - 1) 2^e >= max - min, zp = -min / 2^e rounded to nearest even,
// clipped to the codes. hi, lo: bit patterns of the largest value and of the least one's magnitude, 0 where there is none; Inf counts as 65504.
// In single precision: 2^b - 1 times a power of two is a float, so that it is no less than max - min just when it is no less than the float
// next above that sum, and min / 2^e is exact. (Every thread does this behind the meeting of the maxima: in 64-bit integers, shifted by
// variables, 504 x 8064 took 7.17 us a quantize call instead of 6.84, 24 x 2048 2.28 instead of 2.17.)
__device__ __forceinline__ void zero_point_scale(unsigned int hi, unsigned int lo, int bits, int& e, int& zp) {
    const float least = __half2float(__ushort_as_half((unsigned short)min(lo, 0x7BFFu)));
    const int range = __float_as_int(__fadd_ru(__half2float(__ushort_as_half((unsigned short)min(hi, 0x7BFFu))), least));
    const int full = ((1 << (bits - 1)) - 1) << (24 - bits);            // the fraction of 2^b - 1: b - 1 ones
    e = range ? (range >> 23) - 127 - (bits - 1) + ((range & 0x7FFFFF) > full ? 1 : 0) : 0;
    zp = min(__float2int_rn(least * __int_as_float((127 - e) << 23)), (1 << bits) - 1);
}

// A CTA may write into another one's shared memory only once that one has started, which being scheduled together does
// not promise: every thread arrives at its kernel's top and waits just before the kernel's first remote store (a CTA
// whose share of X is empty gets there at once). Behind the loads the wait costs next to nothing: without it and with
// it 2.11 / 2.12 us on 6 x 4096, 3.44 / 3.47 us on 48 x 4096, 9.68 / 9.67 us on 2048 x 4096 (quantize calls, graph replay).
__device__ __forceinline__ void cluster_started_arrive() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_started_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// ---- the largest magnitudes of a whole array, without a word that has to be cleared beforehand: every cluster of
// kRangeCtas CTAs leaves one word in the control block, and whoever needs the outcome reads all of them.
constexpr int kRangeCtas = 8;
// What a CTA's threads have seen: bit patterns of halves, the largest positive (or absolute) value and (TWO_SIDED) the largest
// magnitude of a negative one. All threads of all CTAs of the cluster call this, once, behind cluster_started_wait(). peers: a
// shared-memory word per CTA of the cluster; peer_slot: this CTA's word of them in the cluster's first CTA.
template <bool TWO_SIDED, int THREADS>
__device__ __forceinline__ void leave_range(Control* ctl, unsigned int bmax, unsigned int bmin, const unsigned int* peers, unsigned int* peer_slot) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ unsigned int warp_max[THREADS / 32], warp_min[THREADS / 32];
    if (bmax > 0x7C00u) bmax = 0;                            // never publish NaN
    if (bmin > 0x7C00u) bmin = 0;
    bmax = __reduce_max_sync(0xFFFFFFFFu, bmax);
    if (TWO_SIDED) bmin = __reduce_max_sync(0xFFFFFFFFu, bmin);
    if ((threadIdx.x & 31) == 0) {
        warp_max[threadIdx.x >> 5] = bmax;
        warp_min[threadIdx.x >> 5] = bmin;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        bmax = __reduce_max_sync(0xFFFFFFFFu, threadIdx.x < THREADS / 32 ? warp_max[threadIdx.x] : 0u);
        bmin = __reduce_max_sync(0xFFFFFFFFu, threadIdx.x < THREADS / 32 ? warp_min[threadIdx.x] : 0u);
        if (threadIdx.x == 0) *peer_slot = bmax | (bmin << 16);
    }
    cluster.sync();
    if (cluster.block_rank() == 0 && threadIdx.x == 0) {
        unsigned int hi = 0, lo = 0;
#pragma unroll
        for (int r = 0; r < kRangeCtas; ++r) {
            hi = max(hi, peers[r] & 0xFFFFu);
            lo = max(lo, peers[r] >> 16);
        }
        ctl->range[blockIdx.x / kRangeCtas] = hi | (lo << 16);
    }
}
// The words of leave_range, met: largest positive (or absolute) value in the low half, largest magnitude of a negative
// one in the high half. Whole warps call this.
__device__ __forceinline__ unsigned int met_range(const Control* ctl, int words) {
    const unsigned int lane = threadIdx.x & 31;
    const unsigned int w = lane < (unsigned int)words ? ctl->range[lane] : 0u;
    return __reduce_max_sync(0xFFFFFFFFu, w & 0xFFFFu) | (__reduce_max_sync(0xFFFFFFFFu, w >> 16) << 16);
}
}  // namespace

}  // namespace aq
