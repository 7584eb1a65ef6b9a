// Activation side: layer-wise absolute maximum, power-of-two quantization to int8 / int4
// codes (paper Eq. 1, Eq. 2 / Eq. 5 with zp = 0, layer-wise scale of Sec. 4.4), and the
// token selection / gather of Eq. 4.
#include <cooperative_groups.h>

#include "aq_common.cuh"
#include "aq_quant_math.cuh"

namespace cg = cooperative_groups;

namespace aq {

namespace {

__device__ __forceinline__ uint4 quantize16_fp32(const uint4& d0, const uint4& d1, int e, float lo, float hi,
                                                 const uint4* al) {
    uint2 a0, a1;
    if (al) { a0 = make_uint2(al->x, al->y); a1 = make_uint2(al->z, al->w); }
    const uint2 r0 = quantize8_fp32(d0, e, lo, hi, al ? &a0 : nullptr);
    const uint2 r1 = quantize8_fp32(d1, e, lo, hi, al ? &a1 : nullptr);
    return make_uint4(r0.x, r0.y, r1.x, r1.y);
}

// ---- small activations (decode): maximum, exponent and codes in ONE kernel -------------
// One cluster of 8 CTAs x 512 threads holds the whole activation in registers (up to 8 vectors of
// 8 halves per thread), so x is read once; the CTAs' maxima are exchanged through distributed
// shared memory. The kernel also initialises the control block, so no memset precedes it.
// Latency is what it takes: one round trip for x, one for the exchange. us, graph replay, with two meetings, and a division per vector for
// its place, and without: 2 x 768 1.76 / 1.50, 48 x 4096 3.46 / 2.28; layers of 48 rows 4096 x 4096 in groups 10.5 / 9.5. With a zero
// point, which took the two kernels below before, 24 x 2048 x 2048 9.0 / 6.9.
constexpr int kSmallCtas = 8, kSmallThreads = 512, kSmallVecs = 8;
constexpr size_t kSmallMaxElems = (size_t)kSmallCtas * kSmallThreads * kSmallVecs * 8;   // 262144

// ASYM: with a zero point (Eq. 2, Eq. 5-7): least and greatest value, no given exponent, no factors.
template <bool ASYM>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads)
quantize_small_kernel(const uint4* __restrict__ x, int M, int vec_per_row, const int32_t* __restrict__ row_idx,
                      int bits, int scale_mode, int clip_shift_or_exp, Control* __restrict__ ctl,
                      uint2* __restrict__ q, int32_t* __restrict__ scale_exp_out, const uint2* __restrict__ alpha,
                      int k_max, int early_dependents, int32_t* __restrict__ zero_point_out) {
    constexpr int kWarps = kSmallThreads / 32;
    __shared__ unsigned int seen[kSmallCtas * kWarps];      // what every warp of the cluster saw
    __shared__ alignas(8) uint64_t met;                     // all of them are there
    const int rank = (int)cg::this_cluster().block_rank(), warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const uint32_t met_a = (uint32_t)__cvta_generic_to_shared(&met);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(met_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(met_a), "r"((uint32_t)sizeof(seen)) : "memory");
    }
    __syncwarp();
    cluster_started_arrive();
    __syncthreads();
    // The launch allows programmatic stream serialization, so this grid may be set up while the kernel
    // ahead of it drains; nothing is read or written before that kernel has completed. Only then is the
    // dependent launch allowed: a product kernel launched the same way behind this one may be set up on
    // the idle SMs and fetch its weights while this one runs (it waits for this grid before it reads the
    // codes), and by then everything that preceded this kernel on the stream is complete.
    // early_dependents: the caller has promised that nothing in flight writes the weights the product kernel
    // fetches ahead of its own wait, so that kernel may be set up before this one's wait ends as well.
    if (early_dependents) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!early_dependents) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int total = M * vec_per_row;
    uint4 buf[kSmallVecs];
    // all loads first, then the maximum: the loads of a thread are in flight together (one memory round
    // trip for the whole activation instead of one per vector)
#pragma unroll
    for (int i = 0; i < kSmallVecs; ++i) {
        const int v = (i * kSmallCtas + rank) * kSmallThreads + (int)threadIdx.x;
        buf[i] = make_uint4(0, 0, 0, 0);
        if (v < total) {
            if (row_idx) {
                const int m = v / vec_per_row, c = v % vec_per_row;
                buf[i] = __ldg(x + (size_t)row_idx[m] * vec_per_row + c);
            } else {
                buf[i] = __ldg(x + v);
            }
        }
    }
    __half2 hi2 = __float2half2_rn(0.0f), lo2 = hi2;
#pragma unroll
    for (int i = 0; i < kSmallVecs; ++i) {
        const __half2* h = reinterpret_cast<const __half2*>(&buf[i]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {                                  // NaN operands are dropped; absent vectors are zero
            if (ASYM) {
                lo2 = __hmin2(lo2, h[k]);
                hi2 = __hmax2(hi2, h[k]);
            } else {
                hi2 = __hmax2(hi2, __habs2(h[k]));
            }
        }
    }
    lo2 = __habs2(lo2);
    const unsigned int bmax = max((unsigned int)__half_as_ushort(__low2half(hi2)), (unsigned int)__half_as_ushort(__high2half(hi2)));
    const unsigned int bmin = max((unsigned int)__half_as_ushort(__low2half(lo2)), (unsigned int)__half_as_ushort(__high2half(lo2)));
    unsigned int all = __reduce_max_sync(0xFFFFFFFFu, bmax) | (ASYM ? __reduce_max_sync(0xFFFFFFFFu, bmin) << 16 : 0u);
    cluster_started_wait();
    // A warp's word goes to every CTA by an asynchronous remote store that counts on the receiver's barrier (a meeting inside each CTA and
    // one of the cluster before: 48 x 4096 in a layer call 0.3 us more). A CTA waits for all words that are sent to it, and
    // every warp sends its word whatever happens, so nobody writes to a CTA that has left.
    if (lane < kSmallCtas) {
        uint32_t slot, bar;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(slot) : "r"((uint32_t)__cvta_generic_to_shared(&seen[rank * kWarps + warp])), "r"(lane));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(met_a), "r"(lane));
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(slot), "r"(all), "r"(bar) : "memory");
    }
    __syncwarp();
    bool came = false;
    for (const long long t0 = clock64(); !came && (unsigned long long)(clock64() - t0) < 2 * kWaitCycles;) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(met_a) : "memory");
        came = ok != 0;
    }
    __syncwarp();
    all = 0;
#pragma unroll
    for (int i = 0; i < kSmallCtas * kWarps / 32; ++i) all = __vmaxu2(all, seen[i * 32 + lane]);
    all = __reduce_max_sync(0xFFFFFFFFu, all & 0xFFFFu) | (ASYM ? __reduce_max_sync(0xFFFFFFFFu, all >> 16) << 16 : 0u);
    int e, zp = 0;
    if constexpr (ASYM) zero_point_scale(all & 0xFFFFu, all >> 16, bits, e, zp);
    else e = scale_mode == AQ_SCALE_DYNAMIC ? layer_exponent_from_bits(all, bits) - clip_shift_or_exp - k_max : clip_shift_or_exp;
    if (rank == 0 && threadIdx.x == 0) {
        ctl->absmax_bits = ASYM ? 0u : all;
        ctl->scale_exp = e;
        ctl->status = came ? 0u : 13u;
        if (scale_exp_out) *scale_exp_out = e;
        if constexpr (ASYM) {
            ctl->zero_point = zp;
            if (zero_point_out) *zero_point_out = zp;
        }
    }
    if (rank == 0 && threadIdx.x < Control::kSplitWords) ctl->split_flags[threadIdx.x] = 0;    // the product kernel's shared-tile bits
    const float lo = -(float)(1 << (bits - 1)), hi = (float)((1 << (bits - 1)) - 1);
    if (alpha == nullptr && e >= -14 && e <= 14) {           // 2^-e is a normal half: codes in half2 arithmetic
        const __half2 inv2 = __float2half2_rn(__int_as_float((127 - e) << 23));
        const __half2 clo2 = __float2half2_rn(ASYM ? -(float)zp : lo), chi2 = __float2half2_rn(ASYM ? (float)((1 << bits) - 1 - zp) : hi);
        [[maybe_unused]] const __half2 shift2 = __float2half2_rn((float)(zp - (1 << (bits - 1))));
#pragma unroll
        for (int i = 0; i < kSmallVecs; ++i) {
            const int v = (i * kSmallCtas + rank) * kSmallThreads + (int)threadIdx.x;
            if (v < total) {
                uint2 w;
                if (ASYM) quantize8_half2_asym(buf[i], inv2, clo2, chi2, shift2, w.x, w.y);
                else quantize8_half2(buf[i], inv2, clo2, chi2, w.x, w.y);
                q[v] = w;
            }
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < kSmallVecs; ++i) {
        const int v = (i * kSmallCtas + rank) * kSmallThreads + (int)threadIdx.x;
        if (v < total) {
            uint2 al;
            if (alpha) al = __ldg(alpha + v % vec_per_row);
            q[v] = ASYM ? quantize8_fp32_asym(buf[i], __int_as_float((127 - e) << 23), zp, bits) : quantize8_fp32(buf[i], e, lo, hi, alpha ? &al : nullptr);
        }
    }
}

// ---- larger activations: two kernels, each of them plain (no grid-wide meeting, nothing to clear beforehand) ----
// range_kernel: clusters of eight CTAs take contiguous shares of X (16-byte loads, eight in flight per thread), find
// the share's minimum and maximum (symmetric scale: the largest magnitude), meet in distributed shared memory and
// leave one word per cluster in the control block. quantize_kernel: every warp reads those words (at most one per
// lane), and quantizes; X is read again, from L2 as far as it fits (126 MB). The second kernel, and the product behind
// it, are launched with programmatic stream serialization, so that a kernel's launch overlaps its predecessor.
// What it replaced: one cooperative kernel that parked X in shared memory between a grid-wide meeting, behind a node
// that cleared the control block. X crossed HBM and L2 once there, but of 12.1 us (2048 x 4096) 4 were the clearing and
// the cooperative launch and 2 the meeting. In graph replay over rotating inputs: 2048 x 4096 12.1 -> 9.1 us,
// 2048 x 11008 21.9 -> 18.0 us, 1024 x 5120 10.1 -> 6.6 us, 333 x 5120 8.3 -> 5.5 us.
constexpr int kRangeThreads = 512;
constexpr int kRangeInFlight = 8;
constexpr size_t kRangeFewVecs = (size_t)Control::kRangeWords * kRangeThreads * kRangeInFlight * 2;      // 237568 vectors: two turns of all loads in flight
// (Up to there 29 CTAs without a meeting beat clusters on all SMs: quantize calls, graph replay, 100 x 4096 4.12 / 3.69 us, 116 x 8192 4.71 / 3.94,
// 333 x 5120 5.54 / 4.50, 230 x 8192 5.64 / 4.70; with four turns 509 x 4096 5.66 / 4.95, but 400 x 8192 5.85 / 6.13. Layer calls gain less,
// 333 x 5120 x 5120 17.9 / 17.7, and 128 x 13824 x 5120 loses: 23.7 / 24.1. Gathered rows shorter than a CTA's step, every vector behind an index
// of its own: one turn. 2075 of 512 6.07 / 6.68, 1600 of 1152 6.48 / 6.84, but 333 of 5120 6.52 / 6.06, and with a zero point 1600 of 1152 7.20 / 6.77.)

// Place of element number v (per_row elements a row) in the gathered rows, carried along in steps: one division at the
// start instead of one per element (a 64-bit one each cost 8 us on 2458 gathered rows of 7168).
struct RowWalk {
    int m, c, step_m, step_c, per_row;
    __device__ __forceinline__ RowWalk(size_t v, int per_row_, int step) : per_row(per_row_) {
        if (v <= 0xFFFFFFFFull) {
            m = (int)((uint32_t)v / (uint32_t)per_row);
            c = (int)((uint32_t)v - (uint32_t)m * (uint32_t)per_row);
        } else {
            const size_t q = v / (size_t)per_row;
            m = (int)q;
            c = (int)(v - q * (size_t)per_row);
        }
        step_m = step / per_row;
        step_c = step - step_m * per_row;
    }
    __device__ __forceinline__ size_t source(const int32_t* row_idx) const { return (size_t)row_idx[m] * per_row + c; }
    __device__ __forceinline__ void next() {
        m += step_m;
        c += step_c;
        if (c >= per_row) { c -= per_row; ++m; }
    }
};

// CLUSTERS: launched in clusters of kRangeCtas; otherwise every CTA leaves a word of its own (arrays small enough for as many CTAs as
// there are words).
// IN_FLIGHT: loads of a thread in flight.
template <bool ASYM, bool CLUSTERS, int IN_FLIGHT = kRangeInFlight>
__global__ void __launch_bounds__(kRangeThreads, 2)
range_kernel(const uint4* __restrict__ x, size_t vecs /* of 8 halves */, int vec_per_row, const int32_t* __restrict__ row_idx,
             size_t vecs_per_cta, Control* __restrict__ ctl) {
    if constexpr (CLUSTERS) cluster_started_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");      // the kernel ahead may have written X
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t v0 = (size_t)blockIdx.x * vecs_per_cta;
    const size_t v1 = v0 + vecs_per_cta < vecs ? v0 + vecs_per_cta : vecs;
    __half2 hi2 = __float2half2_rn(0.0f), lo2 = hi2;        // the range always contains 0
    RowWalk at(row_idx ? v0 + threadIdx.x : 0, vec_per_row, kRangeThreads);
    for (size_t vb = v0 + threadIdx.x; vb < v1; vb += (size_t)kRangeThreads * IN_FLIGHT) {
        uint4 d[IN_FLIGHT];
#pragma unroll
        for (int i = 0; i < IN_FLIGHT; ++i) {
            const size_t v = vb + (size_t)i * kRangeThreads;
            d[i] = make_uint4(0u, 0u, 0u, 0u);
            if (v < v1) d[i] = __ldg(x + (row_idx ? at.source(row_idx) : v));
            if (row_idx) at.next();
        }
#pragma unroll
        for (int i = 0; i < IN_FLIGHT; ++i) {
            const __half2* h = reinterpret_cast<const __half2*>(&d[i]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {                    // NaN operands are dropped
                if (ASYM) {
                    lo2 = __hmin2(lo2, h[k]);
                    hi2 = __hmax2(hi2, h[k]);
                } else {
                    hi2 = __hmax2(hi2, __habs2(h[k]));
                }
            }
        }
    }
    // as magnitudes: bit patterns of non-negative halves order as integers; +-Inf stays Inf here
    unsigned int bmax = max((unsigned int)__half_as_ushort(__low2half(hi2)), (unsigned int)__half_as_ushort(__high2half(hi2)));
    unsigned int bmin = 0;
    if (ASYM) {
        const __half2 n2 = __habs2(lo2);
        bmin = max((unsigned int)__half_as_ushort(__low2half(n2)), (unsigned int)__half_as_ushort(__high2half(n2)));
    }
    if constexpr (!CLUSTERS) {
        __shared__ unsigned int warp_seen[kRangeThreads / 32];
        const unsigned int seen = __reduce_max_sync(0xFFFFFFFFu, bmax) | (ASYM ? __reduce_max_sync(0xFFFFFFFFu, bmin) << 16 : 0u);
        if ((threadIdx.x & 31) == 0) warp_seen[threadIdx.x >> 5] = seen;
        __syncthreads();
        if (threadIdx.x < 32) {
            const unsigned int w = threadIdx.x < kRangeThreads / 32 ? warp_seen[threadIdx.x] : 0u;
            const unsigned int hi = __reduce_max_sync(0xFFFFFFFFu, w & 0xFFFFu), lo = __reduce_max_sync(0xFFFFFFFFu, w >> 16);
            if (threadIdx.x == 0) ctl->range[blockIdx.x] = hi | (lo << 16);
        }
        return;
    }
    __shared__ unsigned int peers[kRangeCtas];
    cluster_started_wait();
    leave_range<ASYM, kRangeThreads>(ctl, bmax, bmin, peers, cg::this_cluster().map_shared_rank(&peers[cg::this_cluster().block_rank()], 0));
}

// What the product kernel finds in the control block.
__device__ __forceinline__ void publish_control(Control* ctl, unsigned int absmax_bits, int e, int zp, int32_t* scale_exp_out,
                                                int32_t* zero_point_out) {
    if (blockIdx.x != 0) return;
    if (threadIdx.x == 0) {
        ctl->absmax_bits = absmax_bits;
        ctl->scale_exp = e;
        ctl->zero_point = zp;
        ctl->status = 0;
        if (scale_exp_out) *scale_exp_out = e;
        if (zero_point_out) *zero_point_out = zp;
    }
    if (threadIdx.x < Control::kSplitWords) ctl->split_flags[threadIdx.x] = 0;      // the product kernel's shared-tile bits
}

constexpr int kQuantThreads = 256;
constexpr int kQuantUnits = 4;                               // units of 16 elements per thread, all loads in flight

// Loads of a thread's units: unit i is u0 + i * THREADS.
template <int THREADS>
__device__ __forceinline__ void load_units(const uint4* __restrict__ x, size_t u0, size_t total, int units_per_row,
                                           const int32_t* __restrict__ row_idx, uint4 (&d)[kQuantUnits][2]) {
    RowWalk at(row_idx ? u0 : 0, units_per_row, THREADS);
#pragma unroll
    for (int i = 0; i < kQuantUnits; ++i) {
        const size_t u = u0 + (size_t)i * THREADS;
        if (u < total) {
            const size_t src = 2 * (row_idx ? at.source(row_idx) : u);
            d[i][0] = __ldg(x + src);
            d[i][1] = __ldg(x + src + 1);
        }
        if (row_idx) at.next();
    }
}

// words > 0: dynamic scale from that many words of range_kernel; 0: the exponent is given
__global__ void __launch_bounds__(kQuantThreads)
quantize_kernel(const uint4* __restrict__ x, int M, int units_per_row /* 16-element units */,
                const int32_t* __restrict__ row_idx, int bits, int words, int clip_shift_or_exp,
                Control* __restrict__ ctl, uint4* __restrict__ q, int32_t* __restrict__ scale_exp_out,
                const uint4* __restrict__ alpha, int k_max) {
    // After this wait everything ahead (weight packing included) has completed: only now may the product kernel be
    // set up, which fetches weights before its own wait.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t total = (size_t)M * units_per_row;
    const size_t u0 = (size_t)blockIdx.x * (kQuantThreads * kQuantUnits) + threadIdx.x;
    uint4 d[kQuantUnits][2];
    load_units<kQuantThreads>(x, u0, total, units_per_row, row_idx, d);
    unsigned int absmax = 0;
    int e = clip_shift_or_exp;
    if (words) {
        absmax = met_range(ctl, words) & 0xFFFFu;
        e = layer_exponent_from_bits(absmax, bits) - clip_shift_or_exp - k_max;
    }
    publish_control(ctl, absmax, e, 0, scale_exp_out, nullptr);
    const float inv = __int_as_float((127 - e) << 23);      // 2^-e, |e| <= 40
    const float lo = -(float)(1 << (bits - 1)), hi = (float)((1 << (bits - 1)) - 1);
    const bool fast = alpha == nullptr && e >= -14 && e <= 14;   // 2^-e is a normal half
    const bool fast_trip = alpha != nullptr && bits == 4 && e >= -14 && e <= 10;   // so is 2^-(e + alpha), alpha <= 4
    const __half2 inv2 = __float2half2_rn(fast ? inv : 1.0f), lo2 = __float2half2_rn(lo), hi2 = __float2half2_rn(hi);
#pragma unroll
    for (int i = 0; i < kQuantUnits; ++i) {
        const size_t u = u0 + (size_t)i * kQuantThreads;
        if (u >= total) break;
        uint4 out;
        if (fast) {
            quantize8_half2(d[i][0], inv2, lo2, hi2, out.x, out.y);
            quantize8_half2(d[i][1], inv2, lo2, hi2, out.z, out.w);
        } else {
            uint4 al;
            if (alpha) al = __ldg(alpha + (size_t)(u % units_per_row));
            if (fast_trip) {
                quantize8_half2_trip(d[i][0], e, make_uint2(al.x, al.y), out.x, out.y);
                quantize8_half2_trip(d[i][1], e, make_uint2(al.z, al.w), out.z, out.w);
            } else {
                out = quantize16_fp32(d[i][0], d[i][1], e, lo, hi, alpha ? &al : nullptr);
            }
        }
        q[u] = out;
    }
}

// ---- zero-point variant (Eq. 2, Eq. 5-7 with alpha = 0, power-of-two scale) ---------------
// Codes from the minimum and maximum that range_kernel left (`words` words), as quantize_kernel.
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
quantize_asym_kernel(const uint4* __restrict__ x, int M, int units_per_row /* 16-element units */,
                     const int32_t* __restrict__ row_idx, int bits, int words, Control* __restrict__ ctl,
                     uint4* __restrict__ q, int32_t* __restrict__ scale_exp_out, int32_t* __restrict__ zero_point_out) {
    asm volatile("griddepcontrol.wait;" ::: "memory");                 // see quantize_kernel
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t total = (size_t)M * units_per_row;
    const size_t u0 = (size_t)blockIdx.x * (THREADS * kQuantUnits) + threadIdx.x;
    uint4 d[kQuantUnits][2];
    load_units<THREADS>(x, u0, total, units_per_row, row_idx, d);
    const unsigned int met = met_range(ctl, words);
    int e, zp;
    zero_point_scale(met & 0xFFFFu, met >> 16, bits, e, zp);
    publish_control(ctl, 0u, e, zp, scale_exp_out, zero_point_out);
    const int qr_i = (1 << bits) - 1, half_range = 1 << (bits - 1);
    const float inv = __int_as_float((127 - e) << 23);      // 2^-e
    const float fzp = (float)zp, fqr = (float)qr_i;
    const bool fast = e >= -14 && e <= 14;                   // 2^-e is a normal half
    const __half2 inv2 = __float2half2_rn(fast ? inv : 1.0f);
    const __half2 clo2 = __float2half2_rn(-fzp), chi2 = __float2half2_rn(fqr - fzp);
    const __half2 shift2 = __float2half2_rn((float)(zp - half_range));
#pragma unroll
    for (int i = 0; i < kQuantUnits; ++i) {
        const size_t u = u0 + (size_t)i * THREADS;
        if (u >= total) break;
        uint32_t out[4];
        if (fast) {
            quantize8_half2_asym(d[i][0], inv2, clo2, chi2, shift2, out[0], out[1]);
            quantize8_half2_asym(d[i][1], inv2, clo2, chi2, shift2, out[2], out[3]);
        } else {
            const uint2 c0 = quantize8_fp32_asym(d[i][0], inv, zp, bits), c1 = quantize8_fp32_asym(d[i][1], inv, zp, bits);
            out[0] = c0.x; out[1] = c0.y; out[2] = c1.x; out[3] = c1.y;
        }
        q[u] = make_uint4(out[0], out[1], out[2], out[3]);
    }
}

// ---- TRIP calibration (Eq. 8 with the clipping of Eq. 5) ---------------------------------
__global__ void __launch_bounds__(256)
absmax_plain_kernel(const __half* __restrict__ x, int M, int K, const int32_t* __restrict__ row_idx,
                    Control* __restrict__ ctl) {
    const size_t total = (size_t)M * K;
    unsigned int b = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(i / K), k = (int)(i % K);
        const unsigned int hb = __half_as_ushort(x[(size_t)(row_idx ? row_idx[m] : m) * K + k]) & 0x7FFFu;
        if (hb <= 0x7C00u) b = max(b, hb);                                  // NaN is ignored
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xFFFFFFFFu, b, o));
    if ((threadIdx.x & 31) == 0 && b != 0) atomicMax(&ctl->absmax_bits, b);
}

// One thread per channel walks the tokens in ascending order and keeps one binary64 error sum per
// candidate factor (product and sum rounded separately), then takes the smallest factor among the
// least errors. Consecutive threads read consecutive halves of a row.
__global__ void __launch_bounds__(128)
trip_calibrate_kernel(const __half* __restrict__ x, int M, int K, const int32_t* __restrict__ row_idx, int bits,
                      int k_max, Control* __restrict__ ctl, uint8_t* __restrict__ alpha_out,
                      int32_t* __restrict__ scale_exp_out) {
    const int e = layer_exponent_from_bits(ctl->absmax_bits, bits) - k_max;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->scale_exp = e;
        if (scale_exp_out) *scale_exp_out = e;
    }
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const double lo = -(double)(1 << (bits - 1)), hi = (double)((1 << (bits - 1)) - 1);
    double err[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int m = 0; m < M; ++m) {
        const float xf = __half2float(x[(size_t)(row_idx ? row_idx[m] : m) * K + k]);
        if (!isfinite(xf)) continue;
        const double xv = (double)xf;
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            if (a <= k_max) {
                const double inv = __longlong_as_double((long long)(1023 - e - a) << 52);    // 2^-(e+a)
                const double step = __longlong_as_double((long long)(1023 + e + a) << 52);   // 2^(e+a)
                const double qv = fmin(fmax(rint(__dmul_rn(xv, inv)), lo), hi);
                const double d = __dsub_rn(xv, __dmul_rn(qv, step));
                err[a] = __dadd_rn(err[a], __dmul_rn(d, d));
            }
        }
    }
    int best = 0;
    double best_err = err[0];
#pragma unroll
    for (int a = 1; a < 5; ++a)
        if (a <= k_max && err[a] < best_err) { best = a; best_err = err[a]; }
    alpha_out[k] = (uint8_t)best;
}

// ---- token selection: the n_keep highest scores, equal scores toward the lower index, ascending indices out ----
// One CTA. Scores become 32-bit keys whose unsigned order is the scores' order (-0 and +0 share a key, so
// they tie as they do in a float comparison). The key T of the n_keep-th highest score is built from the top,
// two bits per pass: a digit is the largest one for which at least n_keep keys are >= the candidate (16
// counting passes, one block-wide sum of three counts each). Every key above T is kept, and of the keys equal to T the first
// n_keep - #{key > T} in index order; one block scan over (greater, equal) counts gives each kept token its
// place in the output. Exactly n_keep indices are written whatever the scores hold (NaNs order by their bit
// patterns: positive ones above +inf, negative ones below -inf).
// REGS: M <= 4 * kSelThreads and each thread keeps its four consecutive tokens' keys in registers for all
// passes (a counting pass is then twelve compares, two rounds of warp reductions and one barrier).
constexpr int kSelThreads = 1024;
constexpr int kSelStage = 8192;           // keys held in shared memory up to this M; beyond it every pass reads the scores

__device__ __forceinline__ uint32_t score_key(float s) {
    uint32_t u = __float_as_uint(s);
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

template <bool REGS>
__global__ void __launch_bounds__(kSelThreads)
token_select_kernel(const float* __restrict__ scores, int M, int n_keep, int32_t* __restrict__ idx) {
    __shared__ uint32_t skeys[REGS ? 1 : kSelStage];
    __shared__ int wsum[2][3][32];
    __shared__ unsigned long long wscan[32];
    __shared__ unsigned long long running;
    asm volatile("griddepcontrol.wait;" ::: "memory");              // set up while the kernel ahead drains
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool staged = !REGS && M <= kSelStage;
    uint32_t kreg[4] = {0u, 0u, 0u, 0u};                 // key 0 is below every candidate of the passes
    if (REGS) {
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (4 * tid + b < M) kreg[b] = score_key(__ldg(scores + 4 * tid + b));
    } else if (staged) {
        for (int j = tid; j < M; j += kSelThreads) skeys[j] = score_key(__ldg(scores + j));
    }
    if (tid == 0) running = 0ull;
    __syncthreads();
    auto key_at = [&](int j) -> uint32_t { return staged ? skeys[j] : score_key(__ldg(scores + j)); };
    // One pass settles two bits of T: the counts of keys >= T | (v << shift) for v = 1, 2, 3, the same values
    // in every thread; T takes the largest v whose count still reaches n_keep. buf alternates so that a pass
    // never overwrites sums a slower warp is still reading.
    uint32_t T = 0u;
    int above = 0;            // #{ key >= T + (1 << settled digits' lowest bit) }: 0 while nothing is settled
    for (int shift = 30; shift >= 0; shift -= 2) {
        const uint32_t c1 = T | (1u << shift), c2 = T | (2u << shift), c3 = T | (3u << shift);
        int n1 = 0, n2 = 0, n3 = 0;
        if (REGS) {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                n1 += (int)(kreg[b] >= c1); n2 += (int)(kreg[b] >= c2); n3 += (int)(kreg[b] >= c3);
            }
        } else {
            for (int j = tid; j < M; j += kSelThreads) {
                const uint32_t k = key_at(j);
                n1 += (int)(k >= c1); n2 += (int)(k >= c2); n3 += (int)(k >= c3);
            }
        }
        n1 = __reduce_add_sync(0xFFFFFFFFu, n1);
        n2 = __reduce_add_sync(0xFFFFFFFFu, n2);
        n3 = __reduce_add_sync(0xFFFFFFFFu, n3);
        const int buf = (shift >> 1) & 1;
        if (lane == 0) { wsum[buf][0][wid] = n1; wsum[buf][1][wid] = n2; wsum[buf][2][wid] = n3; }
        __syncthreads();
        n1 = __reduce_add_sync(0xFFFFFFFFu, wsum[buf][0][lane]);
        n2 = __reduce_add_sync(0xFFFFFFFFu, wsum[buf][1][lane]);
        n3 = __reduce_add_sync(0xFFFFFFFFu, wsum[buf][2][lane]);
        // counts fall with v. The candidate one digit step above the chosen one is the next v, or, for
        // v = 3, the previous pass's upper neighbour, whose count `above` already holds.
        if (n3 >= n_keep)      { T = c3; }
        else if (n2 >= n_keep) { T = c2; above = n3; }
        else if (n1 >= n_keep) { T = c1; above = n2; }
        else                   { above = n1; }
        // A candidate with n_keep keys from it on settles it: those are kept, none equal to the key below (4096 scores that
        // differ are through four passes early, as a rule).
        const uint32_t exact = n3 == n_keep ? c3 : n2 == n_keep ? c2 : n1 == n_keep ? c1 : 0u;
        if (exact) {
            T = exact - 1u;
            above = n_keep;
            break;
        }
    }
    const int greater = above;                          // after the last pass the step is 1: #{ key > T }
    const int need = n_keep - greater;                  // ties at T to keep, lowest indices first

    // four consecutive tokens per thread; counts packed as (equal << 32) | greater
    for (int base = 0; base < M; base += 4 * kSelThreads) {
        const int j0 = base + 4 * tid;
        uint32_t gt = 0u, eq = 0u;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (j0 + b < M) {
                const uint32_t k = REGS ? kreg[b] : key_at(j0 + b);
                gt |= (uint32_t)(k > T) << b;
                eq |= (uint32_t)(k == T) << b;
            }
        }
        const unsigned long long own = ((unsigned long long)__popc(eq) << 32) | (unsigned long long)__popc(gt);
        unsigned long long incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wscan[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            unsigned long long ws = wscan[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, ws, o);
                if (lane >= o) ws += t;
            }
            wscan[lane] = ws;   // inclusive over warps
        }
        __syncthreads();
        const unsigned long long before = running + (wid ? wscan[wid - 1] : 0ull) + incl - own;
        int gt_before = (int)(uint32_t)before, eq_before = (int)(before >> 32);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if ((gt >> b) & 1u) {
                idx[gt_before + min(eq_before, need)] = j0 + b;
                ++gt_before;
            } else if ((eq >> b) & 1u) {
                if (eq_before < need) idx[gt_before + eq_before] = j0 + b;
                ++eq_before;
            }
        }
        __syncthreads();
        if (tid == 0) running += wscan[31];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256)
gather_rows_kernel(const uint4* __restrict__ x, int vec_per_row, const int32_t* __restrict__ idx,
                   int n_keep, uint4* __restrict__ out) {
    const size_t total = (size_t)n_keep * vec_per_row;
    for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < total;
         v += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(v / vec_per_row), c = (int)(v % vec_per_row);
        out[v] = __ldg(x + (size_t)idx[m] * vec_per_row + c);
    }
}

}  // namespace

namespace {
// Returns the number of words range_kernel leaves in the control block.
template <bool ASYM>
cudaError_t launch_range(const __half* x, int M, int K, const int32_t* row_idx, Control* ctl, cudaStream_t stream, int& words) {
    const size_t vecs = (size_t)M * (K / 8);
    if (vecs <= (!ASYM && row_idx && K / 8 < kRangeThreads ? kRangeFewVecs / 2 : kRangeFewVecs)) {
        // no meeting of clusters: as many CTAs as the control block has words for, fewer when one would have less than two vectors a thread
        size_t ctas = (vecs + kRangeThreads * 2 - 1) / (kRangeThreads * 2);
        if (ctas > Control::kRangeWords) ctas = Control::kRangeWords;
        words = (int)ctas;
        return launch_overlapped(range_kernel<ASYM, false>, dim3((unsigned int)ctas), kRangeThreads, stream, reinterpret_cast<const uint4*>(x), vecs, K / 8, row_idx,
                                 (vecs + ctas - 1) / ctas, ctl);
    }
    // as many clusters as the control block has words for (232 CTAs of 512 threads, all resident at once), fewer when
    // a CTA would have less than two vectors per thread
    const size_t per_cluster = (size_t)kRangeCtas * kRangeThreads * 2;
    size_t clusters = (vecs + per_cluster - 1) / per_cluster;
    if (clusters > Control::kRangeWords) clusters = Control::kRangeWords;
    words = (int)clusters;
    const size_t ctas = clusters * kRangeCtas;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)ctas);
    cfg.blockDim = dim3(kRangeThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = kRangeCtas;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    // Ten loads in flight where that saves a turn (2048 x 4096, 8.8 vectors a thread, 7.90 / 7.52 us a quantize call, 2458 x 7168 15.6 / 15.2;
    // where it does not it costs 0.1 us: 1024 x 5120 6.05 / 6.21).
    const size_t per_cta = (vecs + ctas - 1) / ctas, per_thread = (per_cta + kRangeThreads - 1) / kRangeThreads;
    auto* kernel = (per_thread + 9) / 10 < (per_thread + kRangeInFlight - 1) / kRangeInFlight ? range_kernel<ASYM, true, 10> : range_kernel<ASYM, true>;
    return cudaLaunchKernelEx(&cfg, kernel, reinterpret_cast<const uint4*>(x), vecs, K / 8, row_idx, per_cta, ctl);
}

size_t quantize_grid(int M, int K, int threads) {
    const size_t per_cta = (size_t)threads * kQuantUnits;
    return ((size_t)M * (K / 16) + per_cta - 1) / per_cta;
}
}  // namespace

cudaError_t launch_quantize(const __half* x, int M, int K, const int32_t* row_idx, int bits,
                            int scale_mode, int clip_shift_or_exp, Control* ctl, int8_t* q,
                            int32_t* scale_exp_out, cudaStream_t stream, const uint8_t* alpha, int k_max) {
    int words = 0;
    if (scale_mode == AQ_SCALE_DYNAMIC) {
        const cudaError_t e = launch_range<false>(x, M, K, row_idx, ctl, stream, words);
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(quantize_kernel, dim3((unsigned int)quantize_grid(M, K, kQuantThreads)), kQuantThreads, stream, reinterpret_cast<const uint4*>(x), M, K / 16,
                             row_idx, bits, words, clip_shift_or_exp, ctl, reinterpret_cast<uint4*>(q), scale_exp_out,
                             reinterpret_cast<const uint4*>(alpha), k_max);
}

cudaError_t launch_trip_calibrate(const __half* x, int M, int K, const int32_t* row_idx, int bits, int k_max,
                                  Control* ctl, uint8_t* alpha_out, int32_t* scale_exp_out, const DeviceInfo& dev,
                                  cudaStream_t stream) {
    const size_t total = (size_t)M * K;
    size_t blocks = (total + 255) / 256;
    const size_t cap = (size_t)dev.sm_count * 8;
    if (blocks > cap) blocks = cap;
    absmax_plain_kernel<<<(unsigned int)blocks, 256, 0, stream>>>(x, M, K, row_idx, ctl);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    trip_calibrate_kernel<<<(K + 127) / 128, 128, 0, stream>>>(x, M, K, row_idx, bits, k_max, ctl, alpha_out,
                                                               scale_exp_out);
    return cudaGetLastError();
}

cudaError_t launch_quantize_asym(const __half* x, int M, int K, const int32_t* row_idx, int bits, Control* ctl,
                                 int8_t* q, int32_t* scale_exp_out, int32_t* zero_point_out, cudaStream_t stream) {
    int words = 0;
    const cudaError_t e = launch_range<true>(x, M, K, row_idx, ctl, stream, words);
    if (e != cudaSuccess) return e;
    // 256 threads a CTA, or 512 where that makes one to four CTAs an SM. The kernel is set up while range_kernel's CTAs, one or two an SM, still run,
    // and takes few registers (48): up to three of its small CTAs then crowd the SMs with room while others get none. us a quantize call, 256 / 512
    // threads: 504 x 8064 6.84 / 6.74, 1199 x 5504 7.25 / 6.84, 2048 x 4096 7.38 / 7.03; but 333 x 5120 4.59 / 5.20, 2048 x 11008 12.5 / 13.7.
    const size_t ctas = quantize_grid(M, K, kQuantThreads);
    const bool large = ctas > 148 && ctas <= 4 * 148;
    const int threads = large ? 2 * kQuantThreads : kQuantThreads;
    return launch_overlapped(large ? quantize_asym_kernel<2 * kQuantThreads> : quantize_asym_kernel<kQuantThreads>, dim3((unsigned int)quantize_grid(M, K, threads)),
                             threads, stream, reinterpret_cast<const uint4*>(x), M, K / 16, row_idx, bits, words, ctl, reinterpret_cast<uint4*>(q), scale_exp_out,
                             zero_point_out);
}

bool quantize_small_fits(int M, int K) { return (size_t)M * (size_t)K <= kSmallMaxElems; }

cudaError_t launch_quantize_small(const __half* x, int M, int K, const int32_t* row_idx, int bits, int scale_mode,
                                  int clip_shift_or_exp, Control* ctl, int8_t* q, int32_t* scale_exp_out,
                                  cudaStream_t stream, const uint8_t* alpha, int k_max, bool early_dependents) {
    // the kernel touches no memory before the kernel ahead of it has completed
    return launch_overlapped(quantize_small_kernel<false>, dim3(kSmallCtas), kSmallThreads, stream, reinterpret_cast<const uint4*>(x), M, K / 8, row_idx, bits,
                             scale_mode, clip_shift_or_exp, ctl, reinterpret_cast<uint2*>(q), scale_exp_out, reinterpret_cast<const uint2*>(alpha), k_max,
                             early_dependents ? 1 : 0, nullptr);
}

cudaError_t launch_quantize_small_asym(const __half* x, int M, int K, const int32_t* row_idx, int bits, Control* ctl, int8_t* q, int32_t* scale_exp_out,
                                       int32_t* zero_point_out, cudaStream_t stream, bool early_dependents) {
    return launch_overlapped(quantize_small_kernel<true>, dim3(kSmallCtas), kSmallThreads, stream, reinterpret_cast<const uint4*>(x), M, K / 8, row_idx, bits,
                             AQ_SCALE_DYNAMIC, 0, ctl, reinterpret_cast<uint2*>(q), scale_exp_out, nullptr, 0, early_dependents ? 1 : 0, zero_point_out);
}

cudaError_t launch_token_select(const float* scores, int M, int n_keep, int32_t* idx, void* scratch,
                                cudaStream_t stream) {
    (void)scratch;
    if (n_keep == 0) return cudaSuccess;
    if (M <= 4 * kSelThreads)
        return launch_overlapped(token_select_kernel<true>, dim3(1), kSelThreads, stream, scores, M, n_keep, idx);
    return launch_overlapped(token_select_kernel<false>, dim3(1), kSelThreads, stream, scores, M, n_keep, idx);
}

cudaError_t launch_token_compact(const __half* x, int K, const int32_t* idx, int n_keep, __half* out,
                                 const DeviceInfo& dev, cudaStream_t stream) {
    if (n_keep == 0) return cudaSuccess;
    const int vec_per_row = K / 8;
    const size_t total = (size_t)n_keep * vec_per_row;
    size_t blocks = (total + 255) / 256;
    const size_t cap = (size_t)dev.sm_count * 16;
    if (blocks > cap) blocks = cap;
    gather_rows_kernel<<<(unsigned int)blocks, 256, 0, stream>>>(
        reinterpret_cast<const uint4*>(x), vec_per_row, idx, n_keep, reinterpret_cast<uint4*>(out));
    return cudaGetLastError();
}

}  // namespace aq
