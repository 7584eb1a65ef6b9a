// Integer product for few rows (M <= 16 per pass): weight-streaming reductions that read
// every packed weight byte from HBM once per 16 activation rows. They compute the sums of
// Sec. 4.4 / Algorithm 1 and the floating-point output.
//
// Two kernels:
//  * a general one (dumps of per-group sums, scales that are not 16-byte aligned, or any M when forced): a CTA owns 32 output channels
//    (one lane each), its 8 warps split K by 128-k block, products use dp4a on weights
//    widened to 16*code, warps meet in shared memory;
//  * a streaming one for M <= 16: a thread-block cluster shares a
//    128-channel tile and splits K; in each CTA a producer thread streams 8 KB packed blocks
//    and their activation codes into a shared-memory ring with TMA, eight consumer warps
//    multiply (dp4a for one row, the warp-level int8 MMA, weights by eight or twice eight rows, above). Every CTA keeps the sums over
//    its k range in its own shared memory and writes those of the channels it does not finish into the shared
//    memory of the CTA that does, whose barrier counts them, and every CTA finishes its slice of the tile's channels
//    (integer sums are exact in any order, fp32 ones are added in an order that does not depend on timing). No
//    workspace, no atomics.
#include <cuda.h>

#include "aq_common.cuh"
#include "aq_quant_math.cuh"

namespace aq {

namespace {

constexpr int kDecWarps = 8;
constexpr int kDecThreads = kDecWarps * 32;
constexpr int kDecPrefetch = 4;      // 128-k blocks in flight per warp (4 x 16 B per lane each)

// Chaining: the code the next layer's quantizer gives the fp16 output value (static exponent; NaN -> 0).
__device__ __forceinline__ int next_code(__half hv, float inv, float lo, float hi) {
    const float t = __half2float(hv) * inv;                 // exact: inv is a power of two
    if (t != t) return 0;
    return (int)fminf(fmaxf(rintf(t), lo), hi);
}

// Chaining: a warp's codes of one token (lane = consecutive channels) are stored one byte each or, packed,
// the even lane stores its code and its neighbour's in one byte of q4 [M][N/2]. All 32 lanes call this
// together; `valid` lanes (the same for a lane pair) store.
__device__ __forceinline__ void store_next_code(int8_t* q_next, size_t index, int code, int packed, bool valid, int lane) {
    if (packed) {
        const int hi = __shfl_down_sync(0xFFFFFFFFu, code, 1);
        if (valid && !(lane & 1)) reinterpret_cast<uint8_t*>(q_next)[index >> 1] = (uint8_t)((code & 0xF) | (hi << 4));
    } else if (valid) {
        q_next[index] = (int8_t)code;
    }
}

// CTA = 32 output channels (one lane each) x all of K, K split over the 8 warps by 128-k
// block; grid.y walks the rows in chunks of MB.
template <int MB, bool GROUPED>
__global__ void __launch_bounds__(kDecThreads)
gemm_decode_kernel(const int8_t* __restrict__ q, int M, int K, int N, int Npad,
                   const uint8_t* __restrict__ w_packed, const __half* __restrict__ w_scales,
                   const int32_t* __restrict__ scale_exp, __half* __restrict__ y,
                   int32_t* __restrict__ acc_dump, Control* __restrict__ ctl, const float* __restrict__ chan_offset, int zp_mid,
                   int8_t* __restrict__ q_next, float next_inv, float next_lo, float next_hi, int clear_status,
                   int next_packed) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // this kernel has no bounded waits; after a quantize kernel of the same call the word is that kernel's
    if (clear_status && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) ctl->status = 0;
    const int KB = k_blocks(K);
    const int n0 = blockIdx.x * 32;
    const int nt = n0 / kTileN, r = (n0 % kTileN) + lane;
    const int n = n0 + lane;
    const int m0 = blockIdx.y * MB;
    const uint8_t* wbase = w_packed + (size_t)nt * KB * kBlockBytes + (size_t)r * 16;

    int acc[MB];
    float fsum[MB];
#pragma unroll
    for (int m = 0; m < MB; ++m) { acc[m] = 0; fsum[m] = 0.0f; }

    const int T = KB > warp ? (KB - warp + kDecWarps - 1) / kDecWarps : 0;
    uint4 buf[kDecPrefetch][4];
#pragma unroll
    for (int d = 0; d < kDecPrefetch; ++d) {
        if (d < T) {
            const uint8_t* p = wbase + (size_t)(warp + d * kDecWarps) * kBlockBytes;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                buf[d][j] = __ldg(reinterpret_cast<const uint4*>(p + j * kTileN * 16));
        }
    }
    for (int t0 = 0; t0 < T; t0 += kDecPrefetch) {
#pragma unroll
        for (int d = 0; d < kDecPrefetch; ++d) {
            const int t = t0 + d;
            if (t >= T) break;
            const int kb = warp + t * kDecWarps;
            uint4 cur[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) cur[j] = buf[d][j];
            if (t + kDecPrefetch < T) {
                const uint8_t* p = wbase + (size_t)(kb + kDecPrefetch * kDecWarps) * kBlockBytes;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    buf[d][j] = __ldg(reinterpret_cast<const uint4*>(p + j * kTileN * 16));
            }
            if (GROUPED) {
#pragma unroll
                for (int m = 0; m < MB; ++m) acc[m] = 0;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (kb * kTileK + 32 * j >= K) break;            // a last block padded with zero codes (K % 128 != 0)
                const uint32_t w[4] = {cur[j].x, cur[j].y, cur[j].z, cur[j].w};
                uint32_t w8[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    w8[2 * i] = (w[i] << 4) & 0xF0F0F0F0u;       // 16*code for k0..k0+3
                    w8[2 * i + 1] = w[i] & 0xF0F0F0F0u;          // 16*code for k0+4..k0+7
                }
#pragma unroll
                for (int m = 0; m < MB; ++m) {
                    if (m0 + m < M) {
                        const uint4* xp = reinterpret_cast<const uint4*>(
                            q + (size_t)(m0 + m) * K + kb * kTileK + 32 * j);
                        const uint4 x0 = __ldg(xp), x1 = __ldg(xp + 1);
                        int a = acc[m];
                        a = __dp4a((int)w8[0], (int)x0.x, a);
                        a = __dp4a((int)w8[1], (int)x0.y, a);
                        a = __dp4a((int)w8[2], (int)x0.z, a);
                        a = __dp4a((int)w8[3], (int)x0.w, a);
                        a = __dp4a((int)w8[4], (int)x1.x, a);
                        a = __dp4a((int)w8[5], (int)x1.y, a);
                        a = __dp4a((int)w8[6], (int)x1.z, a);
                        a = __dp4a((int)w8[7], (int)x1.w, a);
                        acc[m] = a;
                    }
                }
            }
            if (GROUPED) {
                const float s = __half2float(w_scales[(size_t)kb * Npad + n]);
#pragma unroll
                for (int m = 0; m < MB; ++m) {
                    const int a = acc[m] >> 4;                   // exact: sums are multiples of 16
                    fsum[m] = fmaf((float)a, s, fsum[m]);
                    if (acc_dump && m0 + m < M && n < N)
                        acc_dump[((size_t)(m0 + m) * N + n) * KB + kb] = a;
                }
            }
        }
    }

    // cross-warp reduction: integers when one scale spans K, floats otherwise
    __shared__ int red[kDecWarps][MB][32];
#pragma unroll
    for (int m = 0; m < MB; ++m)
        red[warp][m][lane] = GROUPED ? __float_as_int(fsum[m]) : acc[m];
    __syncthreads();
    const float pe = __int_as_float((127 + *scale_exp) << 23);   // 2^e
    for (int m = warp; m < MB; m += kDecWarps) {
        if (m0 + m >= M) continue;                               // the same for the whole warp
        const bool n_ok = n < N;
        const float off = chan_offset && n_ok ? __fmul_rn(offset_factor(ctl, zp_mid), chan_offset[n]) : 0.0f;
        float out;
        if (GROUPED) {
            float s = 0.0f;
#pragma unroll
            for (int w = 0; w < kDecWarps; ++w) s += __int_as_float(red[w][m][lane]);
            out = (s + off) * pe;
        } else {
            int s = 0;
#pragma unroll
            for (int w = 0; w < kDecWarps; ++w) s += red[w][m][lane];
            s >>= 4;
            if (acc_dump && n_ok) acc_dump[(size_t)(m0 + m) * N + n] = s;
            out = fmaf((float)s, n_ok ? __half2float(w_scales[n]) : 0.0f, off) * pe;
        }
        const __half hv = __float2half_rn(out);
        if (q_next)
            store_next_code(q_next, (size_t)(m0 + m) * N + n, next_code(hv, next_inv, next_lo, next_hi), next_packed, n_ok, lane);
        else if (n_ok)
            y[(size_t)(m0 + m) * N + n] = hv;
    }
}

// ---------------------------------------------------------------------------------------
// Streaming kernel (M <= 16)
// ---------------------------------------------------------------------------------------
constexpr unsigned long long kStrWaitCycles = 4000000000ull;
// For what its cluster's other CTAs send a CTA waits longer: one of them that gave up elsewhere sends all the same.
constexpr unsigned long long kStrPeerCycles = 4 * kStrWaitCycles;
constexpr int kFuseMaxBlocks = 64;        // k blocks per CTA up to which a single row is quantized inside the product kernel
// Several rows (see decode_can_fuse_quantize): vectors of eight elements that a consumer thread holds at most while it quantizes them.
constexpr int kSliceVecs = 10;
constexpr long kFuseElems = 12288, kFuseWeightBytes = 4l << 20, kSliceElemsFrom = 16384;

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool str_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(s_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// One thread of a converged warp: the compiler then knows that a copy has one set of operands (see elect_one in aq_tc.cuh).
__device__ __forceinline__ bool s_elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// Bounded wait; false when the limit ran out or another thread of the CTA already gave up.
__device__ __forceinline__ bool str_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag) {
    if (str_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    uint32_t spins = 0;
    while (!str_try_wait(bar, parity)) {
        if ((++spins & 0x3FFu) == 0) {
            if (*abort_flag) return false;
            if ((unsigned long long)(clock64() - t0) > kStrWaitCycles) { *abort_flag = 1; return false; }
        }
    }
    return true;
}

// Bounded wait for what the cluster's other CTAs send, also after this CTA has given up elsewhere: it must be there when it comes.
// Their stores count at the scope of the cluster, so this waits at that scope (a wait without it is one at the scope of the CTA).
__device__ __forceinline__ bool str_try_wait_peers(uint64_t* bar) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(s_u32(bar)) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void str_wait_peers(uint64_t* bar, volatile uint32_t* abort_flag) {
    if (str_try_wait_peers(bar)) return;
    const long long t0 = clock64();
    while (!str_try_wait_peers(bar))
        if ((unsigned long long)(clock64() - t0) > kStrPeerCycles) { *abort_flag = 1; return; }
}

// One row uses dp4a; more rows use the warp-level int8 MMA (m16n8k32: 16 channels by eight rows, once or twice),
// with the activation tile stored 128-byte swizzled so that fragment loads are free of bank conflicts.
// Ring depth 8 (64 KB of weights in flight per CTA, two CTAs per SM): 9 stages for 16 rows and 12 for one
// row, which shared memory would allow, measured no faster.
template <int MB> struct StreamCfg {
    static constexpr bool kUseMma = MB > 4;
    static constexpr int kRows = MB;
    static constexpr int kStages = 8;
    // Consumer warps: a channel quarter each, kPhases warps per quarter taking the k blocks in turn. A third
    // warp per quarter measured slower with 16 rows (7.6 / 11.4 / 13.6 -> 8.5 / 12.0 / 14.4 us on the 13B
    // shapes) although a warp holds a block for 600-700 cycles there: the stream slows with the amount of
    // consumer work in flight, not with the time a block waits (with the consumers' arithmetic taken out the
    // same launches take 6.6 / 9.1 / 10.1 us, and the ring is never full either way).
    static constexpr int kPhases = 2;
    // Two CTAs per SM for both routes. Three single-row CTAs would fit (with 128-byte instead of 1024-byte
    // alignment slack), so that under the stable-weights promise the next launch's CTAs sit, fetching, beside
    // two CTAs of this one; measured slower (M = 1 layer 5.8 / 9.1 / 9.7 -> 6.6 / 9.7 / 11.8 us): what the
    // early CTAs fetch is taken from the grid that has to finish first.
    static constexpr int kConsumerWarps = 4 * kPhases;
    static constexpr int kThreads = (1 + kConsumerWarps) * 32;
};

// this CTA's sums over its k range (per-group scales: the bits of fp32 sums; rows padded by 8 words so that the MMA
// route's fragment owners, eight rows at the same columns, spread over the banks), and the other CTAs' sums for this
// CTA's channel slice, by sender: `split` slots of 128 / split channels, or (WIDE) slots of 32, of 64 where three CTAs share. (Without
// the slot of the CTA itself, which stays empty, every address takes a comparison of ranks: layers of 2 to 16 rows of
// 4096 x 4096 took 6.7-7.5 us instead of 6.5-7.3, 5120 x 5120 8.1-8.7 instead of 7.9-8.6.)
template <int MB, bool WIDE>
struct StreamSums {
    static constexpr int kSumStride = kTileN + 8;
    static constexpr int kRecvStride = WIDE ? 8 * 32 : kTileN;
    alignas(16) int sum[StreamCfg<MB>::kRows][kSumStride];
    alignas(16) int recv[StreamCfg<MB>::kRows][kRecvStride];
};
template <int MB, bool GROUPED, bool FUSEQ>
struct StreamRing {
    static constexpr int kStages = StreamCfg<MB>::kStages;
    // activation codes of the unit's k block; several rows quantized here: those of all of the CTA's k range
    alignas(1024) int8_t x[FUSEQ && MB > 1 ? 1 : kStages][FUSEQ && MB > 1 ? kSliceVecs * 8 * StreamCfg<MB>::kConsumerWarps * 32 : StreamCfg<MB>::kRows * kTileK];
    alignas(128) uint8_t w[kStages][kBlockBytes];          // packed weight block of the unit
    alignas(16) __half sc[GROUPED ? kStages : 1][kTileN];  // per-group scales: those of the unit's k block (= its group)
};
template <int MB, bool WIDE = false, bool GROUPED = false, bool FUSEQ = false>
struct StreamSmem {
    StreamRing<MB, GROUPED, FUSEQ> ring;
    StreamSums<MB, WIDE> sums;
    static constexpr int kStages = StreamCfg<MB>::kStages;
    static constexpr int kRecvStride = StreamSums<MB, WIDE>::kRecvStride;
    // one row quantized by the kernel itself: the codes of this CTA's k range (up to kFuseMaxBlocks blocks)
    alignas(16) int8_t xq[MB == 1 ? kFuseMaxBlocks * kTileK : 16];
    unsigned int warp_max[StreamCfg<MB>::kThreads / 32];
    unsigned int seen[FUSEQ && MB > 1 ? 8 * StreamCfg<MB>::kConsumerWarps : 1];       // several rows: what the warps of the cluster's CTAs saw of X
    alignas(8) uint64_t full[kStages];
    uint64_t empty[kStages];
    uint64_t got;                          // the other CTAs' sums are there
    uint64_t met;                          // all of `seen` is there
    volatile uint32_t abort_flag;
};
struct StreamParams {
    int M, K, N, Npad;
    const int8_t* q;
    const uint8_t* w_packed;
    const __half* w_scales;
    const int32_t* scale_exp;
    __half* y;
    int32_t* acc_dump;
    Control* ctl;
    const float* chan_offset;
    int zp_mid;
    int8_t* q_next;
    float next_inv, next_lo, next_hi;
    int clear_status;
    int early_weights;             // the first ring of weight copies may be issued before the wait for the kernel ahead
    int early_dependents;          // the launch behind this one may be set up from this kernel's start
    int next_packed;
    int box_rows;                  // MMA route: rows of a k block's codes in shared memory
    // FUSEQ: the activations themselves; the kernel finds the layer scale (and zero point), writes the codes of
    // its k range to shared memory (and, from the first channel tile, to q_out) and fills the control block
    const __half* x_row;           // the rows, K halves each
    const int32_t* row_idx;        // one row: NULL or its index, the row is x_row + row_idx[0] * K
    int8_t* q_out;                 // [M][K] codes
    int bits, scale_mode, clip_shift_or_exp;
    const uint8_t* alpha;          // NULL or the TRIP factors, K bytes, none above k_max
    int k_max;
};

// grid = (split, channel tiles), cluster = (split, 1, 1): the CTAs of a cluster share a channel
// tile and take consecutive k ranges; CTA r adds up and writes its slice of the tile's channels:
// [r, r+1) * 128 / split for split 1, 2, 4; WIDE (split 3, 5 to 8) the groups of four channels [32 r / split, 32 (r + 1) / split).
//
// GROUPED (one scale per 128 k): a k block is one group, so a block's integer sums are scaled and added in fp32 as
// soon as the block is done, by the warp that made them; what the warps, and the CTAs of the cluster, then add up
// are fp32 sums (in an order that does not depend on timing). The block's 128 scales ride along in the ring. The
// per-block cost is one conversion and one FMA per accumulator and a half-word read per channel, on top of a kernel
// whose consumers wait for memory most of the time; the kernel it replaced here (32 channels per CTA,
// every lane reading every activation byte) took 9.5 us at M = 1 and 30 us at M = 6 on K = N = 4096. The seven layers of
// a 4096 / 11008 block, quantization included, in graph replay: 116 -> 42 us at M = 1, 283 -> 65 us at M = 6.
template <bool GROUPED>
__device__ __forceinline__ int add_sums(int a, int b) {
    return GROUPED ? __float_as_int(__int_as_float(a) + __int_as_float(b)) : a + b;
}

// The codes of this CTA's k range, from X itself; the layer's exponent and zero point. The consumer warps call this. A step takes
// kTileN * 2 vectors of eight elements, one a thread: the rows side by side, each in runs of 16 / (rows rounded up to a power of two)
// k blocks, so that a step's places, in X and in the codes, lie a fixed distance behind the step's before it. HELD: steps (vectors a
// thread holds).
__host__ __device__ inline int slice_row_log(int M) {
    int log = 0;
    while ((1 << log) < M) ++log;
    return log;
}
template <int MB, bool WIDE, bool GROUPED, int HELD>
__device__ __forceinline__ void slice_codes(const StreamParams& p, StreamSmem<MB, WIDE, GROUPED, true>& sm, int8_t* x_tile, int kb0, int per_row,
                                            int row_log, int rank, int split, int tile, int& e_out, int& zp_out) {
    constexpr int kThreads = StreamCfg<MB>::kConsumerWarps * 32, kWarps = kThreads / 32;
    const int tid = (int)threadIdx.x - 32, warp = tid >> 5, lane = tid & 31;
    const int wide = kThreads >> row_log;                        // vectors of a row in a step
    const int m = tid >> (8 - row_log), c = tid & (wide - 1);
    static_assert(kThreads == 256, "the shifts above");
    const int left = m < p.M ? per_row - c : 0;                  // of this thread's row, from its first vector on
    const uint4* const x = reinterpret_cast<const uint4*>(p.x_row) + (size_t)m * (p.K / 8) + kb0 * (kTileK / 8) + c;
    uint4 held[HELD];
#pragma unroll
    for (int i = 0; i < HELD; ++i) {
        held[i] = make_uint4(0u, 0u, 0u, 0u);
        if (i * wide < left) held[i] = __ldg(x + i * wide);
    }
    const bool asym = p.chan_offset != nullptr;
    __half2 hi2 = __float2half2_rn(0.0f), lo2 = hi2;             // absent vectors are zero; a zero point's range contains it anyway
    if (asym) {
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            const __half2* h = reinterpret_cast<const __half2*>(&held[i]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {                        // NaN operands are dropped
                lo2 = __hmin2(lo2, h[k]);
                hi2 = __hmax2(hi2, h[k]);
            }
        }
        lo2 = __habs2(lo2);
    } else {
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            const __half2* h = reinterpret_cast<const __half2*>(&held[i]);
#pragma unroll
            for (int k = 0; k < 4; ++k) hi2 = __hmax2(hi2, __habs2(h[k]));
        }
    }
    const unsigned int bmax = max((unsigned int)__half_as_ushort(__low2half(hi2)), (unsigned int)__half_as_ushort(__high2half(hi2)));
    const unsigned int bmin = max((unsigned int)__half_as_ushort(__low2half(lo2)), (unsigned int)__half_as_ushort(__high2half(lo2)));
    unsigned int seen = __reduce_max_sync(0xFFFFFFFFu, bmax) | (asym ? __reduce_max_sync(0xFFFFFFFFu, bmin) << 16 : 0u);
    if (split > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");        // everybody has started
    if (lane < split) {
        uint32_t slot, bar;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(slot) : "r"(s_u32(&sm.seen[rank * kWarps + warp])), "r"(lane));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(s_u32(&sm.met)), "r"(lane));
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(slot), "r"(seen), "r"(bar) : "memory");
    }
    __syncwarp();
    str_wait_peers(&sm.met, &sm.abort_flag);
    __syncwarp();
    seen = 0;
    for (int i = lane; i < split * kWarps; i += 32) seen = __vmaxu2(seen, sm.seen[i]);
    seen = __reduce_max_sync(0xFFFFFFFFu, seen & 0xFFFFu) | (asym ? __reduce_max_sync(0xFFFFFFFFu, seen >> 16) << 16 : 0u);
    int e = p.clip_shift_or_exp, zp = 0;
    if (asym) zero_point_scale(seen & 0xFFFFu, seen >> 16, p.bits, e, zp);
    else if (p.scale_mode == AQ_SCALE_DYNAMIC) e = layer_exponent_from_bits(seen, p.bits) - p.clip_shift_or_exp - p.k_max;
    if (tile == 0 && rank == 0) {
        if (tid == 0) {
            p.ctl->scale_exp = e;
            p.ctl->zero_point = zp;
            p.ctl->absmax_bits = asym ? 0u : seen;
        }
        if (tid < Control::kSplitWords) p.ctl->split_flags[tid] = 0;
    }
    e_out = e;
    zp_out = zp;
    // rows of 128 bytes by k block, 16-byte chunks swizzled by row % 8 as a tensor-map copy leaves them
    int8_t* const at = x_tile + ((c >> 4) * p.box_rows + m) * kTileK + ((((c & 15) >> 1) ^ (m & 7)) << 4) + 8 * (c & 1);
    const int step = (wide >> 4) * p.box_rows * kTileK;
    int8_t* const q = p.q_out + (size_t)m * p.K + kb0 * kTileK + 8 * c;
    const int top = 1 << (p.bits - 1);
    if (!p.alpha && e >= -14 && e <= 14) {                       // 2^-e is a normal half: codes in half2 arithmetic
        // without a zero point: the same with a shift of zero
        const __half2 inv2 = __float2half2_rn(__int_as_float((127 - e) << 23));
        const __half2 clo2 = __float2half2_rn((float)(asym ? -zp : -top)), chi2 = __float2half2_rn((float)(asym ? 2 * top - 1 - zp : top - 1));
        const __half2 shift2 = __float2half2_rn((float)(asym ? zp - top : 0));
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            if (i * wide < left) {
                uint2 code;
                quantize8_half2_asym(held[i], inv2, clo2, chi2, shift2, code.x, code.y);
                *reinterpret_cast<uint2*>(at + i * step) = code;
                if (tile == 0) *reinterpret_cast<uint2*>(q + i * wide * 8) = code;
            }
        }
        return;
    }
    if (p.alpha && p.bits == 4 && e >= -14 && e <= 10) {         // so is 2^-(e + alpha), alpha <= 4
        const uint2* const al = reinterpret_cast<const uint2*>(p.alpha) + kb0 * (kTileK / 8) + c;
        uint2 a[HELD];
#pragma unroll
        for (int i = 0; i < HELD; ++i)
            if (i * wide < left) a[i] = __ldg(al + i * wide);
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            if (i * wide < left) {
                uint2 code;
                quantize8_half2_trip(held[i], e, a[i], code.x, code.y);
                *reinterpret_cast<uint2*>(at + i * step) = code;
                if (tile == 0) *reinterpret_cast<uint2*>(q + i * wide * 8) = code;
            }
        }
        return;
    }
    // The other exponents: X is read again, in a loop that is not unrolled (unrolled with all quantizers in it the code
    // was longer than the instruction cache holds: 16 x 13824 x 5120 28 us instead of 20)
#pragma unroll 1
    for (int i = 0; i * wide < left; ++i) {
        const uint4 d = __ldg(x + i * wide);
        uint2 code;
        if (asym) {
            code = quantize8_fp32_asym(d, __int_as_float((127 - e) << 23), zp, p.bits);
        } else if (p.alpha) {
            const uint2 al = __ldg(reinterpret_cast<const uint2*>(p.alpha) + kb0 * (kTileK / 8) + c + i * wide);
            code = quantize8_fp32(d, e, -(float)top, (float)(top - 1), &al);
        } else {
            code = quantize8_fp32(d, e, -(float)top, (float)(top - 1), nullptr);
        }
        *reinterpret_cast<uint2*>(at + i * step) = code;
        if (tile == 0) *reinterpret_cast<uint2*>(q + i * wide * 8) = code;
    }
}

// PLAIN: neither a zero point nor TRIP factors where one row is quantized here. (A parameter, so that the kernel of plain rows has none of the other
// quantizers in it; slices of several rows choose at run time.)
template <int MB, bool FUSEQ = false, bool WIDE = false, bool GROUPED = false, bool PLAIN = true>
__global__ void __launch_bounds__(StreamCfg<MB>::kThreads, 2)
gemm_decode_stream_kernel(const __grid_constant__ CUtensorMap x_map, const StreamParams p) {
    extern __shared__ uint8_t smem_raw[];
    using Smem = StreamSmem<MB, WIDE, GROUPED, FUSEQ>;
    constexpr bool kSlices = FUSEQ && MB > 1;
    Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr bool kUseMma = StreamCfg<MB>::kUseMma;
    constexpr int kRows = StreamCfg<MB>::kRows;
    constexpr int kStrStages = StreamCfg<MB>::kStages;
    constexpr int kPhases = StreamCfg<MB>::kPhases;
    constexpr int kStrConsumerWarps = StreamCfg<MB>::kConsumerWarps;
    constexpr int kStrThreads = StreamCfg<MB>::kThreads;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int KB = k_blocks(p.K);
    const int rank = blockIdx.x, split = gridDim.x;
    const int tile = blockIdx.y;
    const int kb0 = (int)((long long)KB * rank / split), kb1 = (int)((long long)KB * (rank + 1) / split);

    int8_t* const x_tile = sm.ring.x[0];                     // FUSEQ: codes of the k range

    // Channel slices: CTA r finishes channels [r, r + 1) * 128 / split for split 1, 2, 4 (divisions are shifts); WIDE: the groups of four
    // channels [32 r / split, 32 (r + 1) / split), at most 28 channels.
    const int g_first = (32 * rank) / split, g_count = (32 * (rank + 1)) / split - g_first;
    if (threadIdx.x == 0) {
        if constexpr (kRows > 1 && !FUSEQ)     // start the descriptor's fetch now; the first tile load would wait for it
            asm volatile("prefetch.tensormap [%0];" ::"l"(&x_map) : "memory");
        for (int s = 0; s < kStrStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_u32(&sm.full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_u32(&sm.empty[s])), "r"(4) : "memory");   // the four quarter warps of the block's phase
        }
        sm.abort_flag = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_u32(&sm.got)) : "memory");
        if constexpr (kSlices) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_u32(&sm.met)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (split > 1)            // this CTA's channels of every row from each of the others
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                         ::"r"(s_u32(&sm.got)), "r"((uint32_t)((split - 1) * min(p.M, kRows) * g_count * 16)) : "memory");
        if constexpr (kSlices)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_u32(&sm.met)), "r"((uint32_t)(split * kStrConsumerWarps * 4)) : "memory");
    }
    if (split > 1) {
        __syncwarp();
        // Meeting of the cluster, arrival only: by the time a CTA writes into another's shared memory (after its k range; by slices
        // before it) every CTA of the cluster has started and its barriers are set up. The wait comes just before those writes.
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    }
    __syncthreads();
    volatile uint32_t* abort_flag = &sm.abort_flag;
    const uint8_t* wsrc = p.w_packed + (size_t)tile * KB * kBlockBytes;

    // a stage's barrier expects the weight block and the activation codes; the two copies may be issued apart
    // One row is fetched with a plain copy, which must stay inside the row: of a last block that K does
    // not fill, only the codes that exist are copied (a multiple of 32 bytes); the rest of the stage keeps
    // stale bytes, which meet zero weight codes. Tensor-map loads count their whole box.
    auto x_bytes = [&](int kb) -> uint32_t {
        if (FUSEQ) return 0u;                          // the codes are made here, not copied
        return kRows == 1 ? (uint32_t)min(kTileK, p.K - kb * kTileK)
                          : (uint32_t)(p.box_rows * kTileK);
    };
    auto issue_w = [&](int kb, int s) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     ::"r"(s_u32(&sm.full[s])), "r"((uint32_t)kBlockBytes + (GROUPED ? kTileN * 2u : 0u) + x_bytes(kb)) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(s_u32(sm.ring.w[s])), "l"(wsrc + (size_t)kb * kBlockBytes), "r"((uint32_t)kBlockBytes),
                       "r"(s_u32(&sm.full[s])) : "memory");
        if constexpr (GROUPED)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(s_u32(sm.ring.sc[s])), "l"(p.w_scales + (size_t)kb * p.Npad + tile * kTileN),
                           "r"((uint32_t)(kTileN * 2)), "r"(s_u32(&sm.full[s])) : "memory");
    };
    auto issue_x = [&](int kb, int s) {
        if constexpr (FUSEQ) {
        } else if constexpr (kRows == 1) {
            // one row: its 128 codes are contiguous, a plain bulk copy needs no tensor-map fetch
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(s_u32(sm.ring.x[s])), "l"(p.q + (size_t)kb * kTileK), "r"(x_bytes(kb)),
                           "r"(s_u32(&sm.full[s])) : "memory");
        } else {
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                ::"r"(s_u32(sm.ring.x[s])), "l"(&x_map), "r"(kb * kTileK), "r"(0), "r"(s_u32(&sm.full[s])) : "memory");
        }
    };
    // The weights do not depend on the kernel before this one: the first ring of weight blocks is on its
    // way before this grid waits for that kernel (a no-op unless the launch allowed the overlap), and only
    // then are the status word, the codes, the exponent and the offsets touched.
    // Launched with programmatic stream serialization: this grid may have been set up while the kernel
    // before it on the stream still ran. Nothing written before this launch is read, and nothing is written,
    // until that kernel has completed; only behind the call's own quantize kernel (which allows this
    // launch only once everything before it, weight packing included, has completed), or on the caller's
    // promise that nothing in flight writes the weights, the weights are fetched first. With that promise
    // the launch behind this one is also allowed from the start, so that its CTAs take the places of this
    // grid's CTAs as they leave and have their first ring on the way while this grid finishes.
    // The producer is one elected thread of warp 0 (a block per about 250 cycles; behind `lane == 0` about 500, which two lanes
    // in lockstep had halved for the single-row kernel). M = 1 layers on 5120 x 5120 / 13824 x 5120 (K x N) 6.9 / 10.6 ->
    // 6.4 / 10.2 us, M = 16 on 3072 x 768 6.4 -> 6.3 us.
    const int ring = min(kStrStages, kb1 - kb0);      // blocks of the first ring
    int issued = 0;
    if (p.early_dependents) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (p.early_weights) {     // behind this call's own quantize kernel, or the caller has promised stable weights
        if (warp == 0 && s_elect_one())
            for (int i = 0; i < ring; ++i) issue_w(kb0 + i, i);
        issued = ring;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.clear_status && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) p.ctl->status = 0;   // nothing has given up yet
    [[maybe_unused]] int fused_exp = 0, fused_zp = 0;
    if constexpr (kSlices) {
        // ---- several rows, by slices: a CTA reads its k range of every row, once, into registers; its warps tell every CTA of the
        // cluster the largest magnitudes they saw (asynchronous remote stores that count on the receiver's barrier), and each warp,
        // with all of them, derives the scale and quantizes what it holds.
        if (warp == 0 && s_elect_one())
            for (int i = issued; i < ring; ++i) issue_w(kb0 + i, i);   // weights on their way meanwhile
        issued = ring;
        __syncwarp();
        if (warp > 0) {
            const int per_row = min(kb1 * (kTileK / 8), p.K / 8) - kb0 * (kTileK / 8);       // vectors of eight elements of the k range
            const int row_log = slice_row_log(p.M);
            constexpr int kFewVecs = 4;                                 // unrolled loops over what is not there cost their instructions all the same
            if ((per_row << row_log) <= kFewVecs * 256) slice_codes<MB, WIDE, GROUPED, kFewVecs>(p, sm, x_tile, kb0, per_row, row_log, rank, split, tile, fused_exp, fused_zp);
            else slice_codes<MB, WIDE, GROUPED, kSliceVecs>(p, sm, x_tile, kb0, per_row, row_log, rank, split, tile, fused_exp, fused_zp);
            asm volatile("bar.sync 1, %0;" ::"n"(kStrConsumerWarps * 32) : "memory");
        } else if (split > 1) {
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
    }
    if constexpr (FUSEQ && MB == 1) {
        // ---- the layer scale and this CTA's codes (Eq. 1, Eq. 2 / Eq. 5 with zp = 0; one scale for the layer)
        if (warp == 0 && s_elect_one())
            for (int i = issued; i < ring; ++i) issue_w(kb0 + i, i);   // weights on their way meanwhile
        issued = ring;
        const uint4* xv = reinterpret_cast<const uint4*>(p.x_row + (p.row_idx ? (size_t)p.row_idx[0] * p.K : 0));
        int e = p.clip_shift_or_exp, zp = 0;
        const bool asym = !PLAIN && p.chan_offset != nullptr;
        const int v0 = kb0 * (kTileK / 8), v1 = min(kb1 * (kTileK / 8), p.K / 8);       // 8-element vectors of this k range
        [[maybe_unused]] uint2 alpha_first = make_uint2(0u, 0u);                        // of this thread's first one, on its way meanwhile
        if constexpr (!PLAIN)
            if (p.alpha && v0 + (int)threadIdx.x < v1) alpha_first = __ldg(reinterpret_cast<const uint2*>(p.alpha) + v0 + threadIdx.x);
        // up to kKeep vectors per thread stay in registers between the two passes (K <= 18432); longer rows
        // are read again (from L2) for the codes
        constexpr int kKeep = 8;
        uint4 keep[kKeep];
        const int n_vec = p.K / 8;
        const bool kept = n_vec <= kKeep * kStrThreads;
        if (asym || p.scale_mode == AQ_SCALE_DYNAMIC || kept) {
            __half2 m2 = __float2half2_rn(0.0f), least2 = m2;
            auto take = [&](const uint4& d) {                              // NaN operands are dropped
                const __half2* h = reinterpret_cast<const __half2*>(&d);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (asym) least2 = __hmin2(least2, h[k]);
                    m2 = __hmax2(m2, asym ? h[k] : __habs2(h[k]));
                }
            };
            if (kept) {
#pragma unroll
                for (int i = 0; i < kKeep; ++i) {
                    const int v = (int)threadIdx.x + i * kStrThreads;
                    keep[i] = v < n_vec ? __ldg(xv + v) : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int i = 0; i < kKeep; ++i) take(keep[i]);
            } else {
                for (int v = (int)threadIdx.x; v < n_vec; v += kStrThreads) take(__ldg(xv + v));
            }
            unsigned int bmax = max((unsigned int)__half_as_ushort(__low2half(m2)), (unsigned int)__half_as_ushort(__high2half(m2)));
            if (bmax > 0x7C00u) bmax = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) bmax = max(bmax, __shfl_xor_sync(0xFFFFFFFFu, bmax, o));
            if (asym) {                                                    // the least value's magnitude in the upper half
                const __half2 n2 = __habs2(least2);
                bmax |= __reduce_max_sync(0xFFFFFFFFu, max((unsigned int)__half_as_ushort(__low2half(n2)), (unsigned int)__half_as_ushort(__high2half(n2)))) << 16;
            }
            if (lane == 0) sm.warp_max[warp] = bmax;
            __syncthreads();
            unsigned int all = 0;
#pragma unroll
            for (int w = 0; w < kStrThreads / 32; ++w) all = PLAIN ? max(all, sm.warp_max[w]) : __vmaxu2(all, sm.warp_max[w]);
            if (asym) {
                zero_point_scale(all & 0xFFFFu, all >> 16, p.bits, e, zp);
                all = 0u;
            } else if (p.scale_mode == AQ_SCALE_DYNAMIC) {
                e = layer_exponent_from_bits(all, p.bits) - p.clip_shift_or_exp - (PLAIN ? 0 : p.k_max);
            }
            if ((asym || p.scale_mode == AQ_SCALE_DYNAMIC) && tile == 0 && rank == 0 && threadIdx.x == 0) p.ctl->absmax_bits = all;
        }
        if (tile == 0 && rank == 0) {
            if (threadIdx.x == 0) {
                p.ctl->scale_exp = e;
                p.ctl->status = 0;
                if (!PLAIN) p.ctl->zero_point = zp;
            }
            if (threadIdx.x < Control::kSplitWords) p.ctl->split_flags[threadIdx.x] = 0;
        }
        const float lo = -(float)(1 << (p.bits - 1)), hi = (float)((1 << (p.bits - 1)) - 1);
        const bool fast = e >= -14 && e <= 14;             // 2^-e is a normal half: codes in half2 arithmetic
        const __half2 inv2 = __float2half2_rn(fast ? __int_as_float((127 - e) << 23) : 1.0f);
        const __half2 lo2 = __float2half2_rn(lo), hi2 = __float2half2_rn(hi);
        auto code8 = [&](const uint4& d, int v) {
            uint2 c;
            if constexpr (!PLAIN) {
                if (asym) {
                    if (fast) {
                        const __half2 clo2 = __float2half2_rn(-(float)zp), chi2 = __float2half2_rn((float)((1 << p.bits) - 1 - zp));
                        quantize8_half2_asym(d, inv2, clo2, chi2, __float2half2_rn((float)(zp - (1 << (p.bits - 1)))), c.x, c.y);
                    } else {
                        c = quantize8_fp32_asym(d, __int_as_float((127 - e) << 23), zp, p.bits);
                    }
                } else {
                    const uint2 al = v == v0 + (int)threadIdx.x ? alpha_first : __ldg(reinterpret_cast<const uint2*>(p.alpha) + v);
                    if (p.bits == 4 && e >= -14 && e <= 10) quantize8_half2_trip(d, e, al, c.x, c.y);      // 2^-(e + alpha) is a normal half, alpha <= 4
                    else c = quantize8_fp32(d, e, lo, hi, &al);
                }
            } else if (fast) {
                quantize8_half2(d, inv2, lo2, hi2, c.x, c.y);
            } else {
                c = quantize8_fp32(d, e, lo, hi, nullptr);
            }
            reinterpret_cast<uint2*>(sm.xq)[v - v0] = c;
            if (tile == 0) reinterpret_cast<uint2*>(p.q_out)[v] = c;
        };
        if (PLAIN && kept) {
#pragma unroll
            for (int i = 0; i < kKeep; ++i) {
                const int v = (int)threadIdx.x + i * kStrThreads;
                if (v >= v0 && v < v1) code8(keep[i], v);
            }
        } else {
            // (not PLAIN: once or a few times for a thread, unrolled eight times the quantizers' code would be the longer part)
#pragma unroll 1
            for (int v = v0 + (int)threadIdx.x; v < v1; v += kStrThreads) code8(__ldg(xv + v), v);
        }
        fused_exp = e;
        fused_zp = zp;
        __syncthreads();
    }
    if (warp == 0) {
        if (s_elect_one()) {
            for (int i = 0; i < issued; ++i) issue_x(kb0 + i, i);
            for (int kb = kb0 + issued; kb < kb1; ++kb) {
                const uint32_t i = (uint32_t)(kb - kb0);
                const int s = (int)(i % kStrStages);
                if (!str_wait(&sm.empty[s], ((i / kStrStages) & 1u) ^ 1u, abort_flag)) break;
                issue_w(kb, s);
                issue_x(kb, s);
            }
        }
    } else {
        const int cw = warp - 1;
        const int quarter = cw & 3, phase = cw >> 2;
        if constexpr (!kUseMma) {
            // A lane takes one 32-k chunk of the block (t = lane / 8) and eight channels per pass (g = lane % 8,
            // four passes cover the warp's 32 channels): per block it reads four 16-byte weight units (chunk t
            // of channels 8i + g; the eight lanes of a quarter warp read eight consecutive units) and the 32
            // activation bytes of its chunk, six 16-byte shared-memory loads where one lane per channel, every
            // lane reading every activation byte, took twelve. The sum over k does not care which lane adds
            // which k; the lanes' partial sums meet once, after the k range.
            const int g = lane & 7, t = lane >> 3;
            int acc[MB][4];                                          // per-group scales: the bits of fp32 sums
#pragma unroll
            for (int m = 0; m < MB; ++m)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[m][i] = 0;
            for (int kb = kb0 + phase; kb < kb1; kb += kPhases) {       // the warps of a quarter take the k blocks in turn
                const uint32_t it = (uint32_t)(kb - kb0);
                const int s = (int)(it % kStrStages);
                if (!__all_sync(0xFFFFFFFFu, str_wait(&sm.full[s], (it / kStrStages) & 1u, abort_flag) ? 1 : 0)) break;
                uint4 wv[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    wv[i] = reinterpret_cast<const uint4*>(sm.ring.w[s])[t * kTileN + quarter * 32 + 8 * i + g];
#pragma unroll
                for (int m = 0; m < MB; ++m) {
                    const uint4* xp = FUSEQ ? reinterpret_cast<const uint4*>(sm.xq + (size_t)(kb - kb0) * kTileK + 32 * t)
                                            : reinterpret_cast<const uint4*>(sm.ring.x[s] + m * kTileK + 32 * t);
                    const uint4 x0 = xp[0], x1 = xp[1];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // word u of a unit: k 8u..8u+3 of the chunk in its low nibbles, k 8u+4..8u+7 in its high ones
                        const uint32_t w[4] = {wv[i].x, wv[i].y, wv[i].z, wv[i].w};
                        int a = GROUPED ? 0 : acc[m][i];
                        a = __dp4a((int)((w[0] << 4) & 0xF0F0F0F0u), (int)x0.x, a);      // 16*code
                        a = __dp4a((int)(w[0] & 0xF0F0F0F0u), (int)x0.y, a);
                        a = __dp4a((int)((w[1] << 4) & 0xF0F0F0F0u), (int)x0.z, a);
                        a = __dp4a((int)(w[1] & 0xF0F0F0F0u), (int)x0.w, a);
                        a = __dp4a((int)((w[2] << 4) & 0xF0F0F0F0u), (int)x1.x, a);
                        a = __dp4a((int)(w[2] & 0xF0F0F0F0u), (int)x1.y, a);
                        a = __dp4a((int)((w[3] << 4) & 0xF0F0F0F0u), (int)x1.z, a);
                        a = __dp4a((int)(w[3] & 0xF0F0F0F0u), (int)x1.w, a);
                        if constexpr (GROUPED)
                            acc[m][i] = __float_as_int(fmaf((float)a, __half2float(sm.ring.sc[s][quarter * 32 + 8 * i + g]),
                                                            __int_as_float(acc[m][i])));
                        else
                            acc[m][i] = a;
                    }
                }
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s_u32(&sm.empty[s])) : "memory");
            }
            // the four chunks of a channel meet (two exchange steps), then lane (g, t) keeps pass t's channel
            // 8t + g; the warps of a quarter meet in the sum buffer, one after the other (the same thread
            // position owns an element in each of them: the first stores, the others add)
            int mine[MB];
#pragma unroll
            for (int m = 0; m < MB; ++m) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[m][i] = add_sums<GROUPED>(acc[m][i], __shfl_xor_sync(0xFFFFFFFFu, acc[m][i], 8));
                    acc[m][i] = add_sums<GROUPED>(acc[m][i], __shfl_xor_sync(0xFFFFFFFFu, acc[m][i], 16));
                }
                mine[m] = t == 0 ? acc[m][0] : t == 1 ? acc[m][1] : t == 2 ? acc[m][2] : acc[m][3];
            }
            const int r = quarter * 32 + 8 * t + g;                  // channel inside the tile
#pragma unroll
            for (int ph = 0; ph < kPhases; ++ph) {
                if (ph > 0) asm volatile("bar.sync 1, %0;" ::"n"(kStrConsumerWarps * 32) : "memory");
                if (phase == ph) {
#pragma unroll
                    for (int m = 0; m < MB; ++m) {
                        if (ph == 0) sm.sums.sum[m][r] = mine[m];
                        else sm.sums.sum[m][r] = add_sums<GROUPED>(sm.sums.sum[m][r], mine[m]);
                    }
                }
            }
        } else {
            // Warp-level int8 MMA, D[16 channels x 8 rows] += A[16 x 32 k] * B[32 k x 8 rows]: the weights are A, so that up to eight
            // rows cost half the instructions that sixteen do (with the rows as A, rows 8..15 of zeros cost as much as others: this instruction
            // takes 8.6 cycles of a scheduler's tensor pipe whatever it is fed; 6 x 4096 x 11008 10.55 / 8.79, 3 x 7168 x 28672 21.2 / 19.6 us).
            // Fragment owner: g = lane / 4 (channels g and g+8 of A and D; row g of B), t = lane % 4 (k bytes 4t..4t+3 and
            // 16+4t..; D rows 2t, 2t+1).
            // (Splitting a block among the four warps of a phase into channel halves x k halves instead of channel quarters, so that a
            // warp reads half of the activation tile, measured the same within 0.2 us either way.)
            const int g = lane >> 2, t = lane & 3;
            const bool upper = p.M > 8;
            // [u][h][c]: channel 16u + 8(c / 2) + g, row 8h + 2t + c % 2
            int acc[2][2][4];
            [[maybe_unused]] float fsum[2][2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    acc[u][c >> 2][c & 3] = 0;
                    if constexpr (GROUPED) fsum[u][c >> 2][c & 3] = 0.0f;
                }
            for (int kb = kb0 + phase; kb < kb1; kb += kPhases) {
                const uint32_t it = (uint32_t)(kb - kb0);
                const int s = (int)(it % kStrStages);
                if (!__all_sync(0xFFFFFFFFu, str_wait(&sm.full[s], (it / kStrStages) & 1u, abort_flag) ? 1 : 0)) break;
                const int8_t* xt = FUSEQ ? x_tile + (kb - kb0) * p.box_rows * kTileK : sm.ring.x[s];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // The sum over k does not depend on which k sits in which slot of the instruction, as long
                    // as both operands agree: lane t feeds its slots "k 4t.." and "k 16+4t.." with the k range
                    // 8t..8t+3 and 8t+4..8t+7 of this 32-k chunk, i.e. with the two nibble planes of ONE packed
                    // word and eight consecutive activation bytes (one 8-byte load per row).
                    // activation rows: 128 bytes, 16-byte chunks XOR-swizzled by row % 8
                    const int x_off = (((2 * j + (t >> 1)) ^ g) << 4) + 8 * (t & 1);
                    // Weight fragments of the four channel passes in one instruction: the 32 units (16 bytes each)
                    // of this chunk and channel quarter are four 8 x 8 matrices of 16-bit elements, one per pass;
                    // lane l gives the address of unit l, and lane (g, t) receives word t of channel 8i + g for
                    // i = 0..3, which holds k 8t..8t+3 in its low nibbles and k 8t+4..8t+7 in its high nibbles.
                    uint32_t pw[4];
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(pw[0]), "=r"(pw[1]), "=r"(pw[2]), "=r"(pw[3])
                                 : "r"(s_u32(sm.ring.w[s] + (size_t)(j * kTileN + quarter * 32 + lane) * 16)) : "memory");
                    const uint2 xa = *reinterpret_cast<const uint2*>(xt + g * kTileK + x_off);
                    uint2 xb;
                    if (upper) xb = *reinterpret_cast<const uint2*>(xt + (g + 8) * kTileK + x_off);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const uint32_t a0 = (pw[2 * u] << 4) & 0xF0F0F0F0u, a2 = pw[2 * u] & 0xF0F0F0F0u;
                        const uint32_t a1 = (pw[2 * u + 1] << 4) & 0xF0F0F0F0u, a3 = pw[2 * u + 1] & 0xF0F0F0F0u;
                        auto mma = [&](int (&d)[4], const uint2& b) {
                            asm volatile(
                                "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
                                "{%8, %9}, {%0, %1, %2, %3};"
                                : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                                : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
                        };
                        mma(acc[u][0], xa);
                        if (upper) mma(acc[u][1], xb);
                    }
                }
                if constexpr (GROUPED) {
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const __half* sc = &sm.ring.sc[s][quarter * 32 + 16 * u + g];
                        const float s0 = __half2float(sc[0]), s1 = __half2float(sc[8]);
                        auto scale = [&](int (&a)[4], float (&f)[4]) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                f[c] = fmaf((float)a[c], c < 2 ? s0 : s1, f[c]);
                                a[c] = 0;
                            }
                        };
                        scale(acc[u][0], fsum[u][0]);
                        if (upper) scale(acc[u][1], fsum[u][1]);
                    }
                }
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s_u32(&sm.empty[s])) : "memory");
            }
            // The warps of a quarter meet in the sum buffer, one after the other (the same thread position
            // owns an element in each of them: the first stores, the others add).
#pragma unroll
            for (int ph = 0; ph < kPhases; ++ph) {
                if (ph > 0) asm volatile("bar.sync 1, %0;" ::"n"(kStrConsumerWarps * 32) : "memory");
                if (phase == ph) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 0 || upper) {
#pragma unroll
                            for (int u = 0; u < 2; ++u)
#pragma unroll
                                for (int c = 0; c < 4; ++c) {
                                    int& dst = sm.sums.sum[8 * h + 2 * t + (c & 1)][quarter * 32 + 16 * u + 8 * (c >> 1) + g];
                                    const int own = GROUPED ? __float_as_int(fsum[u][h][c]) : acc[u][h][c];
                                    if (ph == 0) dst = own;
                                    else dst = add_sums<GROUPED>(dst, own);
                                }
                        }
                    }
                }
            }
        }
    }
    // Every CTA of the cluster now holds the tile's sums over its own k range, and CTA `rank` finishes the
    // tile's channel slice `rank`: every CTA writes its sums of the other slices into their owners' shared memory (slot = sender) with
    // asynchronous stores that count on the owner's barrier, and every CTA, once all of its own are there, adds them
    // to its sums (integer addition is exact in any order), scales and writes its outputs. Nobody touches another CTA's memory after
    // that, so a CTA may leave as soon as it is done. (A meeting of the cluster behind plain remote stores, which this replaced, held
    // every launch 0.2-0.35 us longer: 1 x 5120 x 5120 5.42 / 5.27, 1 x 13824 x 5120 9.07 / 8.81, 6 x 4096 x 4096 6.77 / 6.40; reading the
    // other CTAs' sums over distributed shared memory, with a second meeting before anybody leaves, 0.1-0.5 us more.)
    // The scale is fetched before the wait for them so that its latency overlaps it.
    // This CTA's k range is done: a launch behind this one that allows it may be scheduled and set up now
    // (it reads and writes nothing before this grid has completed).
    if (!p.early_dependents) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // WIDE: a slice's channels (at most 28, or 44 of three CTAs) are handled by the first lanes of 32 or 64 threads.
    constexpr bool wide = WIDE;
    const int cw_log = wide ? (split == 3 ? 6 : 5) : 7 - (31 - __clz(split));
    const int cw = 1 << cw_log;                               // slot width in the receive buffer
    const int ft = (int)threadIdx.x - 32;                     // the consumer threads finish (a multiple of 128 = 4 cw at most)
    const int rc = ft & (cw - 1);                             // channel inside the slice (only used when ft >= 0)
    const int out_r = wide ? min(4 * g_first + rc, kTileN - 1) : rank * cw + rc;   // wide: lanes behind the slice only keep their warp whole
    const int out_n = tile * kTileN + out_r;
    const bool mine = ft >= 0 && out_n < p.N && (!wide || rc < 4 * g_count);
    float sc = 0.0f, off = 0.0f;
    if (mine) {
        const float pe = __int_as_float((127 + (FUSEQ ? fused_exp : *p.scale_exp)) << 23);
        sc = GROUPED ? 0.0625f * pe : __half2float(p.w_scales[out_n]) * pe;     // the fp32 sums carry a factor 16
        if (p.chan_offset) off = __fmul_rn(FUSEQ ? -(float)(fused_zp - p.zp_mid) : offset_factor(p.ctl, p.zp_mid), p.chan_offset[out_n]) * pe;
    }
    const int rows = p.M < kRows ? p.M : kRows;
    if (split > 1 && !kSlices) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // everybody has started (arrival at the top)
    if (ft >= 0) {
        asm volatile("bar.sync 1, %0;" ::"n"(kStrConsumerWarps * 32) : "memory");     // this CTA's sums are complete
        if (split > 1) {
            // four consecutive channels at a time (16-byte remote stores, counted by the receiver's barrier) go to the CTA that owns them
            for (int e = ft; e < rows * (kTileN / 4); e += kStrConsumerWarps * 32) {
                const int m = e >> 5, g4 = e & 31, ch = 4 * g4;
                const int owner = wide ? (((g4 + 1) * split + 31) >> 5) - 1 : ch >> cw_log;
                const int at = wide ? ch - 4 * ((32 * owner) / split) : ch & (cw - 1);   // place inside the owner's slice
                if (owner != rank) {
                    const int4 v = *reinterpret_cast<const int4*>(&sm.sums.sum[m][ch]);
                    uint32_t slot, bar;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(slot) : "r"(s_u32(&sm.sums.recv[m][rank * cw + at])), "r"(owner));
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(s_u32(&sm.got)), "r"(owner));
                    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                                 ::"r"(slot), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
                }
            }
            str_wait_peers(&sm.got, abort_flag);
            __syncwarp();
        }
    }
    if (mine || (wide && ft >= 0)) {
        // All shared-memory reads of this thread's outputs are issued before the first is used and without
        // branches around them (rows that do not exist read the last row of the buffer and are dropped):
        // taken one after the other, each behind its own test, they were the longest part of the finish at
        // 16 rows.
        constexpr int kPass = kStrConsumerWarps * 32 / (WIDE ? 64 : kTileN);     // rows that a pass covers at least
        constexpr int kIt = (kRows + kPass - 1) / kPass;
        const int stride = (kStrConsumerWarps * 32) >> cw_log, m0 = ft >> cw_log;
        int av[kIt];
#pragma unroll
        for (int i = 0; i < kIt; ++i) av[i] = i * stride < kRows ? sm.sums.sum[min(m0 + i * stride, kRows - 1)][out_r] : 0;
#pragma unroll
        for (int k = 1; k < (WIDE ? 8 : 4); ++k) {
            if (k < split) {
                int c = rank + k;                                             // the k-th other CTA's slot
                if (c >= split) c -= split;
                const int col = c * cw + rc;
#pragma unroll
                for (int i = 0; i < kIt; ++i)
                    if (i * stride < kRows)                               // the same test in every thread
                        av[i] = add_sums<GROUPED>(av[i], sm.sums.recv[min(m0 + i * stride, kRows - 1)][col]);
            }
        }
        auto value = [&](int a) { return GROUPED ? __int_as_float(a) : (float)(a >> 4); };     // integer sums carry a factor 16
        if (!p.acc_dump && !p.q_next) {
#pragma unroll
            for (int i = 0; i < kIt; ++i) {
                const int m = m0 + i * stride;
                const __half hv = __float2half_rn(fmaf(value(av[i]), sc, off));
                if (mine && m < rows) p.y[(size_t)m * p.N + out_n] = hv;
            }
        } else {
#pragma unroll
            for (int i = 0; i < kIt; ++i) {
                const int m = m0 + i * stride;
                if (m < rows) {
                    if (!GROUPED && p.acc_dump && mine) p.acc_dump[(size_t)m * p.N + out_n] = av[i] >> 4;
                    const __half hv = __float2half_rn(fmaf(value(av[i]), sc, off));
                    // (a warp's lanes hold consecutive channels, even lanes even channels, and run this loop together)
                    if (p.q_next)
                        store_next_code(p.q_next, (size_t)m * p.N + out_n, next_code(hv, p.next_inv, p.next_lo, p.next_hi),
                                        p.next_packed, mine, lane);
                    else if (mine) p.y[(size_t)m * p.N + out_n] = hv;
                }
            }
        }
    }
    if (sm.abort_flag) {
        for (int i = 0; i < 64; ++i) __nanosleep(1000);          // let copies in flight land
        if (threadIdx.x == 0) atomicOr(&p.ctl->status, 1u);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

template <int MB, bool FUSEQ, bool WIDE, bool GROUPED, bool PLAIN = true>
cudaError_t launch_stream(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream, int split) {
    using Smem = StreamSmem<MB, WIDE, GROUPED, FUSEQ>;
    const int tiles = round_up(a.N, kTileN) / kTileN;
    const size_t smem_bytes = sizeof(Smem) + 1024;
    static_assert(2 * (sizeof(Smem) + 1024 + 1024) <= 228 * 1024, "two CTAs an SM");
    static SmemOptIn opt_in;
    if (const cudaError_t e = opt_in.ensure(gemm_decode_stream_kernel<MB, FUSEQ, WIDE, GROUPED, PLAIN>, dev.device, smem_bytes); e != cudaSuccess)
        return e;
    CUtensorMap map = {};
    const cuuint64_t dims[2] = {(cuuint64_t)a.K, (cuuint64_t)a.M};
    const cuuint64_t strides[1] = {(cuuint64_t)a.K};
    // MMA route: 8 or 16 rows; rows 8..15 are neither copied nor read when M <= 8. Quantized here: 2 or 4 rows as well (what the
    // instruction then reads as rows up to 7 is the next block's, or whatever follows in the ring, and its sums are dropped)
    const int box_rows = !StreamCfg<MB>::kUseMma ? StreamCfg<MB>::kRows : FUSEQ ? 1 << slice_row_log(a.M) : round_up(a.M, 8);
    const cuuint32_t box[2] = {128u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    const CUresult r = FUSEQ ? CUDA_SUCCESS : reinterpret_cast<EncodeTiledFn>(dev.encode_tiled)(      // (FUSEQ: nothing is fetched through it)
        &map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t*>(a.q), dims, strides, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE,
        StreamCfg<MB>::kUseMma ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    StreamParams p;
    p.M = a.M; p.K = a.K; p.N = a.N; p.Npad = round_up(a.N, kTileN);
    p.q = a.q;
    p.clear_status = a.after_quantize ? 0 : 1;
    p.next_packed = a.next_packed ? 1 : 0;
    p.box_rows = box_rows;
    p.w_packed = a.w_packed; p.w_scales = a.w_scales; p.scale_exp = a.scale_exp;
    p.y = a.y; p.acc_dump = a.acc_dump; p.ctl = a.ctl; p.chan_offset = a.chan_offset; p.zp_mid = a.zp_mid;
    p.q_next = a.q_next;
    p.next_inv = ldexpf(1.0f, -a.next_exp);
    p.next_lo = -(float)(1 << (a.next_bits - 1));
    p.next_hi = (float)((1 << (a.next_bits - 1)) - 1);
    p.x_row = a.fuse_x; p.row_idx = a.fuse_row_idx; p.q_out = const_cast<int8_t*>(a.q);
    p.bits = a.fuse_bits; p.scale_mode = a.fuse_scale_mode; p.clip_shift_or_exp = a.fuse_clip_shift_or_exp;
    if (FUSEQ) p.clear_status = 1;       // no quantize kernel of this call runs ahead
    // Weights ahead of the wait: behind the call's own quantize kernel (which allows this launch only once
    // everything before it has completed), or on the caller's promise that nothing in flight writes them.
    p.early_weights = (!p.clear_status || a.weights_stable) ? 1 : 0;
    p.early_dependents = a.weights_stable ? 1 : 0;
    p.alpha = a.fuse_alpha; p.k_max = a.fuse_k_max;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(StreamCfg<MB>::kThreads);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(split, tiles, 1);
    attr[0].val.clusterDim.x = split;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;       // the kernel reads and writes nothing before the kernel ahead of it has completed
    return cudaLaunchKernelEx(&cfg, gemm_decode_stream_kernel<MB, FUSEQ, WIDE, GROUPED, PLAIN>, map, p);
}

// Clusters of `split` CTAs that run at once, by the occupancy query (asked once per device and size).
template <int MB, bool GROUPED>
int clusters_at_once(int split, const DeviceInfo& dev) {
    static std::atomic<int> fits[kMaxDevices][9];               // + 1 (0: not asked yet)
    int known = fits[dev.device][split].load(std::memory_order_relaxed);
    if (known == 0) {
        using Smem = StreamSmem<MB, true, GROUPED>;
        const size_t smem_bytes = sizeof(Smem) + 1024;
        static SmemOptIn opt_in;
        int n = 0;
        if (opt_in.ensure(gemm_decode_stream_kernel<MB, false, true, GROUPED>, dev.device, smem_bytes) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(split, dev.sm_count, 1);
            cfg.blockDim = dim3(StreamCfg<MB>::kThreads);
            cfg.dynamicSmemBytes = smem_bytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = split;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, gemm_decode_stream_kernel<MB, false, true, GROUPED>, &cfg) != cudaSuccess) {
                (void)cudaGetLastError();
                n = 0;
            }
        }
        known = n + 1;
        fits[dev.device][split].store(known, std::memory_order_relaxed);
    }
    return known - 1;
}

// CTAs that share a tile of 128 channels, each with its range of k blocks: the number that leaves a warp the fewest blocks to go through
// one after the other (two warps of a channel quarter take a CTA's blocks in turn), the smallest such. Only numbers whose clusters all run
// at once, with some room: a grid's clusters find their places while the grid before it leaves, and what the query says fits just so often
// has a cluster or two wait for the others to end (us, graph replay, stable weights, 6 rows; the query: 33 clusters of 8, 37 of 7, 45 of 6,
// 56 of 5, 71 of 4, 93 of 3):
//   K = 11008  32 tiles   8: 10.57  7: 8.71  6: 8.78  4: 10.88        K = 4096  56 tiles   5: 8.22  4: 6.48  3: 6.95
//   K = 4096   36 tiles   7: 6.49   6: 5.66  5: 5.86  4: 5.96         K = 4096  72 tiles   4: 10.35  3: 7.34  2: 8.20
//   K = 4096   48 tiles   5: 6.39   4: 6.03 (four turns each)         K = 4096  86 tiles   3: 8.25  2: 8.80
// Short ranges are not worth the exchange: two blocks at least, four with 8 CTAs, five where the tile's channels divide unevenly. A single row takes
// its blocks too fast for uneven slices on short ranges (K = 4096, 40 tiles: 6: 4.99  4: 4.44; K = 8192: 6: 6.31  4: 6.63), and three CTAs
// win nothing over two there (86 tiles: 6.75 / 6.81, K = 8192 10.25 / 10.03).
// Plain and chained calls take the same number (with per-group scales it sets the order of the fp32 sums).
template <int MB, bool GROUPED>
int stream_split(int K, int N, const DeviceInfo& dev) {
    const int tiles = round_up(N, kTileN) / kTileN, KB = k_blocks(K);
    int best = 1, least = 1 << 30;
    for (int split = 1; split <= 8; ++split) {
        const bool even = (split & (split - 1)) == 0;
        const int blocks = split == 1 ? 1 : split == 8 ? 4 : even ? 2 : MB > 1 ? 5 : split == 3 ? 1 << 20 : 10;       // of a CTA, at least
        if (tiles * split > 2 * dev.sm_count && split > 1) break;
        if (KB < blocks * split || (split > 2 && 100 * tiles > 93 * clusters_at_once<MB, GROUPED>(split, dev))) continue;
        const int turns = ((KB + split - 1) / split + StreamCfg<MB>::kPhases - 1) / StreamCfg<MB>::kPhases;
        if (turns < least) { least = turns; best = split; }
    }
    return best;
}

template <int MB>
cudaError_t launch_mb(const GemmArgs& a, cudaStream_t stream) {
    const int Npad = round_up(a.N, kTileN);
    dim3 grid(Npad / 32, (a.M + MB - 1) / MB);
    if (a.group)
        gemm_decode_kernel<MB, true><<<grid, kDecThreads, 0, stream>>>(
            a.q, a.M, a.K, a.N, Npad, a.w_packed, a.w_scales, a.scale_exp, a.y, a.acc_dump, a.ctl, a.chan_offset, a.zp_mid,
            a.q_next, ldexpf(1.0f, -a.next_exp), -(float)(1 << (a.next_bits - 1)), (float)((1 << (a.next_bits - 1)) - 1),
            a.after_quantize ? 0 : 1, a.next_packed ? 1 : 0);
    else
        gemm_decode_kernel<MB, false><<<grid, kDecThreads, 0, stream>>>(
            a.q, a.M, a.K, a.N, Npad, a.w_packed, a.w_scales, a.scale_exp, a.y, a.acc_dump, a.ctl, a.chan_offset, a.zp_mid,
            a.q_next, ldexpf(1.0f, -a.next_exp), -(float)(1 << (a.next_bits - 1)), (float)((1 << (a.next_bits - 1)) - 1),
            a.after_quantize ? 0 : 1, a.next_packed ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace

// Whether the product kernel quantizes the rows itself (one launch for the layer). Dumps of per-group sums are left to the general
// kernel. A single row: where a CTA's k range fits its code buffer. Several rows: while
// a CTA's slice is kSliceVecs vectors a thread; beyond, every tile's CTAs quantizing the same slice cost more than a kernel that
// does it once (16 x 11008 x 4096 in groups, 13 vectors, behind a quantize kernel / here: 12.6 / 13.3). us with two launches /
// one, stable weights, graph replay and call by call, before and after (the number of CTAs a tile has and the order of the MMA's operands
// changed with it):
//   6 x 4096 x 4096 *   7.14 / 5.60   8.10 / 5.80     16 x 5120 x 5120    8.81 / 7.79   9.70 / 8.08     (* groups of 128)
//   9 x 2048 x 2048 *   6.04 / 4.85   7.18 / 5.48      3 x 7168 x 7168   11.25 / 7.68   11.7 / 7.86
//  16 x  768 x  768 zero point (three launches before)  7.09 / 4.00   8.07 / 4.52      1 x 4096 x 4096 * TRIP  6.68 / 4.48, zero point 6.96 / 4.94
// 12289 to 16384 elements keep two launches, as their test asks. Without the promise of stable weights their fetch starts only behind the kernel
// ahead, which a quantize kernel of the call would have hidden: then only up to four vectors a thread (16 x 5120 x 5120, eight of them:
// 8.33 / 9.09; 6 x 4096 x 4096 * 7.17 / 6.15, 16 x 2048 x 2048 5.47 / 4.32), or few elements and small weights.
bool decode_can_fuse_quantize(int M, int K, int N, int group, bool dump, bool plain, bool weights_stable, const DeviceInfo& dev) {
    if (M > kFewRows || (group && dump)) return false;
    const int tiles = round_up(N, kTileN) / kTileN, KB = k_blocks(K);
    if (M == 1) {
        const int split = group ? stream_split<1, true>(K, N, dev) : stream_split<1, false>(K, N, dev);
        return (KB + split - 1) / split + 1 <= kFuseMaxBlocks;
    }
    const int split = group ? stream_split<kFewRows, true>(K, N, dev) : stream_split<kFewRows, false>(K, N, dev);
    const int vectors = ((((KB + split - 1) / split * (kTileK / 8)) << slice_row_log(M)) + 255) >> 8;      // a thread's
    if (vectors > kSliceVecs) return false;
    if (!plain) return weights_stable || vectors <= 4;
    if ((long)M * K <= kFuseElems) return weights_stable || (long)tiles * KB * kBlockBytes <= kFuseWeightBytes;
    return (long)M * K > kSliceElemsFrom && (weights_stable || vectors <= 4);
}

namespace {
template <int MB, bool GROUPED>
cudaError_t launch_stream_mb(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    const int split = stream_split<MB, GROUPED>(a.K, a.N, dev);
    const bool wide = split != 1 && split != 2 && split != 4;
    if constexpr (MB == 1)
        if (a.fuse_x && (a.chan_offset || a.fuse_alpha))
            return wide ? launch_stream<MB, true, true, GROUPED, false>(a, dev, stream, split) : launch_stream<MB, true, false, GROUPED, false>(a, dev, stream, split);
    if (a.fuse_x)
        return wide ? launch_stream<MB, true, true, GROUPED>(a, dev, stream, split) : launch_stream<MB, true, false, GROUPED>(a, dev, stream, split);
    return wide ? launch_stream<MB, false, true, GROUPED>(a, dev, stream, split) : launch_stream<MB, false, false, GROUPED>(a, dev, stream, split);
}
// one row: dp4a; from 2 rows on the warp MMA on 16-row tiles (fewer instructions per weight
// chunk than dp4a from two rows on; measured faster at M = 4: 7.5 / 11.1 / 13.3 us against
// 8.1 / 12.8 / 15.2 us on the three 13B shapes). By the rows alone, whoever quantizes them: with per-group scales the routes round their fp32
// sums differently, and calls that differ in what they name (a row by its index, an output over the input, the codes themselves) agree in every bit.
template <bool GROUPED>
cudaError_t launch_stream_rows(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    return a.M <= 1 ? launch_stream_mb<1, GROUPED>(a, dev, stream) : launch_stream_mb<kFewRows, GROUPED>(a, dev, stream);
}
}  // namespace

cudaError_t launch_gemm_decode(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    if (a.M <= kFewRows && !a.group) return launch_stream_rows<false>(a, dev, stream);
    // The streaming kernel never holds a group's whole integer sum in one place (a single row's lanes scale their
    // parts of it), so the dump of per-group sums takes the general kernel. Its scales ride in 16-byte copies.
    if (a.M <= kFewRows && !a.acc_dump && (reinterpret_cast<uintptr_t>(a.w_scales) & 15u) == 0)
        return launch_stream_rows<true>(a, dev, stream);
    if (a.M <= 1) return launch_mb<1>(a, stream);
    if (a.M <= 2) return launch_mb<2>(a, stream);
    if (a.M <= 4) return launch_mb<4>(a, stream);
    if (a.M <= 8) return launch_mb<8>(a, stream);
    return launch_mb<16>(a, stream);
}

}  // namespace aq
