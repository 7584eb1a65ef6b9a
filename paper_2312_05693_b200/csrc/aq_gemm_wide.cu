// Integer product with one scale per output channel (Sec. 4.4) on tiles of 256 channels x 128 or 192 tokens.
//
// The per-channel kernel of aq_gemm_tensor.cu moves 40 KB from L2 per 128-k block and SM (a 256-token
// activation tile and one packed 128-channel weight block) and runs within 20 % of what the L2 -> SM path
// delivers for that pattern. Here a CTA's tile covers TWO adjacent 128-channel blocks that share one
// activation tile of 128 or 192 tokens: 32 KB per k block for the products of 40 KB there, or 40 KB for one
// and a half times as many, so the same path feeds a fifth to a half more work. The two channel halves are
// two accumulators in tensor memory, each fed by its own MMA-issuing thread from its own weight slices, which
// its own group of four unpack warps writes; the activation tile in shared memory is the B operand of both.
// Each half has its own pair of accumulator barriers: the epilogue takes the halves one after the other.
// Roles: warp 0 = TMA producer of the activation tiles, warp 2 = of the two weight blocks, warps 1 and 3 =
// MMA issuers (half 0 / half 1), warps 4-7 and 8-11 = unpack (half 0 / half 1), warps 12-19 = epilogue.
// Needs an even number of 128-channel blocks; other shapes take the kernel of aq_gemm_tensor.cu.
// CLUSTER (128-token tiles): too few tiles for the SMs (short prompts, narrow layers). The CTAs of
// a cluster share a tile and take consecutive ranges of its k blocks; the tile's tokens are cut into eight runs, every
// CTA sends the integer sums of the runs it does not own into their owners' shared memory (the operand ring, idle by
// then) and finishes its own. Integer additions: the same results in any order; no scratch in memory, no flags.
#include <cooperative_groups.h>
#include <cuda.h>

#include "aq_common.cuh"
#include "aq_tc.cuh"

namespace cg = cooperative_groups;

namespace aq {

namespace {

constexpr int kWThreads = 20 * 32;
constexpr int kWFirstUnpack = 4, kWFirstEpi = 12, kWEpiWarps = 8;
constexpr int kWRegsControl = 40, kWRegsUnpack = 48, kWRegsEpi = 168;     // of the 96 x 640 the launch allocates
static_assert(128 * kWRegsControl + 256 * kWRegsUnpack + 256 * kWRegsEpi <= kWThreads * 96,
              "register plan exceeds the launch allocation");
constexpr int kWStageRows = 32;           // tokens per TMA store of an epilogue warp
constexpr int kWRuns = 8;                 // CLUSTER: token runs of a tile
template <int BM>
struct WCfg {
    static constexpr int kStages = BM == 128 ? 6 : 5;          // shared-memory ring: activation tile + two packed weight blocks per stage
    static constexpr int kSlices = (512 - 2 * BM) / 32;        // weight slices in tensor memory: (k block, half) pairs: 8 or 4
    static constexpr int kAccCols = 2 * BM;                    // two accumulators (one per channel half)
    static constexpr int kCols = BM / 2;                       // token columns of one epilogue warp (per half)
    static_assert(kCols % kWStageRows == 0 && kCols <= 96, "epilogue register plan");
};

template <int BM>
struct WSmem {
    static constexpr int kStages = WCfg<BM>::kStages;
    alignas(1024) uint8_t x[kStages][BM * 128];                // activation tiles, 128-byte swizzled rows
    alignas(128) uint8_t w[kStages][2][kBlockBytes];           // the two packed weight blocks of a k block
    alignas(128) __half ystage[kWEpiWarps][kWStageRows][32];
    alignas(8) uint64_t tma_full[kStages];                     // both producers' bytes landed -> unpack warps
    uint64_t smem_empty[kStages];                              // both halves' MMAs done -> TMA producers
    uint64_t a_full[8];                                        // a half's unpack warps stored the slice -> its MMA issuer
    uint64_t a_empty[8];                                       // MMA done with the slice -> unpack warps
    uint64_t acc_full[2];                                      // a half's last MMAs of the tile done -> epilogue
    uint64_t acc_empty[2];                                     // epilogue has the half's sums in registers -> its issuer
    uint32_t tmem_base;
    volatile uint32_t abort_flag;
};

struct WParams {
    int M, K, N, Npad, KB;
    int n_tiles_m, n_tiles;        // token tiles; tiles (token tile x channel pair)
    const uint8_t* w_packed;
    const __half* w_scales;
    const int32_t* scale_exp;
    __half* y;
    int32_t* acc_dump;
    Control* ctl;
    const float* chan_offset;      // NULL or [N]: per-channel term, times offset_factor
    int zp_mid;
    int8_t* q_next;
    float next_inv, next_lo, next_hi;
    int next_packed;
    int y_tma;
    int clear_status;              // no quantize kernel of the call has set the control block up
};

__device__ __forceinline__ int w_chain_code(__half hv, float inv, float lo, float hi) {
    const float t = __half2float(hv) * inv;                 // exact: inv is a power of two
    if (t != t) return 0;
    return (int)fminf(fmaxf(rintf(t), lo), hi);
}
__device__ __forceinline__ void w_stage_code(__half* stage, int c, int lane, int code, int packed) {
    if (packed) {
        const int hi = __shfl_down_sync(0xFFFFFFFFu, code, 1);
        if (!(lane & 1)) reinterpret_cast<uint8_t*>(stage)[c * 16 + (lane >> 1)] = (uint8_t)((code & 0xF) | (hi << 4));
    } else {
        reinterpret_cast<int8_t*>(stage)[c * 32 + lane] = (int8_t)code;
    }
}

__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

// OFFSET: add the per-channel term of the zero-point variant. CHAIN: write the next layer's codes instead
// of fp16 outputs.
template <int BM, bool OFFSET, bool CHAIN, bool CLUSTER>
__global__ void __launch_bounds__(kWThreads, 1)
gemm_wide_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap y_map, const WParams p) {
    extern __shared__ uint8_t smem_raw[];
    using Smem = WSmem<BM>;
    Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int kWBM = BM, kWStages = WCfg<BM>::kStages, kWSlices = WCfg<BM>::kSlices, kWAccCols = WCfg<BM>::kAccCols;
    constexpr int kCols = WCfg<BM>::kCols;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int KB = p.KB;
    static_assert(!CLUSTER || BM == 128, "runs of 16 tokens");
    const int rank = CLUSTER ? (int)blockIdx.x : 0, split = CLUSTER ? (int)gridDim.x : 1;
    const int my_tiles = CLUSTER ? 1 : (p.n_tiles > (int)blockIdx.x ? (p.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0);
    const int kb0 = CLUSTER ? KB * rank / split : 0, kb1 = CLUSTER ? KB * (rank + 1) / split : KB;
    const uint32_t total_iters = (uint32_t)my_tiles * (uint32_t)(kb1 - kb0);
    auto tile_at = [&](int tl) { return CLUSTER ? (int)blockIdx.y : (int)(blockIdx.x + tl * gridDim.x); };
    [[maybe_unused]] int met = 0;                    // CLUSTER: meetings this warp has been to

    if (p.clear_status && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) p.ctl->status = 0;   // nothing has given up yet
    if (threadIdx.x == 0) {
        for (int s = 0; s < kWStages; ++s) {
            mbar_init(&sm.tma_full[s], 2);
            mbar_init(&sm.smem_empty[s], 2);
        }
        for (int i = 0; i < kWSlices; ++i) {
            mbar_init(&sm.a_full[i], 4);
            mbar_init(&sm.a_empty[i], 1);
        }
        for (int h = 0; h < 2; ++h) {
            mbar_init(&sm.acc_full[h], 1);
            mbar_init(&sm.acc_empty[h], kWEpiWarps);
        }
        sm.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sm.tmem_base)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    const uint32_t tmem_acc = tmem;                 // half h at column h * BM
    const uint32_t tmem_a = tmem + kWAccCols;       // then the slices of 32 columns
    volatile uint32_t* abort_flag = &sm.abort_flag;

    if (warp < kWFirstUnpack) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kWRegsControl));
        if (warp == 0 || warp == 2) {
            // ------------- TMA producers
            if (elect_one()) {
                uint32_t st = 0, ph = 1u;
                const uint32_t full0 = smem_u32(sm.tma_full), empty0 = smem_u32(sm.smem_empty);
                if (warp == 0) {
                    // behind the call's own quantize kernel (programmatic stream serialization) the codes are
                    // touched only after that grid has completed; the weight producer does not wait
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    const uint32_t x0 = smem_u32(sm.x[0]);
                    for (int tl = 0; tl < my_tiles; ++tl) {
                        const int m0 = tile_at(tl) % p.n_tiles_m * kWBM;
                        for (int k = kb0 * kTileK; k < kb1 * kTileK; k += kTileK) {
                            if (!mbar_wait_a(empty0 + 8u * st, ph, abort_flag, 1u)) goto role_done;
                            mbar_arrive_expect_tx_a(full0 + 8u * st, kWBM * 128);
                            tma_load_2d_a(x0 + st * (uint32_t)(kWBM * 128), &x_map, k, m0, full0 + 8u * st);
                            if (++st == (uint32_t)kWStages) { st = 0; ph ^= 1u; }
                        }
                    }
                } else {
                    const uint32_t w0 = smem_u32(sm.w[0][0]);
                    for (int tl = 0; tl < my_tiles; ++tl) {
                        const int np = tile_at(tl) / p.n_tiles_m;
                        const uint8_t* src = p.w_packed + ((size_t)(2 * np) * KB + kb0) * kBlockBytes;
                        for (int kb = kb0; kb < kb1; ++kb) {
                            if (!mbar_wait_a(empty0 + 8u * st, ph, abort_flag, 1u)) goto role_done;
                            mbar_arrive_expect_tx_a(full0 + 8u * st, 2 * kBlockBytes);
                            const uint32_t dst = w0 + st * (uint32_t)(2 * kBlockBytes);
                            tma_load_1d_a(dst, src, kBlockBytes, full0 + 8u * st);
                            tma_load_1d_a(dst + kBlockBytes, src + (size_t)KB * kBlockBytes, kBlockBytes, full0 + 8u * st);
                            src += kBlockBytes;
                            if (++st == (uint32_t)kWStages) { st = 0; ph ^= 1u; }
                        }
                    }
                }
            }
        } else {
            // ------------- MMA issuers: warp 1 = channel half 0, warp 3 = half 1
            const int h = warp >> 1;
            if (elect_one()) {
                // One thread's chain of look, four MMAs and commits: elected threads, and ring positions and phases in counters,
                // here and in the producers (K = 5120, N = 13824 at 1024 rows 55.6 -> 47.4 us; K = 13824, N = 5120 at 333 rows,
                // in clusters, 35.3 -> 31.1 us).
                constexpr uint32_t idesc = idesc_i8(128, kWBM);
                const uint64_t bdesc0 = smem_desc_sw128(smem_u32(sm.x[0]));
                const uint32_t d_addr = tmem_acc + (uint32_t)(h * kWBM);
                uint32_t s = 0, ai = (uint32_t)h, ph = 0;
                for (int tl = 0; tl < my_tiles; ++tl) {
                    if (!mbar_wait(&sm.acc_empty[h], ((uint32_t)tl & 1u) ^ 1u, abort_flag, 4u)) goto role_done;
                    for (int kb = kb0; kb < kb1; ++kb) {
                        // the unpack warps publish a slice only after the stage's TMA bytes (activation tile
                        // included) have landed, so this one wait covers both operands
                        if (!mbar_wait(&sm.a_full[ai], ph, abort_flag, 5u)) goto role_done;
                        tc_fence_after();
                        const uint32_t a_addr = tmem_a + ai * (uint32_t)kAColsPerStage;
                        const uint64_t bdesc = bdesc0 + (uint64_t)(s * (uint32_t)(kWBM * 128 / 16));
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            tc_mma_i8_ts(d_addr, a_addr + 8 * j, bdesc + (uint64_t)(2 * j), idesc, (kb == kb0 && j == 0) ? 0u : 1u);
                        tc_commit(&sm.a_empty[ai]);
                        tc_commit(&sm.smem_empty[s]);
                        if (++s == (uint32_t)kWStages) s = 0;
                        ai += 2;
                        if (ai >= (uint32_t)kWSlices) { ai -= kWSlices; ph ^= 1u; }
                    }
                    tc_commit(&sm.acc_full[h]);
                }
            }
        }
    } else if (warp < kWFirstEpi) {
        // --------------------------------------------------- weight unpack -> tensor memory (one group per half)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kWRegsUnpack));
        const int quarter = warp & 3;
        const int h = (warp - kWFirstUnpack) >> 2;
        const int r = quarter * 32 + lane;            // row inside the half's 128-channel block = TMEM lane
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        int pending = -1;                             // slice whose stores have been issued but not published
        uint32_t s = 0, s_ph = 0u, ai = (uint32_t)h, a_ph = 1u;
        for (uint32_t it = 0; it < total_iters; ++it) {
            if (!mbar_wait_warp(&sm.tma_full[s], s_ph, abort_flag, 6u)) goto role_done;
            const uint4* src = reinterpret_cast<const uint4*>(sm.w[s][h]) + r;
            uint4 d[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) d[j] = src[j * kTileN];
            if (pending >= 0) {                       // the previous stores had the loads above to finish
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.a_full[pending]);
            }
            if (!mbar_wait_warp(&sm.a_empty[ai], a_ph, abort_flag, 7u)) goto role_done;
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t w[4] = {d[j].x, d[j].y, d[j].z, d[j].w};
                uint32_t v[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    v[2 * i] = (w[i] << 4) & 0xF0F0F0F0u;           // 16*code for k0..k0+3
                    v[2 * i + 1] = w[i] & 0xF0F0F0F0u;              // 16*code for k0+4..k0+7
                }
                tc_st8(tmem_a + lane_addr + (uint32_t)(ai * kAColsPerStage + 8 * j), v);
            }
            pending = (int)ai;
            if (++s == (uint32_t)kWStages) { s = 0; s_ph ^= 1u; }
            ai += 2;
            if (ai >= (uint32_t)kWSlices) { ai -= kWSlices; a_ph ^= 1u; }
        }
        if (pending >= 0) {
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.a_full[pending]);
        }
    } else {
        // ----------------------------------------------------------------------- epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kWRegsEpi));
        const int ew = warp - kWFirstEpi;
        const int quarter = warp & 3;
        const int chalf = ew >> 2;                    // which half of the tile's token columns
        const int r = quarter * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const int col0 = chalf * kCols;
        asm volatile("griddepcontrol.wait;" ::: "memory");               // see the activation producer
        const float pe = __int_as_float((127 + *p.scale_exp) << 23);     // 2^e
        [[maybe_unused]] const float off_factor = OFFSET ? offset_factor(p.ctl, p.zp_mid) : 0.0f;
        __half* stage = &sm.ystage[ew][0][0];
        for (int tl = 0; tl < my_tiles; ++tl) {
            const int tile = tile_at(tl);
            const int mt = tile % p.n_tiles_m, np = tile / p.n_tiles_m;
            const int m_base = mt * kWBM + col0;
            float sc[2], off_pe[2];
            bool n_ok[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int n = (2 * np + h) * kTileN + r;
                n_ok[h] = n < p.N;
                sc[h] = __half2float(p.w_scales[n]) * 0.0625f * pe;      // sums carry a factor 16 (n < Npad: the scale array is padded)
                off_pe[h] = (OFFSET && n_ok[h]) ? __fmul_rn(off_factor, p.chan_offset[n]) * pe : 0.0f;
            }
            if constexpr (CLUSTER) {
                // run c of the tile's tokens belongs to CTA c % split (so that both of a lane quarter's warps have runs to send and to
                // finish; in slices of neighbouring runs 333 x 13824 x 5120, clusters of two, took 33.5 us instead of 31.5); the receiving area of a CTA is laid out as
                // [sender][run of the slice][half][4 columns][channel][column]. The sums stay in tensor memory and are
                // read once to be sent and once to be finished.
                constexpr int kRun = BM / kWRuns, kRunInts = 2 * kRun * kTileN;
                constexpr int kRing = kWStages * (BM * 128 + 2 * kBlockBytes), kRunBytes = kRunInts * 4;
                static_assert(offsetof(Smem, x) + sizeof(sm.x) == offsetof(Smem, w) && 4 * kRunBytes <= kRing && 2 * 3 * kRunBytes <= kRing &&
                                  3 * 2 * kRunBytes <= kRing && 4 * 2 * kRunBytes <= kRing && 5 * 2 * kRunBytes <= kRing &&
                                  6 * 2 * kRunBytes <= kRing && 7 * kRunBytes <= kRing,
                              "the operand ring (activation tiles, then weight blocks) holds what a CTA receives in clusters of two to eight");
                cg::cluster_group cluster = cg::this_cluster();
                int* ring = reinterpret_cast<int*>(&sm.x[0][0]);
                const int slice_runs = (kWRuns + split - 1) / split;     // the most a CTA owns
                bool ok = true;
                for (int h = 0; h < 2; ++h) ok = ok && mbar_wait_warp(&sm.acc_full[h], 0u, abort_flag, 8u);
                tc_fence_after();
                cluster_meet();                                        // every CTA's operand ring is idle
                met = 1;
                if (!ok) goto role_done;
#pragma unroll 1
                for (int h = 0; h < 2; ++h)
#pragma unroll 1
                    for (int c0 = 0; c0 < kCols; c0 += 32) {
                        uint32_t v[32];
                        tc_ld32(tmem_acc + lane_addr + (uint32_t)(h * kWBM + col0 + c0), v);
                        tc_wait_ld();
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int c = (col0 + c0) / kRun + i, owner = c % split;
                            if (owner == rank || mt * kWBM + c * kRun >= p.M) continue;
                            const int from = rank < owner ? rank : rank - 1;
                            int4* dst = reinterpret_cast<int4*>(cluster.map_shared_rank(ring, owner) +
                                                                (size_t)(from * slice_runs + c / split) * kRunInts) + h * (kRun / 4) * kTileN + r;
#pragma unroll
                            for (int q = 0; q < kRun / 4; ++q)
                                dst[q * kTileN] = make_int4((int)v[i * kRun + 4 * q], (int)v[i * kRun + 4 * q + 1],
                                                            (int)v[i * kRun + 4 * q + 2], (int)v[i * kRun + 4 * q + 3]);
                        }
                    }
                cluster_meet();                                        // all sums have arrived; nobody writes here any more
                met = 2;
#pragma unroll 1
                for (int c = rank; c < kWRuns; c += split) {
                    // (this warp's runs among those its CTA owns)
                    if (c * kRun < col0 || c * kRun >= col0 + kCols || mt * kWBM + c * kRun >= p.M) continue;
                    const int m0 = mt * kWBM + c * kRun;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t v[kRun];
                        tc_ld16(tmem_acc + lane_addr + (uint32_t)(h * kWBM + c * kRun), v);
                        tc_wait_ld();
                        for (int from = 0; from < split - 1; ++from) {
                            const int4* src = reinterpret_cast<const int4*>(ring + (size_t)(from * slice_runs + c / split) * kRunInts) +
                                              h * (kRun / 4) * kTileN + r;
#pragma unroll
                            for (int q = 0; q < kRun / 4; ++q) {
                                const int4 o = src[q * kTileN];
                                v[4 * q] += (uint32_t)o.x;
                                v[4 * q + 1] += (uint32_t)o.y;
                                v[4 * q + 2] += (uint32_t)o.z;
                                v[4 * q + 3] += (uint32_t)o.w;
                            }
                        }
                        const int n = (2 * np + h) * kTileN + r, n0 = (2 * np + h) * kTileN + quarter * 32;
                        if (p.y_tma) {
                            if (lane == 0) tma_store_wait_read();
                            __syncwarp();
                        }
#pragma unroll
                        for (int k = 0; k < kRun; ++k) {
                            const __half hv = __float2half_rn(OFFSET ? fmaf((float)(int)v[k], sc[h], off_pe[h]) : (float)(int)v[k] * sc[h]);
                            if (p.y_tma) {
                                if constexpr (CHAIN)
                                    w_stage_code(stage, k, lane, w_chain_code(hv, p.next_inv, p.next_lo, p.next_hi), p.next_packed);
                                else
                                    stage[k * 32 + lane] = hv;
                            } else if (n_ok[h] && m0 + k < p.M) {
                                if constexpr (CHAIN)
                                    p.q_next[(size_t)(m0 + k) * p.N + n] = (int8_t)w_chain_code(hv, p.next_inv, p.next_lo, p.next_hi);
                                else
                                    p.y[(size_t)(m0 + k) * p.N + n] = hv;
                            }
                            if (p.acc_dump && n_ok[h] && m0 + k < p.M) p.acc_dump[(size_t)(m0 + k) * p.N + n] = (int)v[k] >> 4;
                        }
                        if (p.y_tma) {
                            fence_proxy_async();
                            __syncwarp();
                            if (lane == 0 && n0 < p.N) tma_store_2d(&y_map, stage, (CHAIN && p.next_packed) ? n0 >> 1 : n0, m0);
                        }
                    }
                }
                goto role_done;
            }
            // One half after the other: the half's sums (this warp's columns) go to registers and its
            // accumulator returns to its issuer at once, so that conversion and stores overlap the next tile's MMAs.
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!mbar_wait_warp(&sm.acc_full[h], (uint32_t)tl & 1u, abort_flag, 8u)) goto role_done;
                tc_fence_after();
                uint32_t v[kCols];
#pragma unroll
                for (int c0 = 0; c0 < kCols; c0 += 32)
                    tc_ld32(tmem_acc + lane_addr + (uint32_t)(h * kWBM + col0 + c0), *reinterpret_cast<uint32_t(*)[32]>(&v[c0]));
                tc_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.acc_empty[h]);
                const int n = (2 * np + h) * kTileN + r;
                const int n0 = (2 * np + h) * kTileN + quarter * 32;
                if (p.y_tma) {
#pragma unroll
                    for (int r0 = 0; r0 < kCols; r0 += kWStageRows) {
                        if (lane == 0) tma_store_wait_read();     // the previous store has read the staging rows
                        __syncwarp();
#pragma unroll
                        for (int c = 0; c < kWStageRows; ++c) {
                            const __half hv = __float2half_rn(OFFSET ? fmaf((float)(int)v[r0 + c], sc[h], off_pe[h])
                                                                     : (float)(int)v[r0 + c] * sc[h]);
                            if constexpr (CHAIN)
                                w_stage_code(stage, c, lane, w_chain_code(hv, p.next_inv, p.next_lo, p.next_hi), p.next_packed);
                            else
                                stage[c * 32 + lane] = hv;
                        }
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0 && n0 < p.N && m_base + r0 < p.M)
                            tma_store_2d(&y_map, stage, (CHAIN && p.next_packed) ? n0 >> 1 : n0, m_base + r0);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < kCols; ++c) {
                        const int m = m_base + c;
                        if (n_ok[h] && m < p.M) {
                            const __half hv = __float2half_rn(OFFSET ? fmaf((float)(int)v[c], sc[h], off_pe[h])
                                                                     : (float)(int)v[c] * sc[h]);
                            if constexpr (CHAIN)
                                p.q_next[(size_t)m * p.N + n] = (int8_t)w_chain_code(hv, p.next_inv, p.next_lo, p.next_hi);
                            else
                                p.y[(size_t)m * p.N + n] = hv;
                        }
                    }
                }
                if (p.acc_dump) {
#pragma unroll
                    for (int c = 0; c < kCols; ++c) {
                        const int m = m_base + c;
                        if (n_ok[h] && m < p.M) p.acc_dump[(size_t)m * p.N + n] = (int)v[c] >> 4;
                    }
                }
            }
        }
    }

role_done:
    if (warp >= kWFirstEpi && lane == 0) tma_store_wait_read();   // staging rows live until read
    __syncwarp();
    if constexpr (CLUSTER)
        for (; met < 2; ++met) cluster_meet();                  // every warp comes to both meetings
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (sm.abort_flag) {
        for (int i = 0; i < 64; ++i) __nanosleep(1000);          // let copies in flight land
        if (threadIdx.x == 0) atomicCAS(&p.ctl->status, 0u, sm.abort_flag);
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

typedef CUresult (*WEncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Tiles in turn on a persistent grid, or one per cluster of `split` CTAs.
template <int BM, bool OFFSET, bool CHAIN, bool CLUSTER>
cudaError_t launch_wide_t(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream, int split) {
    constexpr int kWBM = BM;
    const size_t smem_bytes = sizeof(WSmem<BM>) + 1024;
    static SmemOptIn opt_in;
    if (const cudaError_t e = opt_in.ensure(gemm_wide_kernel<BM, OFFSET, CHAIN, CLUSTER>, dev.device, smem_bytes); e != cudaSuccess)
        return e;
    WEncodeTiledFn enc = reinterpret_cast<WEncodeTiledFn>(dev.encode_tiled);
    CUtensorMap map;
    const cuuint64_t dims[2] = {(cuuint64_t)a.K, (cuuint64_t)a.M};
    const cuuint64_t strides[1] = {(cuuint64_t)a.K};
    const cuuint32_t box[2] = {128u, (cuuint32_t)kWBM};
    const cuuint32_t estr[2] = {1u, 1u};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t*>(a.q), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    const cuuint32_t store_rows = CLUSTER ? BM / kWRuns : kWStageRows;
    CUtensorMap ymap = map;   // placeholder when the store path is off
    int y_tma = 0;
    if (CHAIN) {
        if (a.next_packed && (a.N % 32 != 0 || (reinterpret_cast<uintptr_t>(a.q_next) & 15u) != 0))
            return cudaErrorInvalidValue;                    // packed codes only leave through the TMA store
        if (a.N % 16 == 0 && (reinterpret_cast<uintptr_t>(a.q_next) & 15u) == 0) {
            const cuuint64_t row_bytes = a.next_packed ? (cuuint64_t)a.N / 2 : (cuuint64_t)a.N;
            const cuuint64_t ydims[2] = {row_bytes, (cuuint64_t)a.M};
            const cuuint64_t ystrides[1] = {row_bytes};
            const cuuint32_t ybox[2] = {a.next_packed ? 16u : 32u, store_rows};
            if (enc(&ymap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, a.q_next, ydims, ystrides, ybox, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
            y_tma = 1;
        }
    } else if (a.N % 8 == 0 && (reinterpret_cast<uintptr_t>(a.y) & 15u) == 0) {
        const cuuint64_t ydims[2] = {(cuuint64_t)a.N, (cuuint64_t)a.M};
        const cuuint64_t ystrides[1] = {(cuuint64_t)a.N * 2};
        const cuuint32_t ybox[2] = {32u, store_rows};
        if (enc(&ymap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, a.y, ydims, ystrides, ybox, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        y_tma = 1;
    }
    WParams p;
    p.M = a.M; p.K = a.K; p.N = a.N; p.Npad = round_up(a.N, kTileN); p.KB = k_blocks(a.K);
    p.n_tiles_m = (a.M + kWBM - 1) / kWBM;
    p.n_tiles = p.n_tiles_m * (p.Npad / (2 * kTileN));
    p.w_packed = a.w_packed; p.w_scales = a.w_scales; p.scale_exp = a.scale_exp;
    p.y = a.y; p.acc_dump = a.acc_dump; p.ctl = a.ctl; p.chan_offset = a.chan_offset; p.zp_mid = a.zp_mid;
    p.q_next = a.q_next;
    p.next_inv = ldexpf(1.0f, -a.next_exp);
    p.next_lo = -(float)(1 << (a.next_bits - 1));
    p.next_hi = (float)((1 << (a.next_bits - 1)) - 1);
    p.next_packed = a.next_packed ? 1 : 0;
    p.y_tma = y_tma;
    p.clear_status = a.after_quantize ? 0 : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = CLUSTER ? dim3(split, p.n_tiles) : dim3(p.n_tiles < dev.sm_count ? p.n_tiles : dev.sm_count);
    cfg.blockDim = dim3(kWThreads);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = a.after_quantize ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = split;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CLUSTER ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, gemm_wide_kernel<BM, OFFSET, CHAIN, CLUSTER>, map, ymap, p);
}

}  // namespace

namespace {
// Clusters of `split` CTAs that run at once (one CTA fills an SM; a GPC holds only so many clusters of a size).
int wide_clusters(const DeviceInfo& dev, int split) {
    static std::atomic<int> known[kMaxDevices][9];               // + 1 (0: not asked yet)
    int k = known[dev.device][split].load(std::memory_order_relaxed);
    if (k == 0) {
        const size_t smem_bytes = sizeof(WSmem<128>) + 1024;
        static SmemOptIn opt_in;
        int n = 0;
        if (opt_in.ensure(gemm_wide_kernel<128, false, false, true>, dev.device, smem_bytes) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(split, 1);
            cfg.blockDim = dim3(kWThreads);
            cfg.dynamicSmemBytes = smem_bytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = split;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, gemm_wide_kernel<128, false, false, true>, &cfg) != cudaSuccess) {
                (void)cudaGetLastError();
                n = 0;
            }
        }
        k = n + 1;
        known[dev.device][split].store(k, std::memory_order_relaxed);
    }
    return k - 1;
}

// How a shape is run, and what it costs in nanoseconds (fitted with the prices of channel_plan, see there): rounds of tiles over the SMs x k
// blocks x the time of a k block, which the L2 -> SM path sets (32 KB per k block on 128-token tiles, 40 KB on 192-token tiles)
// unless the tensor pipe's 512 / 768 cycles are longer. 128-token tiles that are few enough for all of them to run at once in
// clusters may do so: fewer k blocks in a row for an exchange. 333 rows, N = 5120 (60 tiles, clusters of two): K = 13824 49.2 -> 35.3 us.
// (Only the last, partial round in clusters behind whole rounds: measured slower, K = 13824, N = 5120 at 1024 rows, 148 + 12 tiles,
// 68 us against 57.6 on 192-token tiles.)
struct WidePlan {
    int bm, split;                   // token tile; CTAs that share a tile
    long cost;
};
WidePlan wide_plan(const GemmArgs& a, const DeviceInfo& dev) {
    const int pairs = round_up(a.N, kTileN) / (2 * kTileN), KB = k_blocks(a.K), sms = dev.sm_count;
    const int tiles192 = (a.M + 191) / 192 * pairs, tiles128 = (a.M + 127) / 128 * pairs;
    constexpr int kCall = 106, kRound = 2750, kBlock128 = 231, kBlock192 = 381, kExchange = 5700, kExchangeCta = 62;
    WidePlan best = {192, 1, kCall + (long)((tiles192 + sms - 1) / sms) * (kRound + (long)KB * kBlock192)};
    const long cost128 = kCall + (long)((tiles128 + sms - 1) / sms) * (kRound + (long)KB * kBlock128);
    if (cost128 <= best.cost) best = {128, 1, cost128};
    for (int s = 2; s <= 8 && s <= KB && s * tiles128 <= sms; ++s) {
        if (wide_clusters(dev, s) < tiles128) continue;
        const long c = kCall + (long)((KB + s - 1) / s) * kBlock128 + kExchange + (long)(s - 2) * kExchangeCta;
        if (c < best.cost) best = {128, s, c};
    }
    return best;
}

template <bool OFFSET, bool CHAIN>
cudaError_t launch_wide_v(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    const WidePlan w = wide_plan(a, dev);
    if (w.bm == 192) return launch_wide_t<192, OFFSET, CHAIN, false>(a, dev, stream, 1);
    if (w.split == 1) return launch_wide_t<128, OFFSET, CHAIN, false>(a, dev, stream, 1);
    return launch_wide_t<128, OFFSET, CHAIN, true>(a, dev, stream, w.split);
}
}  // namespace

// Whether the pair tiles are the better choice: where their schedule is no longer than `other`, that of the tiles of one
// channel block (channel_plan).
bool gemm_wide_applies(const GemmArgs& a, const DeviceInfo& dev, long other) {
    if (a.group || (round_up(a.N, kTileN) / kTileN) % 2 != 0) return false;
    return wide_plan(a, dev).cost <= other;
}

cudaError_t launch_gemm_wide(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    if (a.q_next) {
        if (a.chan_offset) return cudaErrorInvalidValue;       // the two variants are not combined
        return launch_wide_v<false, true>(a, dev, stream);
    }
    if (a.chan_offset) return launch_wide_v<true, false>(a, dev, stream);
    return launch_wide_v<false, false>(a, dev, stream);
}

}  // namespace aq
