// Integer product on the 5th-generation tensor cores (tcgen05, kind::i8) with TMEM
// accumulators, for the sums of Sec. 4.4 / Algorithm 1 and the floating-point output.
//
// Operand roles are swapped with respect to y = x w^T: the 128 output channels of a tile
// are the MMA's M dimension and the tokens its N dimension, so that
//   * the 4-bit weights stay packed in shared memory (one contiguous 8 KB bulk copy per
//     128 x 128 block): four warps widen each nibble to the int8 value 16*code with two
//     logic ops per word and store the result straight into tensor memory, where the MMA
//     reads it as its A operand, so the widened weights never take shared-memory bandwidth;
//   * every epilogue thread owns one output channel, so its weight scale(s) sit in a
//     register and the per-128-k group rescaling costs one FMA per element;
//   * the int8 activation tile (tokens x 128 k) is the only shared-memory operand, staged
//     by TMA with the 128-byte swizzle and read through an MMA shared-memory descriptor.
//
// One persistent CTA per SM walks a static list of (channel tile, token tile) pairs.
// Warp roles: 0 and 2 = TMA producers (activations / weights), 1 = MMA issuer (and owner of the TMEM
// allocation), 3 = watches the accumulator barriers for the epilogue (per-group mode), 4-11 = weight unpack
// (two groups of four taking alternate k blocks; the per-group kernel on 192-token tiles has one),
// 12-19 = epilogue; registers are moved from
// the first two roles to the epilogue with setmaxnreg. The issuing threads are chosen with elect.sync: then the
// compiler knows that one thread is active, and a k block's four MMAs and three commits take about 100 cycles of
// it, a producer's turn about 300. Behind `lane == 0` they took 500 each, and that, not memory or the tensor
// cores, was the pace of every shape with few tokens. Two (one scale per channel)
// or three (per-group scales) accumulator stages in TMEM let the epilogue of one
// accumulation overlap the MMAs of the next ones. Every wait on an mbarrier is bounded; on expiry the CTA records a status
// word, stops issuing work and leaves through the common exit that frees TMEM. The named barriers have no limit; the watcher
// arrives at them whatever has given up, and says which tile is the last (see there).
#include <cooperative_groups.h>
#include <cuda.h>

#include "aq_common.cuh"
#include "aq_tc.cuh"

namespace cg = cooperative_groups;

namespace aq {

namespace {

constexpr int kUnpackGroups = 2;              // groups of four unpack warps; group g takes k blocks g, g+2, ...
constexpr int kFirstUnpackWarp = 4;           // warps 0-3 (one warpgroup): two TMA producers, the MMA issuer
constexpr int kWarps = 20;
constexpr int kThreads = kWarps * 32;
// Registers per thread after the roles split (setmaxnreg works on aligned groups of four warps):
// (Unpack warps with 40 instead of 48: 128 x 4096 x 11008 in groups 20.1 -> 19.0 us, 333 x 5120 x 5120 24.7 -> 23.4, 1000 x 1024 x 4096
// 15.8 -> 15.2; the 64- and 192-token tiles within 1 %.)
constexpr int kRegsControl = 40, kRegsUnpack = 40;
// The warps behind the control warpgroup are unpack warps, then epilogue warps. Eight epilogue warps (two per
// TMEM lane quarter, half of the token columns each) follow two groups of unpack warps; the per-group
// kernels with 192-token tiles run twelve (three per quarter, a third of the columns each) behind
// the one unpack group they need: there the per-group rescaling sets the pace, and a third warp per
// scheduler hides the latency of the other two's barrier and tensor-memory round trips.
template <int BM, bool GROUPED>
struct Roles {
    static constexpr int kEpiWarps = (GROUPED && BM == 192) ? 12 : 8;
    static constexpr int kFirstEpiWarp = kWarps - kEpiWarps;
    static constexpr int kRegsEpilogue = kEpiWarps == 12 ? 128 : 168;
    static constexpr int kColsPerEpiWarp = BM / (kEpiWarps / 4);
    // setmaxnreg can only hand out what the launch allocated (96 registers for each of the threads): a
    // larger request would wait forever.
    static_assert(128 * kRegsControl + 32 * (kFirstEpiWarp - kFirstUnpackWarp) * kRegsUnpack +
                          32 * kEpiWarps * kRegsEpilogue <= kThreads * 96,
                  "register plan exceeds the launch allocation");
};
template <int BM>
struct TileConfig {
    // shared-memory ring depth: activation tile + packed weight block (+ scales) per stage
    // (64 tokens: a turn of the ring, from the copy's issue to the MMA's commit, takes about 3500 cycles. Twelve stages,
    // both unpack groups and elected issuers: a layer of 48 rows 4096 x 4096 18.6 -> 14.3 us, 4096 x 11008 19.0 -> 15.0 us,
    // 11008 x 4096 27.4 -> 21.9 us; with one scale per channel, 4096 x 4224, 17.4 -> 11.6 us.)
    static constexpr int kNumStages = BM >= 192 ? 5 : BM > 64 ? 7 : 12;
};

template <int BM, int EPI_WARPS>
struct SharedStorage {
    static constexpr int kNumStages = TileConfig<BM>::kNumStages;
    alignas(1024) uint8_t x[kNumStages][BM * 128];   // activation tiles, 128-byte swizzled rows
    alignas(128) uint8_t w[kNumStages][kBlockBytes]; // packed weight blocks (128 channels x 128 k)
    // Weight scales of each block's group (grouped mode), in a ring three slots deeper than the
    // stage ring. A slot is rewritten for block i only after the MMAs of block i - kNumStages
    // completed, which (three accumulator stages) needs the epilogue of every block up to
    // i - kNumStages - 3 to have finished: all reads of the slot's previous content are done.
    static constexpr int kNumScaleSlots = kNumStages + 3;
    alignas(16) __half sc[kNumScaleSlots][kTileN];
    // Each epilogue warp stages fp16 outputs of its 32 channels here, kStageRows tokens at a time
    // (token-major rows of 64 bytes), and hands them to a TMA store.
    static constexpr int kStageRows = BM / (EPI_WARPS / 4) <= 64 ? BM / (EPI_WARPS / 4) : 32;
    alignas(128) __half ystage[EPI_WARPS][kStageRows][32];
    alignas(8) uint64_t tma_full[kNumStages];        // both producers' bytes landed -> unpack warps
    uint64_t smem_empty[kNumStages];                 // MMA done (+ epilogue took the scales) -> TMA producers
    uint64_t a_full[8];                              // unpack warps stored the slice -> MMA
    uint64_t a_empty[8];                             // MMA done with the slice -> unpack warps
    uint64_t acc_full[3];                            // MMA -> epilogue
    uint64_t acc_empty[3];                           // epilogue -> MMA
    uint32_t tmem_base;
    volatile uint32_t abort_flag;
    volatile int given_up;                           // per-group mode: the tile the watcher gave up in, the CTA's last
};

struct TensorParams {
    int M, K, N, Npad;
    int n_tiles_m, n_tiles;        // token tiles; total tiles
    const uint8_t* w_packed;
    const __half* w_scales;
    const int32_t* scale_exp;
    __half* y;
    int32_t* acc_dump;
    Control* ctl;
    const float* chan_offset;      // NULL or [N]: per-channel term added before the 2^e factor, times offset_factor
    int zp_mid;
    int split_base;                // SPLIT kernels: CTAs 2j and 2j+1 share tile split_base + j, half of K each
    float* split_scratch;          // [shared tile][half][epilogue warp][column][lane] fp32 partial outputs
    int8_t* q_next;                // chaining: the next layer's codes [M][N] are written instead of y
    float next_inv, next_lo, next_hi;   // 2^-next_exp and the code range of the next layer
    int next_packed;               // chaining: 4-bit codes leave two per byte (even channel in the low nibble)
    int y_tma;                     // outputs leave through y_map (needs N % 8 == 0 and a 16-byte aligned y)
    int clear_status;              // no quantize kernel of the call has set the control block up
    unsigned long long wait_cycles;   // limit of a wait
};

__device__ __forceinline__ __half ld_shared_half(uint32_t addr) {
    unsigned short v;
    asm volatile("ld.shared.b16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return __ushort_as_half(v);
}
// Waits for a phase that only needs the epilogue warps to go on, and so is sure to come, whatever has given up elsewhere (all
// lanes of a warp). Limited all the same: in tries, since on a GPU that is taken away from all warps for a while only the clock
// goes on, and over all such waits together (a tile takes some 10^3 of them).
constexpr uint32_t kDrainTries = 1u << 22;
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity, uint32_t& tries_left) {
    while (!__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity)) && tries_left > 0) --tries_left;
}
// One column of this thread's row, waited for.
__device__ __forceinline__ int tc_ld1(uint32_t taddr) {
    uint32_t v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;" : "=r"(v) : "r"(taddr) : "memory");
    return (int)v;
}
// Two fp32 FMAs with the same factor in one instruction: no more of them a clock than single ones, but half the issue slots.
__device__ __forceinline__ void fma_pair(float& a0, float& a1, float x0, float x1, float s) {
    asm("{\n\t.reg .b64 a, x, s;\n\t"
        "mov.b64 a, {%0, %1};\n\tmov.b64 x, {%2, %3};\n\tmov.b64 s, {%4, %4};\n\t"
        "fma.rn.f32x2 a, x, s, a;\n\tmov.b64 {%0, %1}, a;\n\t}"
        : "+f"(a0), "+f"(a1)
        : "f"(x0), "f"(x1), "f"(s));
}

// The code the next layer's quantizer gives the fp16 output value (static exponent; NaN -> 0), in the low byte. Clamped first,
// the value rounds to the nearest even integer by the addition of 1.5 * 2^23, whose low bits then hold it; the instructions
// for rounding and for conversion issue at an eighth of the rate.
__device__ __forceinline__ int chain_code(__half hv, float inv, float lo, float hi) {
    const float t = __half2float(hv) * inv;                 // exact: inv is a power of two
    const int code = __float_as_int(fminf(fmaxf(t, lo), hi) + 12582912.0f);
    return t == t ? code : 0;
}

// Chaining: a warp's 32 codes of one token (lane = channel) go to the staging row: one byte each, or, for
// packed 4-bit codes, the even lane stores its code and its neighbour's in one byte (rows of 16 bytes).
// All 32 lanes call this together.
__device__ __forceinline__ void stage_code(__half* stage, int c, int lane, int code, int packed) {
    if (packed) {
        const int hi = __shfl_down_sync(0xFFFFFFFFu, code, 1);
        if (!(lane & 1)) reinterpret_cast<uint8_t*>(stage)[c * 16 + (lane >> 1)] = (uint8_t)((code & 0xF) | (hi << 4));
    } else {
        reinterpret_cast<int8_t*>(stage)[c * 32 + lane] = (int8_t)code;
    }
}

// Staged fp16 rows (32 channels a token) become rows of codes in place, sixteen rows a turn: a lane takes eight channels of a
// row in one load and one store, twice. The codes take bytes of rows that this turn or an earlier one has read. (Unrolled behind
// the outputs' arithmetic, with a byte store per code, rounding and conversion instructions, chained layer calls took 10.7 us at
// 65 rows of 768 x 768 and 70.1 at 2048 of 4096 x 4096; 8.8 and 65.3 now; the plain calls take 8.1 and 62.9.)
template <int ROWS>
__device__ __forceinline__ void stage_codes(__half* stage, int lane, float inv, float lo, float hi, int packed) {
    static_assert(ROWS % 16 == 0, "sixteen rows a turn");
    uint8_t* src = reinterpret_cast<uint8_t*>(stage) + lane * 16;
    uint8_t* dst = reinterpret_cast<uint8_t*>(stage) + lane * (packed ? 4 : 8);
#pragma unroll 1
    for (int turn = 0; turn < ROWS / 16; ++turn) {
        uint4 d[2];
        uint2 w[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) d[u] = *reinterpret_cast<const uint4*>(src + 512 * u);
        src += 1024;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const __half2* h = reinterpret_cast<const __half2*>(&d[u]);
            uint32_t c[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) c[i] = (uint32_t)chain_code(i & 1 ? __high2half(h[i >> 1]) : __low2half(h[i >> 1]), inv, lo, hi);
            w[u].x = __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
            w[u].y = __byte_perm(__byte_perm(c[4], c[5], 0x0040), __byte_perm(c[6], c[7], 0x0040), 0x5410);
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (packed) {
                // nibbles of the even and the odd bytes, a code pair a byte
                const uint32_t p0 = (w[u].x & 0x000F000Fu) | ((w[u].x >> 4) & 0x00F000F0u);
                const uint32_t p1 = (w[u].y & 0x000F000Fu) | ((w[u].y >> 4) & 0x00F000F0u);
                *reinterpret_cast<uint32_t*>(dst) = __byte_perm(p0, p1, 0x6420);
                dst += 128;
            } else {
                *reinterpret_cast<uint2*>(dst) = w[u];
                dst += 256;
            }
        }
        __syncwarp();
    }
}

// OFFSET: add the per-channel term of the zero-point variant. CHAIN: write the next layer's codes
// instead of fp16 outputs. Separate instantiations, so that the code of the plain kernels does not
// change with them. SPLIT (per-group scales only): the launch covers the tiles of a last, partial round;
// every tile is shared by two CTAs that take half of the k range each, leave fp32 partial sums in
// scratch, and whichever epilogue warp arrives second adds the other's sums and writes the outputs
// (nobody waits). CLUSTER: tiles so few that all of them run at once in clusters of two to eight
// CTAs (up to a few hundred rows on narrow layers). The CTAs of a cluster share a tile and take consecutive ranges of its
// k blocks; every epilogue warp sends the sums (fp32 with per-group scales, otherwise integers) of the token runs that
// another CTA finishes into that CTA's operand ring (idle by then), the cluster meets, and each adds what it received to
// its own in the order of the senders' ranks.
template <int BM, bool GROUPED, bool OFFSET, bool CHAIN, bool SPLIT = false, bool CLUSTER = false>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tensor_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap y_map,
                   const TensorParams p) {
    extern __shared__ uint8_t smem_raw[];
    using R = Roles<BM, GROUPED>;
    constexpr int kEpiWarps = R::kEpiWarps, kFirstEpiWarp = R::kFirstEpiWarp, kRegsEpilogue = R::kRegsEpilogue;
    using Smem = SharedStorage<BM, kEpiWarps>;
    Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);

    constexpr int kNumStages = TileConfig<BM>::kNumStages;
    // accumulator stages in tensor memory: three for per-group rescaling, otherwise as many
    // 2 (or 1 for the 256-token tile) as leave room for the weight-slice ring
    constexpr int kNumAcc = GROUPED ? (BM > 128 ? 2 : 3) : (BM >= 256 ? 1 : 2);
    constexpr int kAccStride = BM;                    // columns between accumulator stages
    constexpr int kAccCols = kNumAcc * kAccStride;
    // the rest of tensor memory (up to 8 slices) is the ring of unpacked weight slices (A operand)
    constexpr int kNumASlices = (512 - kAccCols) / kAColsPerStage >= 8 ? 8 : (512 - kAccCols) / kAColsPerStage;
    static_assert(kNumASlices >= 4 && kNumASlices % kUnpackGroups == 0, "weight-slice ring");
    static_assert(!GROUPED || kNumAcc <= 3, "the scale ring's depth assumes at most three accumulator stages");
    constexpr int kTmemColsUsed = kAccCols + kNumASlices * kAColsPerStage;
    constexpr int kTmemCols = kTmemColsUsed <= 128 ? 128 : kTmemColsUsed <= 256 ? 256 : 512;
    static_assert(kTmemColsUsed <= 512, "tensor memory has 512 columns");
    static_assert(BM % 32 == 0 && BM >= 64 && BM <= 256, "token tile");
    // Which epilogue warps share the watcher's barrier. Twelve: the four of a third of the columns, one on each scheduler, so that the
    // three warps of a scheduler may be at different places of their blocks (with the three of a lane quarter, which share a scheduler,
    // K, N = 4096, 4096 / 4096, 11008 / 11008, 4096 at M = 2048 take 61.3 / 125.8 / 131.9 us, so 60.5 / 123.3 / 129.6). Eight: the two of a lane
    // quarter (by halves 509 x 4096 x 4096 with a zero point 22.3 -> 23.0).
    constexpr int kMeetGroups = kEpiWarps == 12 ? 3 : 4;
    constexpr int kColsPerEpiWarp = R::kColsPerEpiWarp;   // each quarter's columns are split between two or three warps
    static_assert(kColsPerEpiWarp % 16 == 0 && (!GROUPED || kColsPerEpiWarp % 32 == 0), "epilogue chunking");

    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int KB = k_blocks(p.K);      // a last block that K does not fill: zero weight codes meet the tensor map's zero fill
    static_assert(!SPLIT || (GROUPED && !OFFSET), "tiles of a last round are shared with per-group scales, without a zero point");
    static_assert(!CLUSTER || (!SPLIT && BM <= 192), "what a CTA receives fits its operand ring");
    const int rank = CLUSTER ? (int)blockIdx.x : 0, split = CLUSTER ? (int)gridDim.x : 1;
    [[maybe_unused]] int met = 0;                    // CLUSTER: meetings this warp has been to
    auto tile_at = [&](int tl) {
        return CLUSTER ? (int)blockIdx.y : SPLIT ? p.split_base + ((int)blockIdx.x >> 1) : (int)(blockIdx.x + tl * gridDim.x);
    };
    const int my_tiles = SPLIT || CLUSTER ? 1
                               : (p.n_tiles > (int)blockIdx.x
                                      ? (p.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0);
    // the k blocks of a work item: all of them, or a range of them when the tile is shared
    const int kb_first = CLUSTER ? KB * rank / split : SPLIT ? (((int)blockIdx.x & 1) ? KB / 2 : 0) : 0;
    const int kb_last = CLUSTER ? KB * (rank + 1) / split : SPLIT ? (((int)blockIdx.x & 1) ? KB : KB / 2) : KB;

    if (p.clear_status && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) p.ctl->status = 0;   // nothing has given up yet
    if (threadIdx.x == 0) {
        for (int s = 0; s < kNumStages; ++s) {
            mbar_init(&sm.tma_full[s], 2);
            mbar_init(&sm.smem_empty[s], 1);
        }
        for (int i = 0; i < kNumASlices; ++i) {
            mbar_init(&sm.a_full[i], 4);
            mbar_init(&sm.a_empty[i], 1);
        }
        for (int a = 0; a < kNumAcc; ++a) {
            mbar_init(&sm.acc_full[a], 1);
            mbar_init(&sm.acc_empty[a], kEpiWarps);
        }
        sm.abort_flag = 0;
        sm.given_up = -1;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sm.tmem_base)), "r"((uint32_t)kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    const uint32_t tmem_acc = tmem;                 // columns [0, kNumAcc*BM)
    const uint32_t tmem_a = tmem + kAccCols;        // then kNumASlices slices of 32 columns
    volatile uint32_t* abort_flag = &sm.abort_flag;

    if (warp < kFirstUnpackWarp) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsControl));
      if (warp == 0 || warp == 2) {
        // ------------- TMA producers: warp 0 streams activation tiles, warp 2 weight blocks (+ scales)
        if (elect_one()) {
            // Launched behind the call's own quantize kernel with programmatic stream serialization, this
            // grid is set up while that one drains: the codes (and, in the epilogue, the exponent and the
            // offsets) are touched only after it has completed; the weight producer does not wait. A no-op
            // for a normal launch.
            // Ring positions are carried in counters and addresses are shared-memory words: one thread whose every
            // instruction waits for the one before paces this loop.
            uint32_t st = 0, ph = 1u;
            const uint32_t full0 = smem_u32(sm.tma_full), empty0 = smem_u32(sm.smem_empty);
            if (warp == 0) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                const uint32_t x0 = smem_u32(sm.x[0]);
                for (int tl = 0; tl < my_tiles; ++tl) {
                    const int tile = tile_at(tl);
                    const int m0 = tile % p.n_tiles_m * BM;
                    for (int k = kb_first * kTileK; k < kb_last * kTileK; k += kTileK) {
                        if (!mbar_wait_a(empty0 + 8u * st, ph, abort_flag, 1u, p.wait_cycles)) goto role_done;
                        mbar_arrive_expect_tx_a(full0 + 8u * st, BM * 128);
                        tma_load_2d_a(x0 + st * (uint32_t)(BM * 128), &x_map, k, m0, full0 + 8u * st);
                        if (++st == (uint32_t)kNumStages) { st = 0; ph ^= 1u; }
                    }
                }
            } else {
                const uint32_t w0 = smem_u32(sm.w[0]), sc0 = smem_u32(sm.sc[0]);
                uint32_t slot = 0;
                for (int tl = 0; tl < my_tiles; ++tl) {
                    const int tile = tile_at(tl);
                    const int nt = tile / p.n_tiles_m;
                    const uint8_t* wsrc = p.w_packed + ((size_t)nt * KB + kb_first) * kBlockBytes;
                    const __half* ssrc = p.w_scales + (size_t)kb_first * p.Npad + nt * kTileN;
                    for (int kb = kb_first; kb < kb_last; ++kb) {
                        if (!mbar_wait_a(empty0 + 8u * st, ph, abort_flag, 1u, p.wait_cycles)) goto role_done;
                        mbar_arrive_expect_tx_a(full0 + 8u * st, kBlockBytes + (GROUPED ? kTileN * 2 : 0));
                        tma_load_1d_a(w0 + st * (uint32_t)kBlockBytes, wsrc, kBlockBytes, full0 + 8u * st);
                        wsrc += kBlockBytes;
                        if (GROUPED) {
                            tma_load_1d_a(sc0 + slot * (uint32_t)(kTileN * 2), ssrc, kTileN * 2, full0 + 8u * st);
                            ssrc += p.Npad;
                            if (++slot == (uint32_t)Smem::kNumScaleSlots) slot = 0;
                        }
                        if (++st == (uint32_t)kNumStages) { st = 0; ph ^= 1u; }
                    }
                }
            }
        }
      } else {
        if (GROUPED && warp == 3) {
            // ------------- watcher: tells the epilogue warps, through named barriers of an accumulator stage (one a column third or lane quarter: kMeetGroups),
            // that an accumulation is complete. A look at an mbarrier costs a warp some 200 cycles in this kernel even where
            // the phase is long over, a named barrier some 30, and the epilogue's chain per block sets the pace (K, N = 4096,
            // 11008 at M = 2048: 124 -> 120 us).
            // A stage's barrier is not arrived at again before its warps have come by: the next accumulation in it needs
            // their release.
            // Who can give up here, and raise the flag: the two producers (1), the MMA issuer (2, 3), the unpack warps (6, 7)
            // and this warp (9). The first three only stop: what they would have made never comes, and this warp sees the
            // flag, or its own limit, in its wait for it. So it alone decides. The epilogue warps, which wait without a
            // limit, never look at the flag; once a wait here has ended without its phase they get the rest of the tile's arrivals
            // all the same, each behind their release of the stage's previous block, and before the tile's last arrival
            // the word that this tile is given up. It is written once and names the tile, so a warp that is still at
            // an earlier tile's end does not take it for its own. Behind that tile all of them leave, and so does this warp:
            // no barrier is left with a part of its warps, and the CTA is through a tile's worth of arrivals after the limit.
            // That the releases come rests on the epilogue warps waiting for no one but this warp, once the kernel ahead has
            // completed; so this warp waits for that kernel too before the first such arrival.
            uint32_t ph = 0;                                           // a bit per accumulator stage
            bool live = true;
            auto tell = [&](uint32_t a) {
                tc_fence_after();
                tc_fence_before();
#pragma unroll
                for (int g = 0; g < kMeetGroups; ++g)
                    asm volatile("bar.arrive %0, %1;" ::"r"(1 + g * kNumAcc + (int)a), "n"(32 + kEpiWarps * 32 / kMeetGroups) : "memory");
                ph ^= 1u << a;
            };
            for (int tl = 0; tl < my_tiles && live; ++tl) {
                uint32_t a = 0;
                int kb = kb_first;
                for (; kb < kb_last; ++kb) {
                    live = mbar_wait_warp(&sm.acc_full[a], (ph >> a) & 1u, abort_flag, 9u, p.wait_cycles);
                    if (!live) break;
                    tell(a);
                    if (++a == (uint32_t)kNumAcc) a = 0;
                }
                if (!live) {
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    uint32_t tries_left = kDrainTries;
                    for (; kb < kb_last; ++kb) {
                        drain_wait(&sm.acc_empty[a], ((ph >> a) & 1u) ^ 1u, tries_left);
                        if (kb == kb_last - 1 && lane == 0) sm.given_up = tl;
                        __syncwarp();
                        tell(a);
                        if (++a == (uint32_t)kNumAcc) a = 0;
                    }
                }
            }
        }
        // ------------- MMA issuer (one thread: a second one taking the odd k blocks of per-group products changes nothing
        // since both are elected threads)
        if (warp == 1 && elect_one()) {
            constexpr uint32_t idesc = idesc_i8(128, BM);
            if (GROUPED) {
                // Every k block is one accumulation into its own accumulator stage; a tile's first block takes stage 0. Ring
                // positions and phases are carried in counters: the divisions that gave them from the block's number
                // were most of this loop, one thread whose every instruction waits for the one before.
                uint32_t st = 0, ai = 0, a_ph = 0u, acc_ph = ~0u;             // acc_ph: a bit per accumulator stage
                const uint64_t bdesc0 = smem_desc_sw128(smem_u32(sm.x[0]));
                for (int tl = 0; tl < my_tiles; ++tl) {
                    uint32_t a = 0;
                    for (int kb = kb_first; kb < kb_last; ++kb) {
                        const uint32_t a_bit = (acc_ph >> a) & 1u;
                        const bool got_a = mbar_try_wait(&sm.a_full[ai], a_ph);       // both asked before either answer is used
                        const bool got_acc = mbar_try_wait(&sm.acc_empty[a], a_bit);
                        if (!got_acc && !mbar_wait(&sm.acc_empty[a], a_bit, abort_flag, 2u, p.wait_cycles)) goto role_done;
                        if (!got_a && !mbar_wait(&sm.a_full[ai], a_ph, abort_flag, 3u, p.wait_cycles)) goto role_done;
                        tc_fence_after();
                        const uint32_t d_addr = tmem_acc + a * (uint32_t)kAccStride;
                        const uint32_t a_addr = tmem_a + ai * (uint32_t)kAColsPerStage;
                        const uint64_t bdesc = bdesc0 + (uint64_t)(st * (uint32_t)(BM * 128 / 16));
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            tc_mma_i8_ts(d_addr, a_addr + 8 * j, bdesc + (uint64_t)(2 * j), idesc, j > 0 ? 1u : 0u);
                        tc_commit(&sm.acc_full[a]);
                        tc_commit(&sm.a_empty[ai]);
                        tc_commit(&sm.smem_empty[st]);
                        acc_ph ^= 1u << a;
                        if (++a == (uint32_t)kNumAcc) a = 0;
                        if (++st == (uint32_t)kNumStages) st = 0;
                        if (++ai == (uint32_t)kNumASlices) { ai = 0; a_ph ^= 1u; }
                    }
                }
            } else {
                uint32_t st = 0, ai = 0, a_ph = 0u;
                const uint64_t bdesc0 = smem_desc_sw128(smem_u32(sm.x[0]));
                for (int tl = 0; tl < my_tiles; ++tl) {
                    const int a = (int)((uint32_t)tl % kNumAcc);
                    const uint32_t aph = ((uint32_t)tl / kNumAcc) & 1u;
                    if (!mbar_wait(&sm.acc_empty[a], aph ^ 1u, abort_flag, 4u, p.wait_cycles)) goto role_done;
                    const uint32_t d_addr = tmem_acc + (uint32_t)(a * kAccStride);
                    uint32_t accumulate = 0u;
                    for (int kb = kb_first; kb < kb_last; ++kb) {
                        // the unpack warps publish a slice only after the stage's TMA bytes (activation
                        // tile included) have landed, so this one wait covers both operands
                        if (!mbar_wait(&sm.a_full[ai], a_ph, abort_flag, 5u, p.wait_cycles)) goto role_done;
                        tc_fence_after();
                        const uint32_t a_addr = tmem_a + ai * (uint32_t)kAColsPerStage;
                        const uint64_t bdesc = bdesc0 + (uint64_t)(st * (uint32_t)(BM * 128 / 16));
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            // 32 k per instruction: 8 TMEM columns of A, 32 bytes along the swizzled row of B
                            tc_mma_i8_ts(d_addr, a_addr + 8 * j, bdesc + (uint64_t)(2 * j), idesc, accumulate);
                            accumulate = 1u;
                        }
                        tc_commit(&sm.a_empty[ai]);
                        tc_commit(&sm.smem_empty[st]);
                        if (++st == (uint32_t)kNumStages) st = 0;
                        if (++ai == (uint32_t)kNumASlices) { ai = 0; a_ph ^= 1u; }
                    }
                    tc_commit(&sm.acc_full[a]);
                }
            }
        }
      }
    } else if (warp < kFirstEpiWarp) {
        // --------------------------------------------------- weight unpack -> tensor memory
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsUnpack));
        const int quarter = warp & 3;
        const int group = (warp - kFirstUnpackWarp) >> 2;
        const int r = quarter * 32 + lane;            // row inside the 128-channel tile = TMEM lane
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const uint32_t total_iters = (uint32_t)my_tiles * (uint32_t)(kb_last - kb_first);
        int pending = -1;                             // slice whose store has been issued but not published
        // Per-group kernels on 192-token tiles have one group of unpack warps: the epilogue sets the pace there, and a second group
        // (four warps more, 120 registers for the epilogue) wins 0.5 % at M = 2048. On 128-token tiles the second group shortens the
        // block: 509 x 11008 x 4096 with a zero point 44.4 -> 43.0 us, 333 x 5120 x 5120 25.1 -> 24.7.
        constexpr int kActiveGroups = GROUPED && BM > 128 ? 1 : kUnpackGroups;
        if (group >= kActiveGroups) goto role_done;
        uint32_t s = (uint32_t)group, s_ph = 0u, ai = (uint32_t)group, a_ph = 1u;
        for (uint32_t it = group; it < total_iters; it += kActiveGroups) {
            if (!mbar_wait_warp(&sm.tma_full[s], s_ph, abort_flag, 6u, p.wait_cycles)) goto role_done;
            const uint4* src = reinterpret_cast<const uint4*>(sm.w[s]) + r;
            uint4 d[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) d[j] = src[j * kTileN];
            if (pending >= 0) {                       // the previous stores had the loads above to finish
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.a_full[pending]);
            }
            if (!mbar_wait_warp(&sm.a_empty[ai], a_ph, abort_flag, 7u, p.wait_cycles)) goto role_done;
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
            s += kActiveGroups;
            if (s >= (uint32_t)kNumStages) { s -= kNumStages; s_ph ^= 1u; }
            ai += kActiveGroups;
            if (ai >= (uint32_t)kNumASlices) { ai -= kNumASlices; a_ph ^= 1u; }
        }
        if (pending >= 0) {
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.a_full[pending]);
        }
    } else {
        // ----------------------------------------------------------------------- epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpilogue));
        const int quarter = warp & 3;
        const int half = (warp - kFirstEpiWarp) >> 2;                                // which half (third) of the token columns
        const int r = quarter * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const int col0 = half * kColsPerEpiWarp;
        [[maybe_unused]] const int meet_group = kMeetGroups == 4 ? quarter : half;
        asm volatile("griddepcontrol.wait;" ::: "memory");               // see the activation producer
        const float pe = __int_as_float((127 + *p.scale_exp) << 23);     // 2^e
        [[maybe_unused]] const float off_factor = OFFSET ? offset_factor(p.ctl, p.zp_mid) : 0.0f;
        [[maybe_unused]] const int G = GROUPED ? KB : 1;
        uint32_t unit = 0;
        // per-group mode: the next block's scale, the lane that releases a stage. (The scale is read from a shared-memory
        // address: stepped as a pointer it was read with generic loads, 5 % of the kernel's time.)
        [[maybe_unused]] uint32_t sc_addr = smem_u32(&sm.sc[0][r]);
        [[maybe_unused]] const uint32_t sc_end = sc_addr + Smem::kNumScaleSlots * kTileN * 2;
        [[maybe_unused]] const bool releases = elect_one();
        [[maybe_unused]] const uint32_t acc_empty0 = smem_u32(sm.acc_empty);
        [[maybe_unused]] const uint32_t taddr0 = __shfl_sync(0xFFFFFFFFu, tmem_acc + lane_addr + (uint32_t)col0, 0);
        // CLUSTER: a warp's columns in runs of four tokens, run c finished by CTA c * split / kRuns; a CTA receives (its own share
        // too) at [sender][epilogue warp][run of its slice][lane], four tokens of a channel (16 bytes) a slot, in its operand
        // ring. The loops over a CTA's own runs are rolled: this code runs once, and what it costs is mostly fetching it
        // (with the runs unrolled K = N = 4096 at 200 rows took 1.4 us longer).
        constexpr int kRuns = kColsPerEpiWarp / 4, kSlot = kEpiWarps * 512, kRing = kNumStages * (BM * 128 + kBlockBytes);
        static_assert(!CLUSTER || (2 * kSlot * ((kRuns + 1) / 2) <= kRing && 3 * kSlot * ((kRuns + 2) / 3) <= kRing &&
                                   4 * kSlot * ((kRuns + 3) / 4) <= kRing && 5 * kSlot * ((kRuns + 4) / 5) <= kRing &&
                                   6 * kSlot * ((kRuns + 5) / 6) <= kRing && 7 * kSlot * ((kRuns + 6) / 7) <= kRing &&
                                   8 * kSlot * ((kRuns + 7) / 8) <= kRing),
                      "the operand ring (activation tiles, then weight blocks) holds what a CTA receives");
        [[maybe_unused]] const int slice_runs = (kRuns + split - 1) / split;
        [[maybe_unused]] const int run_first = (rank * kRuns + split - 1) / split, run_last = ((rank + 1) * kRuns + split - 1) / split;
        [[maybe_unused]] uint4* ring = reinterpret_cast<uint4*>(&sm) + (warp - kFirstEpiWarp) * slice_runs * 32 + lane;
        [[maybe_unused]] auto send_run = [&](int c, uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3) {
            const int owner = (c * split) / kRuns, first = (owner * kRuns + split - 1) / split;
            *(cg::this_cluster().map_shared_rank(ring, owner) + (rank * kEpiWarps * slice_runs + c - first) * 32) = make_uint4(v0, v1, v2, v3);
        };
        [[maybe_unused]] auto whole_run = [&](int c) {
            uint4 o = ring[(c - run_first) * 32];
#pragma unroll 1
            for (int from = 1; from < split; ++from) {
                const uint4 g = ring[(from * kEpiWarps * slice_runs + c - run_first) * 32];
                if (GROUPED) {
                    o.x = __float_as_uint(__uint_as_float(o.x) + __uint_as_float(g.x));
                    o.y = __float_as_uint(__uint_as_float(o.y) + __uint_as_float(g.y));
                    o.z = __float_as_uint(__uint_as_float(o.z) + __uint_as_float(g.z));
                    o.w = __float_as_uint(__uint_as_float(o.w) + __uint_as_float(g.w));
                } else {
                    o.x += g.x; o.y += g.y; o.z += g.z; o.w += g.w;
                }
            }
            return o;
        };
        // ... and the output of one token of such a run (all lanes of the warp together)
        [[maybe_unused]] auto put = [&](int m, int n, bool n_ok, __half hv) {
            if constexpr (CHAIN) {
                const int code = chain_code(hv, p.next_inv, p.next_lo, p.next_hi);
                const int hi = __shfl_down_sync(0xFFFFFFFFu, code, 1);
                if (n_ok && m < p.M) {
                    if (!p.next_packed) p.q_next[(size_t)m * p.N + n] = (int8_t)code;
                    else if (!(lane & 1)) p.q_next[((size_t)m * p.N + n) >> 1] = (int8_t)((code & 0xF) | (hi << 4));
                }
            } else if (n_ok && m < p.M) {
                p.y[(size_t)m * p.N + n] = hv;
            }
        };
        for (int tl = 0; tl < my_tiles; ++tl) {
            const int tile = tile_at(tl);
            const int mt = tile % p.n_tiles_m, nt = tile / p.n_tiles_m;
            const int n = nt * kTileN + r;
            const int m_base = mt * BM + col0;
            const bool n_ok = n < p.N;
            if constexpr (!GROUPED) {
                const int a = (int)(unit % kNumAcc);
                const uint32_t aph = (unit / kNumAcc) & 1u;
                const float sc = __half2float(p.w_scales[n]) * 0.0625f * pe;   // sums carry a factor 16
                [[maybe_unused]] float off_pe = 0.0f;
                if constexpr (OFFSET) off_pe = (n_ok ? __fmul_rn(off_factor, p.chan_offset[n]) : 0.0f) * pe;
                if (!mbar_wait_warp(&sm.acc_full[a], aph, abort_flag, 8u, p.wait_cycles)) goto role_done;
                tc_fence_after();
                // all of this warp's sums go to registers and the accumulator returns to the MMA at once,
                // so that the conversion and the stores below overlap the next tile's MMAs
                uint32_t v[kColsPerEpiWarp];
#pragma unroll
                for (int c0 = 0; c0 < kColsPerEpiWarp; c0 += 32)
                    tc_ld32(tmem_acc + lane_addr + (uint32_t)(a * kAccStride + col0 + c0), *reinterpret_cast<uint32_t(*)[32]>(&v[c0]));
                tc_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.acc_empty[a]);
                if constexpr (CLUSTER) {
                    cluster_meet();                                      // every CTA's operand ring is idle
#pragma unroll
                    for (int c = 0; c < kRuns; ++c)
                        if (m_base + 4 * c < p.M) send_run(c, v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
                    cluster_meet();                                      // all sums have arrived; nobody writes here any more
                    met = 2;
#pragma unroll 1
                    for (int c = run_first; c < run_last && m_base + 4 * c < p.M; ++c) {
                        const uint4 o = whole_run(c);
                        const int sums[4] = {(int)o.x, (int)o.y, (int)o.z, (int)o.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int m = m_base + 4 * c + i;
                            put(m, n, n_ok, __float2half_rn(OFFSET ? fmaf((float)sums[i], sc, off_pe) : (float)sums[i] * sc));
                            if (p.acc_dump && n_ok && m < p.M) p.acc_dump[(size_t)m * p.N + n] = sums[i] >> 4;
                        }
                    }
                    goto role_done;
                }
                if (p.y_tma) {
                    __half* stage = &sm.ystage[warp - kFirstEpiWarp][0][0];
                    const int n0 = nt * kTileN + quarter * 32;
#pragma unroll
                    for (int r0 = 0; r0 < kColsPerEpiWarp; r0 += Smem::kStageRows) {
                        if (lane == 0) tma_store_wait_read();     // the previous store has read the staging rows
                        __syncwarp();
#pragma unroll
                        for (int c = 0; c < Smem::kStageRows; ++c) {
                            const __half hv = __float2half_rn(OFFSET ? fmaf((float)(int)v[r0 + c], sc, off_pe)
                                                                     : (float)(int)v[r0 + c] * sc);
                            if constexpr (CHAIN)
                                stage_code(stage, c, lane, chain_code(hv, p.next_inv, p.next_lo, p.next_hi), p.next_packed);
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
                    for (int c = 0; c < kColsPerEpiWarp; ++c) {
                        const int m = m_base + c;
                        if (n_ok && m < p.M) {
                            const __half hv =
                                __float2half_rn(OFFSET ? fmaf((float)(int)v[c], sc, off_pe) : (float)(int)v[c] * sc);
                            if constexpr (CHAIN)
                                p.q_next[(size_t)m * p.N + n] = (int8_t)chain_code(hv, p.next_inv, p.next_lo, p.next_hi);
                            else
                                p.y[(size_t)m * p.N + n] = hv;
                        }
                    }
                }
                if (p.acc_dump) {
#pragma unroll
                    for (int c = 0; c < kColsPerEpiWarp; ++c) {
                        const int m = m_base + c;
                        if (n_ok && m < p.M) p.acc_dump[(size_t)m * p.N + n] = (int)v[c] >> 4;
                    }
                }
                ++unit;
            } else {
                float fsum[kColsPerEpiWarp];                             // fp32 partial outputs
#pragma unroll
                for (int c = 0; c < kColsPerEpiWarp; ++c) fsum[c] = 0.0f;
                // One k block, in accumulator stage `a`. Unrolled over the stages, so that a block's barriers and columns are
                // constants beside a few registers, and with its releasing lane chosen before the loop, a block takes a warp
                // some fifteen instructions less of what is not arithmetic (with the watcher, K, N = 4096, 4096 / 4096, 11008 at
                // M = 2048 58.9 / 127.0 -> 56.1 / 120.5 us). What a block costs an epilogue warp, in
                // cycles: the named barrier and the loop 100, the first load with the scale 130, the second with the release 150, and
                // 460 of conversions and FMAs, which the three warps of a scheduler want at the same time.
                auto block = [&](const uint32_t a, int kb) {
                    asm volatile("bar.sync %0, %1;" ::"r"(1 + meet_group * kNumAcc + (int)a), "n"(32 + kEpiWarps * 32 / kMeetGroups) : "memory");   // the watcher's word
                    tc_fence_after();
                    // This block's MMAs are complete, so its stage (scales included) had landed: the
                    // issuer saw the unpack warps' signal, which they gave after seeing the TMA barrier.
                    const float sg = __half2float(ld_shared_half(sc_addr)) * 0.0625f;
                    sc_addr += kTileN * 2;
                    if (sc_addr == sc_end) sc_addr -= Smem::kNumScaleSlots * kTileN * 2;
                    static_assert(kColsPerEpiWarp == 32 || kColsPerEpiWarp == 64, "epilogue register plan");
                    const uint32_t taddr = taddr0 + a * (uint32_t)kAccStride;
                    if (p.acc_dump) {
                        // a rolled loop of its own: unrolled with the arithmetic below, the code of these stores (run only
                        // by tests) kept pushing the loop out of the instruction cache
#pragma unroll 1
                        for (int c = 0; c < kColsPerEpiWarp; ++c) {
                            const int sum = tc_ld1(taddr + (uint32_t)c);
                            if (n_ok && m_base + c < p.M) p.acc_dump[((size_t)(m_base + c) * p.N + n) * G + kb] = sum >> 4;
                        }
                    }
                    // With twelve epilogue warps (128 registers each) a warp's 64 columns pass through one
                    // 32-register buffer in two turns; otherwise all of them are loaded at once.
                    constexpr int kLdCols = (kEpiWarps == 12 && kColsPerEpiWarp == 64) ? 32 : kColsPerEpiWarp;
#pragma unroll
                    for (int c0 = 0; c0 < kColsPerEpiWarp; c0 += kLdCols) {
                        uint32_t v[kLdCols];
                        tc_ld32(taddr + c0, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
                        if (kLdCols == 64) tc_ld32(taddr + c0 + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32 % kLdCols]));
                        tc_wait_ld();
                        if (c0 + kLdCols == kColsPerEpiWarp) {
                            // the sums are in registers: the accumulator stage goes back to the MMA at once
                            tc_fence_before();
                            __syncwarp();
                            if (releases) mbar_arrive_a(acc_empty0 + 8u * a);
                        }
#pragma unroll
                        for (int c = 0; c < kLdCols; c += 2) {
                            // One conversion per element and one FMA per two. (An integer add of the bits of
                            // 1.5 * 2^23 plus a float subtract also converts, on the FMA and ALU pipes, but
                            // costs a third instruction; measured 8-16 % slower. Paired FMAs, the issuers' counters and
                            // the dump's code outside this loop: K, N = 4096, 4096 / 4096, 11008 / 11008, 4096 at
                            // M = 2048 65.1 / 139.2 / 137.5 -> 61.7 / 135.3 / 133.3 us.)
                            fma_pair(fsum[c0 + c], fsum[c0 + c + 1], (float)(int)v[c], (float)(int)v[c + 1], sg);
                        }
                    }
                };
                for (int kb = kb_first; kb < kb_last; kb += kNumAcc) {
#pragma unroll
                    for (int a = 0; a < kNumAcc; ++a)
                        if (kb + a < kb_last) block((uint32_t)a, kb + a);
                }
                if (__any_sync(0xFFFFFFFFu, sm.given_up == tl)) goto role_done;   // the watcher's word: these are not the tile's sums
                [[maybe_unused]] bool emit = true;
                if constexpr (SPLIT) {
                    const int ew = warp - kFirstEpiWarp, slot = (int)blockIdx.x >> 1, hf = (int)blockIdx.x & 1;
                    float* mine = p.split_scratch + ((size_t)(slot * 2 + hf) * kEpiWarps + ew) * (kColsPerEpiWarp * 32);
                    const float* other = p.split_scratch + ((size_t)(slot * 2 + (hf ^ 1)) * kEpiWarps + ew) * (kColsPerEpiWarp * 32);
#pragma unroll
                    for (int c = 0; c < kColsPerEpiWarp; ++c) __stcg(mine + c * 32 + lane, fsum[c]);
                    __threadfence();
                    __syncwarp();
                    const int bit_index = slot * kEpiWarps + ew;
                    unsigned int old = 0;
                    if (lane == 0) old = atomicOr(&p.ctl->split_flags[bit_index >> 5], 1u << (bit_index & 31));
                    old = __shfl_sync(0xFFFFFFFFu, old, 0);
                    emit = ((old >> (bit_index & 31)) & 1u) != 0;
                    if (emit) {
                        __threadfence();
#pragma unroll
                        for (int c = 0; c < kColsPerEpiWarp; ++c) fsum[c] += __ldcg(other + c * 32 + lane);
                    }
                }
                if constexpr (CLUSTER) {
                    cluster_meet();
#pragma unroll
                    for (int c = 0; c < kRuns; ++c)
                        if (m_base + 4 * c < p.M)
                            send_run(c, __float_as_uint(fsum[4 * c]), __float_as_uint(fsum[4 * c + 1]), __float_as_uint(fsum[4 * c + 2]),
                                     __float_as_uint(fsum[4 * c + 3]));
                    cluster_meet();
                    met = 2;
                    const float off_n = OFFSET && n_ok ? __fmul_rn(off_factor, p.chan_offset[n]) : 0.0f;
#pragma unroll 1
                    for (int c = run_first; c < run_last && m_base + 4 * c < p.M; ++c) {
                        const uint4 o = whole_run(c);
                        const float sums[4] = {__uint_as_float(o.x), __uint_as_float(o.y), __uint_as_float(o.z), __uint_as_float(o.w)};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            put(m_base + 4 * c + i, n, n_ok, __float2half_rn((OFFSET ? sums[i] + off_n : sums[i]) * pe));
                    }
                    goto role_done;
                }
                if constexpr (OFFSET) {                                  // read after the k loop
                    const float off_n = n_ok ? __fmul_rn(off_factor, p.chan_offset[n]) : 0.0f;
#pragma unroll
                    for (int c = 0; c < kColsPerEpiWarp; ++c) fsum[c] += off_n;
                }
                if (SPLIT && !emit) {
                    // the other CTA's warp writes this tile's outputs
                } else if (p.y_tma) {
                    static_assert(Smem::kStageRows == kColsPerEpiWarp, "per-group kernels stage a warp's whole tile");
                    // the previous tile's store must have read the staging rows before they change
                    __half* stage = &sm.ystage[warp - kFirstEpiWarp][0][0];
                    if (lane == 0) tma_store_wait_read();
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < kColsPerEpiWarp; ++c) stage[c * 32 + lane] = __float2half_rn(fsum[c] * pe);
                    if constexpr (CHAIN) {
                        __syncwarp();
                        stage_codes<kColsPerEpiWarp>(stage, lane, p.next_inv, p.next_lo, p.next_hi, p.next_packed);
                    }
                    fence_proxy_async();
                    __syncwarp();
                    const int n0 = nt * kTileN + quarter * 32;
                    if (lane == 0 && n0 < p.N && m_base < p.M)
                        tma_store_2d(&y_map, stage, (CHAIN && p.next_packed) ? n0 >> 1 : n0, m_base);
                } else {
#pragma unroll
                    for (int c = 0; c < kColsPerEpiWarp; ++c) {
                        const int m = m_base + c;
                        if (n_ok && m < p.M) {
                            const __half hv = __float2half_rn(fsum[c] * pe);
                            if constexpr (CHAIN)
                                p.q_next[(size_t)m * p.N + n] = (int8_t)chain_code(hv, p.next_inv, p.next_lo, p.next_hi);
                            else
                                p.y[(size_t)m * p.N + n] = hv;
                        }
                    }
                }
            }
        }
    }

role_done:
    if (warp >= kFirstEpiWarp && lane == 0) tma_store_wait_read();   // staging rows live until read
    __syncwarp();
    if constexpr (CLUSTER)
        for (; met < 2; ++met) cluster_meet();                       // every warp comes to both meetings
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (sm.abort_flag) {
        // Give copies that may still be in flight time to land before shared memory is released.
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
        if (threadIdx.x == 0) atomicCAS(&p.ctl->status, 0u, sm.abort_flag);   // the first CTA to give up names its wait
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kTmemCols)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// Rate probe: what this GPU's tensor cores deliver on kind::i8 when nothing else is in the way.
// One CTA per SM; one thread issues `iters` rounds of four 128 x 256 x 32 MMAs on operands that
// stay where they are (pseudo-random bytes, so that the data toggles as real codes do): both from
// shared memory, or A from tensor memory as in the product kernel. No loads, no epilogue. Batches
// of 32 rounds are committed to two alternating barriers and the issuer stays one batch ahead,
// so the pipe never drains and the queue stays bounded.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void tc_mma_i8_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

struct ProbeSmem {
    alignas(1024) uint8_t a[128 * 128];     // 128 rows x 128 k, 128-byte swizzled rows
    alignas(1024) uint8_t b[256 * 128];     // 256 rows x 128 k
    alignas(8) uint64_t bar[2];
    uint32_t tmem_base;
    volatile uint32_t abort_flag;
};

__global__ void __launch_bounds__(128, 1) int8_probe_kernel(int iters, int a_from_tmem, Control* ctl) {
    extern __shared__ uint8_t smem_raw[];
    ProbeSmem& sm = *reinterpret_cast<ProbeSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    uint32_t* words = reinterpret_cast<uint32_t*>(sm.a);
    for (int i = threadIdx.x; i < (int)(sizeof(sm.a) + sizeof(sm.b)) / 4; i += blockDim.x) {
        uint32_t v = (uint32_t)i * 2654435761u + blockIdx.x * 40503u;       // any bytes will do
        v ^= v >> 15; v *= 2246822519u; v ^= v >> 13;
        words[i] = v;
    }
    fence_proxy_async();
    if (threadIdx.x == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        sm.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sm.tmem_base)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    const uint32_t tmem_a = tmem + 256;            // after the 256 accumulator columns
    if (a_from_tmem) {                             // 128 lanes x 32 columns of bytes for the A operand
        uint32_t v[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = words[(threadIdx.x * 32 + j * 8 + i) & 4095];
            tc_st8(tmem_a + ((uint32_t)(warp * 32) << 16) + 8 * j, v);
        }
        tc_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0 && elect_one()) {
        constexpr uint32_t idesc = idesc_i8(128, 256);
        constexpr int kBatch = 32;
        const uint64_t adesc = smem_desc_sw128(smem_u32(sm.a)), bdesc = smem_desc_sw128(smem_u32(sm.b));
        const int batches = (iters + kBatch - 1) / kBatch;
        bool ok = true;
        for (int bt = 0; bt < batches && ok; ++bt) {
            if (bt >= 2) ok = mbar_wait(&sm.bar[bt & 1], (uint32_t)((bt >> 1) - 1) & 1u, &sm.abort_flag, 12u);
            if (!ok) break;
            const int n = min(kBatch, iters - bt * kBatch);
            for (int it = 0; it < n; ++it) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (a_from_tmem) tc_mma_i8_ts(tmem, tmem_a + 8 * j, bdesc + (uint64_t)(2 * j), idesc, 1u);
                    else tc_mma_i8_ss(tmem, adesc + (uint64_t)(2 * j), bdesc + (uint64_t)(2 * j), idesc, 1u);
                }
            }
            tc_commit(&sm.bar[bt & 1]);
        }
        // drain: the last one or two batches
        for (int bt = max(batches - 2, 0); bt < batches && ok; ++bt)
            ok = mbar_wait(&sm.bar[bt & 1], (uint32_t)(bt >> 1) & 1u, &sm.abort_flag, 12u);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (sm.abort_flag && threadIdx.x == 0) atomicCAS(&ctl->status, 0u, sm.abort_flag);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// Shared tiles pay from K = 8192 on with 64- and 128-token tiles and from K = 4096 on with 192-token
// tiles, where half a tile is worth more (see launch_bm).
constexpr int split_min_k_blocks(int bm) { return bm >= 192 ? 32 : 64; }

// Tiles of a last, partial round behind whole ones that are run as shared tiles (0: none). The plan, the launch and the size of
// the scratch all ask here.
inline int shared_tiles(long tiles, int sms, int k_blocks, int bm) {
    const int rem = (int)(tiles % sms);
    return tiles >= sms && 2 * rem <= sms && k_blocks >= split_min_k_blocks(bm) && rem <= Control::kMaxSplitTiles ? rem : 0;
}

// Clusters of `split` CTAs that run at once (one CTA fills an SM; a GPC holds only so many of a size).
template <int BM, bool GROUPED>
int tile_clusters(const DeviceInfo& dev, int split) {
    static std::atomic<int> known[kMaxDevices][9];               // + 1 (0: not asked yet)
    int k = known[dev.device][split].load(std::memory_order_relaxed);
    if (k == 0) {
        const size_t smem_bytes = sizeof(SharedStorage<BM, Roles<BM, GROUPED>::kEpiWarps>) + 1024;
        auto kernel = gemm_tensor_kernel<BM, GROUPED, false, false, false, true>;
        static SmemOptIn opt_in;
        int n = 0;
        if (opt_in.ensure(kernel, dev.device, smem_bytes) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(split, 1);
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = smem_bytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = split;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
                (void)cudaGetLastError();
                n = 0;
            }
        }
        k = n + 1;
        known[dev.device][split].store(k, std::memory_order_relaxed);
    }
    return k - 1;
}

// How a per-group product is run: token tile and CTAs that share a tile. Up to 64 tokens the tile is 64. Otherwise 128 (eight
// epilogue warps, three accumulator stages) or 192 (twelve epilogue warps, two stages), whichever gives the shorter schedule:
// rounds of tiles over the SMs, a last round whose tiles two CTAs share, or all tiles at once in clusters, where the k blocks
// saved outweigh the exchange (layers of 48 rows, K x N = 4096 x 4096 14.3 -> 10.8 us, 11008 x 4096 21.9 -> 15.7 us, 5120 x 5120
// 17.6 -> 13.3 us; of 128 rows, 11008 x 4096 30.9 -> 22.5 us).
// The times were fitted to layer calls with every schedule forced, 131 layers of 65 to 3000 rows, 768 <= K <= 28672, 768 <= N <= 28672 (a
// layer's schedules against one another, in graph replay, those within 60 % of its best). The schedule taken is then 0.3 % slower than the
// best in the mean and 5 % at the worst; with the prices of before the last changes to these kernels it was 1.1 and 22 %
// (631 rows, 20480 x 6400: 159 us on 192-token tiles, 131 on 128). Up to 64 rows 0.8 and 9 %, refitted or not. On 126 other products of
// 65 to 3000 rows 0.4 and 7 %.
struct GroupedPlan {
    int bm, split;
};
struct GroupedTimes {                // microseconds
    float call, round, block;        // layer call; round of tiles, k block of it
    float shared, shared_block;      // a last round of shared tiles: launch and exchange, k block of half a tile
    float exchange, exchange_cta;    // clusters of two; each CTA more
};
constexpr GroupedTimes grouped_times(int bm) {
    return bm == 64 ? GroupedTimes{4.56f, 0.91f, 0.266f, 6.44f, 0.317f, 1.9f, 0.06f}
         : bm == 128 ? GroupedTimes{6.45f, 0.82f, 0.337f, 0.0f, 0.700f, 2.56f, 0.23f}
                     : GroupedTimes{6.68f, 1.28f, 0.416f, 4.99f, 0.678f, 3.17f, 0.19f};
}
// What the size of the workspace, which is part of the interface, goes by: the prices that it was first computed with.
constexpr GroupedTimes grouped_size_times(int bm) {
    return bm == 64 ? GroupedTimes{4.56f, 0.91f, 0.266f, 6.44f, 0.317f, 1.9f, 0.06f}
         : bm == 128 ? GroupedTimes{6.45f, 0.96f, 0.440f, 8.05f, 0.423f, 2.9f, 0.14f}
                     : GroupedTimes{6.63f, 1.47f, 0.499f, 9.23f, 0.523f, 3.85f, 0.41f};
}
size_t shared_scratch_bytes(long rem, int bm) { return (size_t)rem * 2 * bm * kTileN * sizeof(float); }
// scratch_bytes: what there is for shared tiles.
GroupedPlan grouped_plan(int M, int K, int N, const DeviceInfo& dev, size_t scratch_bytes, bool clusters, GroupedTimes (*times)(int) = grouped_times) {
    const int kbs = K / kTileK, n_tiles_n = round_up(N, kTileN) / kTileN, sms = dev.sm_count;
    GroupedPlan best = {64, 1};
    float best_time = 3.0e38f;
    auto consider = [&](int bm) {
        const GroupedTimes t = times(bm);
        const long tiles = (long)((M + bm - 1) / bm) * n_tiles_n, rem = shared_tiles(tiles, sms, kbs, bm);
        const bool halves = rem > 0 && shared_scratch_bytes(rem, bm) <= scratch_bytes;
        const long rounds = halves ? tiles / sms : (tiles + sms - 1) / sms;
        const float plain = t.call + (float)rounds * (t.round + (float)kbs * t.block) +
                            (halves ? t.shared + (float)((kbs + 1) / 2) * t.shared_block : 0.0f);
        if (plain < best_time) { best_time = plain; best = {bm, 1}; }
        if (!clusters) return;
        for (int s = 2; s <= 8 && s <= kbs && s * tiles <= sms; ++s) {
            const float shared = t.call + t.round + (float)((kbs + s - 1) / s) * t.block + t.exchange + (float)(s - 2) * t.exchange_cta;
            if (shared >= best_time) continue;
            const int fit = bm == 64 ? tile_clusters<64, true>(dev, s) : bm == 128 ? tile_clusters<128, true>(dev, s) : tile_clusters<192, true>(dev, s);
            if (fit >= tiles) { best_time = shared; best = {bm, s}; }
        }
    };
    if (M <= 64) {
        consider(64);
    } else {
        consider(128);
        consider(192);
    }
    return best;
}

// One scale per channel, tiles of one channel block: 64 tokens up to 64 rows, else 128 or (beyond 128 rows) 256 in rounds over the SMs, or
// all 64- or 128-token tiles at once in clusters, where the k blocks saved outweigh the exchange. Prices in nanoseconds, fitted together
// with those of the tiles of two channel blocks (wide_plan) as the per-group ones were, 174 layers of 17 to 3000 rows: beyond
// 64 rows the schedule taken is 0.2 % slower than the best in the mean, 7 % at the worst, where it was 2.8 and 33 % (186 rows of 1312 x 1312
// 10.2 us in clusters, 8.3 on whole tiles; 705 rows of 3648 x 9056 34.8 us on 256 tokens, 30.1 on 128). On 294 other products, 65 to 3000 rows,
// K and N from 512 to 14000 to the 32: 0.8 % in the mean, 15 % at the worst (946 rows of 6944 x 704 14.6 us, 12.6 on 128-token tiles in pairs).
struct ChannelPlan {
    int bm, split;
    long cost;
};
ChannelPlan channel_plan(int M, int K, int N, const DeviceInfo& dev) {
    const bool small = M <= 64;
    const int KB = k_blocks(K), sms = dev.sm_count, bm = small ? 64 : 128;
    const int round = small ? 0 : 1000, block = small ? 117 : 179, exchange = small ? 1380 : 2723, exchange_cta = small ? 28 : 92;
    const long blocks_n = round_up(N, kTileN) / kTileN, tiles = (M + bm - 1) / bm * blocks_n;
    ChannelPlan best = {bm, 1, (tiles + sms - 1) / sms * (round + (long)KB * block)};
    if (M > 128) {
        const long c = ((M + 255) / 256 * blocks_n + sms - 1) / sms * (1522 + (long)KB * 354);
        if (c < best.cost) best = {256, 1, c};
    }
    for (int s = 2; s <= 8 && s <= KB && s * tiles <= sms; ++s) {
        const long c = round + (long)((KB + s - 1) / s) * block + exchange + (long)(s - 2) * exchange_cta;
        if (c >= best.cost) continue;
        if ((bm == 64 ? tile_clusters<64, false>(dev, s) : tile_clusters<128, false>(dev, s)) >= tiles) best = {bm, s, c};
    }
    return best;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// tile_limit >= 0: only the first tile_limit tiles (whole rounds). SPLIT: the tiles from split_base on, two CTAs each.
// CLUSTER: one tile per cluster of `cluster` CTAs.
template <int BM, bool GROUPED, bool OFFSET, bool CHAIN, bool SPLIT = false, bool CLUSTER = false>
cudaError_t launch_off(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream, int tile_limit = -1,
                       int split_base = 0, int split_tiles = 0, int cluster = 1) {
    using Smem = SharedStorage<BM, Roles<BM, GROUPED>::kEpiWarps>;
    const size_t smem_bytes = sizeof(Smem) + 1024;
    static SmemOptIn opt_in;
    if (const cudaError_t e = opt_in.ensure(gemm_tensor_kernel<BM, GROUPED, OFFSET, CHAIN, SPLIT, CLUSTER>, dev.device, smem_bytes);
        e != cudaSuccess)
        return e;
    CUtensorMap map;
    const cuuint64_t dims[2] = {(cuuint64_t)a.K, (cuuint64_t)a.M};
    const cuuint64_t strides[1] = {(cuuint64_t)a.K};
    const cuuint32_t box[2] = {128u, (cuuint32_t)BM};
    const cuuint32_t estr[2] = {1u, 1u};
    const CUresult r = reinterpret_cast<EncodeTiledFn>(dev.encode_tiled)(
        &map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t*>(a.q), dims, strides, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;

    CUtensorMap ymap = map;   // placeholder when the store path is off
    int y_tma = 0;
    if (CHAIN) {
        // the staged rows hold one byte per value (or per two values when packed): a map over the code
        // matrix, 32-byte (16-byte) rows
        if (a.next_packed && (a.N % 32 != 0 || (reinterpret_cast<uintptr_t>(a.q_next) & 15u) != 0))
            return cudaErrorInvalidValue;                    // packed codes only leave through the TMA store
        if (a.N % 16 == 0 && (reinterpret_cast<uintptr_t>(a.q_next) & 15u) == 0) {
            const cuuint64_t row_bytes = a.next_packed ? (cuuint64_t)a.N / 2 : (cuuint64_t)a.N;
            const cuuint64_t ydims[2] = {row_bytes, (cuuint64_t)a.M};
            const cuuint64_t ystrides[1] = {row_bytes};
            const cuuint32_t ybox[2] = {a.next_packed ? 16u : 32u, (cuuint32_t)Smem::kStageRows};
            const CUresult ry = reinterpret_cast<EncodeTiledFn>(dev.encode_tiled)(
                &ymap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, a.q_next, ydims, ystrides, ybox, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (ry != CUDA_SUCCESS) return cudaErrorInvalidValue;
            y_tma = 1;
        }
    } else if (a.N % 8 == 0 && (reinterpret_cast<uintptr_t>(a.y) & 15u) == 0) {
        const cuuint64_t ydims[2] = {(cuuint64_t)a.N, (cuuint64_t)a.M};
        const cuuint64_t ystrides[1] = {(cuuint64_t)a.N * 2};
        const cuuint32_t ybox[2] = {32u, (cuuint32_t)Smem::kStageRows};
        const CUresult ry = reinterpret_cast<EncodeTiledFn>(dev.encode_tiled)(
            &ymap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, a.y, ydims, ystrides, ybox, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (ry != CUDA_SUCCESS) return cudaErrorInvalidValue;
        y_tma = 1;
    }

    TensorParams p;
    p.y_tma = y_tma;
    p.M = a.M; p.K = a.K; p.N = a.N; p.Npad = round_up(a.N, kTileN);
    p.n_tiles_m = (a.M + BM - 1) / BM;
    p.n_tiles = p.n_tiles_m * (p.Npad / kTileN);
    p.w_packed = a.w_packed; p.w_scales = a.w_scales; p.scale_exp = a.scale_exp;
    p.y = a.y; p.acc_dump = a.acc_dump; p.ctl = a.ctl; p.chan_offset = a.chan_offset; p.zp_mid = a.zp_mid;
    p.q_next = a.q_next;
    p.next_inv = ldexpf(1.0f, -a.next_exp);
    p.next_lo = -(float)(1 << (a.next_bits - 1));
    p.next_hi = (float)((1 << (a.next_bits - 1)) - 1);
    p.next_packed = a.next_packed ? 1 : 0;
    if (tile_limit >= 0) p.n_tiles = tile_limit;
    p.split_base = split_base;
    p.split_scratch = a.split_scratch;
    p.clear_status = !a.after_quantize && split_base == 0 ? 1 : 0;
    p.wait_cycles = a.wait_cycles;
    const int grid = SPLIT ? 2 * split_tiles : (p.n_tiles < dev.sm_count ? p.n_tiles : dev.sm_count);
    if constexpr (SPLIT) {
        // This launch depends on nothing the preceding whole-round launch writes (other tiles of y; the
        // partial sums and their flags are its own), so it may be set up while that one still runs: its
        // CTAs start as SMs become free instead of after a launch gap.
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = smem_bytes;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, gemm_tensor_kernel<BM, GROUPED, OFFSET, CHAIN, SPLIT>, map, ymap, p);
    } else {
        // Behind the call's own quantize kernel the launch may overlap that kernel's drain (the kernel
        // waits for it before it reads what it wrote).
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = CLUSTER ? dim3(cluster, p.n_tiles) : dim3(grid);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = smem_bytes;
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = a.after_quantize ? 1 : 0;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = CLUSTER ? 2 : 1;
        return cudaLaunchKernelEx(&cfg, gemm_tensor_kernel<BM, GROUPED, OFFSET, CHAIN, SPLIT, CLUSTER>, map, ymap, p);
    }
}

template <int BM, bool GROUPED>
cudaError_t launch_bm(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream, int cluster = 1) {
    if (a.q_next && a.chan_offset) return cudaErrorInvalidValue;       // the two variants are not combined
    if constexpr (BM <= 192) {
        if (cluster > 1) {
            if (a.q_next) return launch_off<BM, GROUPED, false, true, false, true>(a, dev, stream, -1, 0, 0, cluster);
            if (a.chan_offset) return launch_off<BM, GROUPED, true, false, false, true>(a, dev, stream, -1, 0, 0, cluster);
            return launch_off<BM, GROUPED, false, false, false, true>(a, dev, stream, -1, 0, 0, cluster);
        }
    }
    if (a.chan_offset) return launch_off<BM, GROUPED, true, false>(a, dev, stream);
    if constexpr (GROUPED) {
        // Behind whole rounds: a last round that would leave more than half of the SMs idle is run as shared tiles, when the
        // reduction is deep enough for half a tile to outweigh the second launch and the exchange of
        // partial sums (measured with 128-token tiles: a loss of 2-5 us at K = 4096, a gain of 8 us at
        // K = 11008; with 192-token tiles a gain of 2 us at K = 4096 already). Chained calls share the same tiles as plain
        // ones: where a sum is cut decides its last fp32 rounding, and the codes are those of the plain call's outputs.
        const int sms = dev.sm_count;
        const int n_tiles = ((a.M + BM - 1) / BM) * (round_up(a.N, kTileN) / kTileN);
        const int rem = shared_tiles(n_tiles, sms, a.K / kTileK, BM), whole = n_tiles - rem;
        const size_t need = shared_scratch_bytes(rem, BM);
        if (rem > 0 && a.split_scratch && a.split_bytes >= need && (reinterpret_cast<uintptr_t>(a.split_scratch) & 15u) == 0) {
            if (!a.after_quantize) {
                const cudaError_t e = cudaMemsetAsync(a.ctl->split_flags, 0, sizeof(a.ctl->split_flags), stream);
                if (e != cudaSuccess) return e;
            }
            const cudaError_t e = a.q_next ? launch_off<BM, true, false, true>(a, dev, stream, whole)
                                           : launch_off<BM, true, false, false>(a, dev, stream, whole);
            if (e != cudaSuccess) return e;
            return a.q_next ? launch_off<BM, true, false, true, true>(a, dev, stream, -1, whole, rem)
                            : launch_off<BM, true, false, false, true>(a, dev, stream, -1, whole, rem);
        }
    }
    if (a.q_next) return launch_off<BM, GROUPED, false, true>(a, dev, stream);
    return launch_off<BM, GROUPED, false, false>(a, dev, stream);
}

}  // namespace

size_t tensor_split_scratch_bytes(int M, int K, int N, int group, int sm_count) {
    if (!group) return 0;
    DeviceInfo dev = {};
    dev.sm_count = sm_count;
    const int bm = grouped_plan(M, K, N, dev, ~(size_t)0, false, grouped_size_times).bm;
    const int n_tiles = ((M + bm - 1) / bm) * (round_up(N, kTileN) / kTileN);
    return shared_scratch_bytes(shared_tiles(n_tiles, sm_count, K / kTileK, bm), bm);
}

cudaError_t launch_int8_probe(int iters, int a_from_tmem, Control* ctl, const DeviceInfo& dev, cudaStream_t stream) {
    const size_t smem_bytes = sizeof(ProbeSmem) + 1024;
    static SmemOptIn opt_in;
    if (const cudaError_t e = opt_in.ensure(int8_probe_kernel, dev.device, smem_bytes); e != cudaSuccess) return e;
    int8_probe_kernel<<<dev.sm_count, 128, smem_bytes, stream>>>(iters, a_from_tmem, ctl);
    return cudaGetLastError();
}

cudaError_t launch_gemm_tensor(const GemmArgs& a, const DeviceInfo& dev, cudaStream_t stream) {
    if (a.group) {
        // the zero-point variant has no shared-tile launch
        const bool may_share = !a.chan_offset && a.split_scratch && (reinterpret_cast<uintptr_t>(a.split_scratch) & 15u) == 0;
        const GroupedPlan g = grouped_plan(a.M, a.K, a.N, dev, may_share ? a.split_bytes : 0, true);
        switch (g.bm) {
            case 64: return launch_bm<64, true>(a, dev, stream, g.split);
            case 192: return launch_bm<192, true>(a, dev, stream, g.split);
            default: return launch_bm<128, true>(a, dev, stream, g.split);
        }
    }
    // one scale per channel: two channel blocks share a token tile where the shape allows it and that is the shorter schedule
    const ChannelPlan c = channel_plan(a.M, a.K, a.N, dev);
    if (gemm_wide_applies(a, dev, c.cost)) return launch_gemm_wide(a, dev, stream);
    switch (c.bm) {
        case 64: return launch_bm<64, false>(a, dev, stream, c.split);
        case 128: return launch_bm<128, false>(a, dev, stream, c.split);
        default: return launch_bm<256, false>(a, dev, stream);    // halves the MMA instructions per unit of work
    }
}

}  // namespace aq
