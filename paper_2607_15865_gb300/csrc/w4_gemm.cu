// w4_gemm.cu -- W4BF16 weight GEMM for the prefill-side projections (tcgen05), and the
// RMSNorm pre-pass of the block's chunk.
//
// A prefill chunk of T tokens turns the block's projections (Listing 1: q/k/v_proj, o_proj)
// into GEMMs, Y[T, N] = X[T, K] . W[N, K]^T, with W in the W4BF16 tile stream of
// attn_w4bf16_gemv (Section 5.1).  Reading: each weight is decoded once into the tensor
// cores' operand type, W_bf16 = bf16((q - z) * s), and the products accumulate in f32.
//
// Computed transposed, Y^T = W . X^T, so that the decoded weights are the MMA's A operand,
// which tcgen05 reads from tensor memory: each decode thread owns one feature row (one TMEM
// lane), decodes its 128 inputs of a group from the record in shared memory and stores the
// 64 bf16 pairs straight into TMEM -- no shared-memory round trip, no swizzle arithmetic, a
// row's scale and zero point read once per group.  X^T is the B operand, K-major from
// shared memory exactly as TMA lays out a box of tokens x 64 inputs of X.
//
// What bounds it: the tensor pipe for hundreds of tokens, the chain of groups for few.  A
// pair of CTAs (cta_group::2) computes 256 features x nt tokens, nt up to 256: each CTA
// decodes its own 128 features (its lanes of A and D) and loads half of the tokens (its half
// of B), so a weight is decoded once per 256 tokens, an MMA (256 x nt x 16) runs nt / 2
// cycles on both SMs, and the one issuing thread makes one wait, eight MMAs and one commit
// per 128-input group.  (One CTA per 256 x 128 tile, its MMAs 128 x 128 x 16, twice the
// decoding and four barrier operations per sixteen MMAs, took 183 us on 4096 x 6144 x 4096;
// this takes 115 us alone and 126 to 128 among
// other calls, under the power cap; 22016 features 392 instead of 588 alone.)  Few tokens leave most SMs idle, so K
// is then split over the pairs of a cluster, which add their f32 partials through distributed
// shared memory (32 tokens x 4096 x 4096: 9 us, 24.6 before).
//
// Clusters of 2 S CTAs (S = split of K) walk output tiles, token tiles fastest.  Per CTA, 576
// threads:
//   warp 0, one lane   producer: per 128-input group this CTA's half of the X tile (two 2-D
//                      TMA boxes, 128-byte swizzle; tokens past T read as zeros) and the 8
//                      weight records of its 128 features into a kStages ring: their codes
//                      as one 4-D TMA box with 64-byte swizzle (row r's 16-byte chunk c lands
//                      at chunk c ^ ((r >> 1) & 3), so the eight rows that a quarter-warp of
//                      decode threads reads at once sit in eight different bank groups),
//                      their scales and zero points as one 3-D box (rows past N read as
//                      zeros, which decode to zero weights);
//   warp 1, one lane   of the pair's even CTA: tcgen05 issuer, per group 8 MMAs 256 x nt x 16
//                      from both CTAs' A buffers and X stages into both accumulators;
//   warps 2-9          decode, warps 2-5 the even groups, 6-9 the odd ones, into A buffer
//                      (group mod kStages).  A stage is loaded only after the MMAs that last
//                      read it, so a full stage also means a free A buffer, and a decoded
//                      buffer also means that this CTA's half of X has landed: the issuer
//                      waits on the eight decode warps of both CTAs and nothing else;
//   warps 10-17        epilogue: each thread one feature and up to 128 tokens, read from
//                      TMEM into packed registers (the optional residual, loaded while the
//                      MMAs run, added in float), the accumulator handed back, then written
//                      to y or, split by feature, to y / y1 / y2.
// TMEM (512 columns): A buffer b at 64 b, the accumulator (nt columns) at 256.
// Every mbarrier wait is bounded (ATTN_DEVERR_TIMEOUT in *err, then the CTA drains and
// leaves); the cluster barriers have no limit, and every thread of every CTA reaches each of
// them whatever its waits did.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>

#include "internal.h"
#include "sm100_ptx.cuh"

namespace attn {
namespace {

constexpr int kThreads = 576;
constexpr int kWarpTma = 0, kWarpMma = 1, kWarpDec0 = 2, kWarpEpi0 = 10;
constexpr int kBF = 256;                    // features per tile: 128 per CTA of the pair
constexpr int kMaxNt = 256;                 // tokens per tile (MMA N): a multiple of 32 up to this
constexpr int kMaxSplit = 4;                // pairs per cluster that share one tile's K
constexpr int kStages = 4;                  // ring stages = A buffers
constexpr int kChunk = 128 * 128;           // up to 128 token rows x 64 bf16 (128 bytes), swizzled
constexpr int kXStage = 2 * kChunk;         // this CTA's half of the X tile x 128 inputs
constexpr int kRecBytes = 1072;             // one weight record: 16 rows x 128 inputs
constexpr int kRecs = 8;                    // records per stage (128 features)
constexpr int kWcStage = kRecs * 16 * 64;   // their codes: 128 rows x 64 bytes, 64-byte swizzle
constexpr int kWsStage = kRecs * 48;        // their scales and zero points: 8 x 48 bytes
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmA = 0, kTmAcc = 256;
constexpr uint64_t kWaitNs = 1000000000ull;

struct L {
    static constexpr int OFF_X = 0;
    static constexpr int OFF_WC = OFF_X + kStages * kXStage;
    static constexpr int OFF_WS = OFF_WC + kStages * kWcStage;
    static constexpr int OFF_BAR = OFF_WS + kStages * kWsStage;
    static constexpr int NBAR = 3 * kStages + 3;
    static constexpr int OFF_TMEM = OFF_BAR + 8 * NBAR;
    static constexpr int OFF_ABORT = OFF_TMEM + 16;
    static constexpr int BYTES = OFF_ABORT + 16;
    static constexpr int ALLOC = BYTES + 1024;  // the dynamic base is aligned up to 1024 in the kernel
};
static_assert(L::ALLOC <= 232448, "shared memory");
// the partials that a split's peers leave in a CTA's idle X ring: (S - 1) x ceil8(nt / S) tokens x 128 f32
static_assert((kMaxSplit - 1) * (kMaxNt / kMaxSplit) * 512 <= kStages * kXStage && kMaxNt / 2 * 512 <= kStages * kXStage,
              "split partials fit in the X ring");
enum Bar {
    B_FULL0 = 0, B_EMPTY0 = kStages, B_AFULL0 = 2 * kStages, B_ACCFULL = 3 * kStages, B_ACCEMPTY, B_DRAIN
};

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// Arrive on the mbarrier at the shared::cluster address `bar` (another CTA's, or this one's).
// What it publishes is ordered by other means (tensor-memory stores by tcgen05.wait::st and
// the tcgen05 fences, the X tile by the copy's own barrier), so it needs no cluster-scope
// release, nor its wait a cluster-scope acquire: with those every group cost the issuing
// thread about 450 cycles and a decode warp about as many.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// mbar_wait whose polls may sleep up to 20 us at a time (the thread wakes when the phase
// completes): sixteen warps of a CTA wait most of the time, and their polls took issue slots
// from the one issuing thread (T 1024, N 6144, K 4096: 39.2 -> 35.4 us; flash_fwd and the
// decode, whose waits are short, got slower with it).
__device__ __forceinline__ bool wait_full(uint32_t bar, uint32_t parity, const volatile int* abort) {
    uint64_t t0 = 0;
    for (uint32_t it = 0;; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 15u) == 0) {
            const uint64_t now = globaltimer_ns();
            if (it == 0) t0 = now;
            if (abort != nullptr && *abort) return false;
            if (now - t0 > kWaitNs) return false;
        }
    }
}

// The CTA-pair forms of the tcgen05 operations (sm100_ptx.cuh has those of one CTA).
__device__ __forceinline__ void tmem_alloc2(uint32_t holder_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder_smem), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void umma2_ts_w(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi,
                                           uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], db, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive once on the barrier at this offset in every CTA of `mask` when every tcgen05 operation
// issued so far by this thread completes.
__device__ __forceinline__ void umma2_commit_mc(uint32_t bar, uint16_t mask) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"(mask)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ uint32_t bf16x2_sub(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ uint32_t bf16x2_mul(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// (128 + q) for the two codes of pair j of a word, as one three-input logic op.
__device__ __forceinline__ uint32_t code_pair(uint32_t w, int j, uint32_t mask, uint32_t magic) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(w >> (4 * j)), "r"(mask), "r"(magic));
    return r;
}

// Where feature n of the output goes: y, or its part of the split output.
struct Dst {
    uint16_t* p;
    int stride, col;
};
__device__ __forceinline__ Dst dst_of(const W4GemmEpi& epi, uint16_t* y, int N, int n) {
    if (n >= epi.n1) return {epi.y2, N - epi.n1, n - epi.n1};
    if (n >= epi.n0) return {epi.y1, epi.n1 - epi.n0, n - epi.n0};
    return {y, epi.n0, n};
}

// SPLIT: the cluster's nsplit pairs share one tile's K (one tile per cluster); otherwise a
// cluster is one pair that walks its tiles.
template <bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1) w4_gemm_kernel(const __grid_constant__ CUtensorMap map_x,
                                                              const __grid_constant__ CUtensorMap map_wc,
                                                              const __grid_constant__ CUtensorMap map_ws, int nt,
                                                              int nsplit, int n_tt, int n_units, int T, int N, int K,
                                                              uint16_t* __restrict__ y, int* err, const W4GemmEpi epi) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gb = smem_raw + (base - raw);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gb + L::OFF_ABORT);
    auto bar = [&](int i) -> uint32_t { return base + L::OFF_BAR + 8u * static_cast<uint32_t>(i); };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int half = static_cast<int>(rank & 1u);             // which CTA of the pair
    const int part = SPLIT ? static_cast<int>(rank >> 1) : 0;  // which split of K
    const int csize = SPLIT ? 2 * nsplit : 2;
    const int u0 = static_cast<int>(blockIdx.x) / csize, ustep = static_cast<int>(gridDim.x) / csize;
    const int ngroup = K / 128;
    const int g0 = SPLIT ? part * ngroup / nsplit : 0, g1 = SPLIT ? (part + 1) * ngroup / nsplit : ngroup;

    if (tid == 0) {
        *abort_flag = 0;
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bar(B_FULL0 + s), 1);
            mbar_init(bar(B_EMPTY0 + s), 1);  // the issuer's commit
            mbar_init(bar(B_AFULL0 + s), 8);  // four decode warps of each CTA (the even CTA's is used)
        }
        mbar_init(bar(B_ACCFULL), 1);
        mbar_init(bar(B_ACCEMPTY), 16);  // eight epilogue warps of each CTA (the even CTA's is used)
        mbar_init(bar(B_DRAIN), 1);
        fence_mbar_init();
        tma_prefetch_desc(&map_x);
        tma_prefetch_desc(&map_wc);
        tma_prefetch_desc(&map_ws);
    }
    if (warp == kWarpMma) tmem_alloc2(base + L::OFF_TMEM, kTmemCols);
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // the other CTAs' barriers exist before anything arrives on them
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<const uint32_t*>(gb + L::OFF_TMEM);
    // A dependent launch: the set-up above overlaps the previous kernel's tail; everything it may
    // have written is read, and anything it may still read is overwritten, only from here on.
    griddep_wait();
    griddep_launch_dependents();

    if (warp == kWarpTma) {
        if (lane == 0) {
            uint32_t gs = 0;  // groups issued
            bool ok = true;
            const uint32_t bytes = static_cast<uint32_t>(nt) * 128u + kWcStage + kWsStage;  // nt/2 tokens x 256 bytes
            for (int u = u0; u < n_units && ok; u += ustep) {
                const int ft = u / n_tt, tt = u - ft * n_tt;
                const int rec0 = (ft * kBF + 128 * half) / 16, t0 = tt * nt + half * (nt / 2);
                for (int G = g0; G < g1; ++G, ++gs) {
                    const int s = static_cast<int>(gs % kStages);
                    if (gs >= kStages &&
                        !wait_full(bar(B_EMPTY0 + s), (gs / kStages - 1u) & 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    // (rows past N and tokens past T read as zeros; every box counts its full size)
                    mbar_arrive_expect_tx(bar(B_FULL0 + s), bytes);
                    tma_load_4d(base + L::OFF_WC + s * kWcStage, &map_wc, 0, 0, G, rec0, bar(B_FULL0 + s));
                    tma_load_3d(base + L::OFF_WS + s * kWsStage, &map_ws, 0, G, rec0, bar(B_FULL0 + s));
                    for (int c = 0; c < 2; ++c)
                        tma_load_2d(base + L::OFF_X + s * kXStage + c * kChunk, &map_x, G * 128 + c * 64, t0,
                                    bar(B_FULL0 + s));
                }
            }
            if (!ok) {
                *abort_flag = 1;
                record_dev_err(err, kDevErrTimeout);
            }
            // every copy issued must land before the CTA may exit
            for (uint32_t g = gs > kStages ? gs - kStages : 0; g < gs; ++g)
                wait_full(bar(B_FULL0 + g % kStages), (g / kStages) & 1u, nullptr);
        }
    } else if (warp == kWarpMma) {
        if (half == 0) {
            // The whole warp runs the loop and one elected lane issues: the loop's values stay in
            // uniform registers, which the MMA takes its operands from.  (Issued inside a branch
            // of one lane, each of the eight MMAs of a group first moved its operands there: a
            // group of 32 tokens took 0.40 us instead of 0.28, of 128 0.40 instead of 0.35.)
            const uint32_t idesc = idesc_bf16_f32(256, nt, false, false);
            constexpr uint32_t kHi = desc_hi_sw128(1024);
            const uint32_t x_lo0 = desc_lo_sw128(base + L::OFF_X, 16);
            const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem, 0);
            const uint16_t mask = static_cast<uint16_t>(3u << (rank & ~1u));  // both CTAs of the pair
            uint32_t gs = 0;
            int tiles_done = 0;
            bool ok = true;
            for (int u = u0; u < n_units && ok; u += ustep, ++tiles_done) {
                // the accumulator is free once the epilogue has read the previous tile's
                if (tiles_done > 0)
                    ok = __all_sync(0xFFFFFFFFu,
                                    wait_full(bar(B_ACCEMPTY), static_cast<uint32_t>(tiles_done - 1) & 1u, abort_flag));
                if (!ok) break;
                for (int G = g0; G < g1; ++G, ++gs) {
                    const int s = static_cast<int>(gs % kStages);
                    ok = __all_sync(0xFFFFFFFFu, wait_full(bar(B_AFULL0 + s), (gs / kStages) & 1u, abort_flag));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t xa = x_lo0 + ((s * kXStage) >> 4);
                    const uint32_t a_col = tm + kTmA + 64u * s, d_col = tm + kTmAcc;
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {
                            const uint32_t c = ((kk >> 2) * kChunk + (kk & 3) * 32) >> 4;
                            umma2_ts_w(d_col, a_col + 8u * kk, xa + c, kHi, idesc, (G > g0 || kk > 0) ? 1u : 0u);
                        }
                        umma2_commit_mc(bar(B_EMPTY0 + s), mask);
                        if (G + 1 == g1) umma2_commit_mc(bar(B_ACCFULL), mask);  // the tile's products
                    }
                    __syncwarp();
                }
            }
            if (!ok && lane == 0) {
                *abort_flag = 1;
                record_dev_err(err, kDevErrTimeout);
            }
            // also after an abort: the MMAs issued so far complete on it
            if (elect_one()) umma2_commit_mc(bar(B_DRAIN), static_cast<uint16_t>(1u << rank));
            __syncwarp();
            wait_full(bar(B_DRAIN), 0u, nullptr);
        }
    } else if (warp < kWarpEpi0) {
        // ------------------------------------------------ decode: one feature row per thread
        const uint32_t set = static_cast<uint32_t>(warp - kWarpDec0) >> 2;  // this warp's groups: gs % 2 == set
        const int q = warp & 3;                                             // TMEM lane quadrant of this warp
        const int fl = q * 32 + lane;                                       // feature within the CTA (= TMEM lane)
        const uint32_t magic = 0x43004300u, mask = 0x000F000Fu;
        const uint32_t afull = mapa_shared(bar(B_AFULL0), rank & ~1u);
        const int sw = (fl >> 1) & 3;  // the 64-byte swizzle of this row
        uint32_t gs = 0;
        bool ok = true;
        for (int u = u0; u < n_units && ok; u += ustep) {
            for (int G = g0; G < g1; ++G, ++gs) {
                if ((gs & 1u) != set) continue;
                const int s = static_cast<int>(gs % kStages);
                ok = __all_sync(0xFFFFFFFFu, wait_full(bar(B_FULL0 + s), (gs / kStages) & 1u, abort_flag));
                if (!ok) break;
                tc_fence_after();
                uint32_t wv[16];
                const uint8_t* row = gb + L::OFF_WC + s * kWcStage + fl * 64;
                const uint8_t* rec = gb + L::OFF_WS + s * kWsStage + (fl >> 4) * 48;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 v = *reinterpret_cast<const uint4*>(row + 16 * (i ^ sw));
                    wv[4 * i] = v.x;
                    wv[4 * i + 1] = v.y;
                    wv[4 * i + 2] = v.z;
                    wv[4 * i + 3] = v.w;
                }
                const uint32_t sc = *reinterpret_cast<const uint16_t*>(rec + (fl & 15) * 2);
                const uint32_t z = rec[32 + (fl & 15)];
                const uint32_t zp = (0x4300u + z) * 0x00010001u;  // (128 + z) in both halves
                const uint32_t sp = sc * 0x00010001u;
                // word i: inputs 8 i .. 8 i + 7; pair p: inputs 8 i + 2 p, + 1 -> TMEM column 4 i + p
                const uint32_t a_col = tmem + (static_cast<uint32_t>(q * 32) << 16) + kTmA + 64u * s;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    uint32_t o[32];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            o[4 * i + p] = bf16x2_mul(bf16x2_sub(code_pair(wv[8 * hh + i], p, mask, magic), zp), sp);
                    tmem_st32(a_col + 32u * hh, o);
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(afull + 8u * s);
            }
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            record_dev_err(err, kDevErrTimeout);
        }
    }

    const int q = warp & 3;
    const int fl = q * 32 + lane;
    const int eh = (warp - kWarpEpi0) >> 2;  // epilogue: which half of the tokens
    const uint32_t lane_row = static_cast<uint32_t>(q * 32) << 16;
    if constexpr (!SPLIT) {
        if (warp >= kWarpEpi0) {
            // -------------------------------------------- epilogue: one feature, 128 tokens per thread
            const uint32_t accempty = mapa_shared(bar(B_ACCEMPTY), rank & ~1u);
            const int nc = min(8, nt / 16 - 8 * eh);  // 16-token chunks of this warp (<= 0: none)
            int tiles_done = 0;
            bool ok = true;
            for (int u = u0; u < n_units && ok; u += ustep, ++tiles_done) {
                const int ft = u / n_tt, tt = u - ft * n_tt;
                const int n = ft * kBF + 128 * half + fl;
                const int tb = tt * nt + 128 * eh;                       // this warp's first token
                const int te = min(T, min(tt * nt + nt, tb + 128));       // and its end
                // two tokens per register: the residual (loaded while the MMAs run; h may be x, and
                // each element is read here before this thread writes it below), then the result
                uint32_t res[64];
#pragma unroll
                for (int i = 0; i < 64; ++i) res[i] = 0u;
                if (epi.residual != nullptr && n < N) {
#pragma unroll
                    for (int i = 0; i < 64; ++i) {
                        const int t = tb + 2 * i;
                        const uint32_t lo = t < te ? epi.residual[static_cast<size_t>(t) * N + n] : 0u;
                        const uint32_t hi = t + 1 < te ? epi.residual[static_cast<size_t>(t + 1) * N + n] : 0u;
                        res[i] = lo | (hi << 16);
                    }
                }
                ok = __all_sync(0xFFFFFFFFu,
                                wait_full(bar(B_ACCFULL), static_cast<uint32_t>(tiles_done) & 1u, abort_flag));
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (c < nc) {
                        uint32_t r[16];
                        tmem_ld16(tmem + lane_row + kTmAcc + 128u * eh + 16u * c, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const uint32_t w = res[8 * c + e];
                            float lo = __uint_as_float(r[2 * e]), hi = __uint_as_float(r[2 * e + 1]);
                            if (epi.residual != nullptr) {
                                lo += __uint_as_float(w << 16);
                                hi += __uint_as_float(w & 0xFFFF0000u);
                            }
                            res[8 * c + e] = pack_bf16x2(lo, hi);
                        }
                    }
                }
                // the accumulator is read: the next tile's MMAs may overwrite it
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(accempty);
                if (n < N) {
                    const Dst d = dst_of(epi, y, N, n);
                    uint16_t* o = d.p + static_cast<size_t>(tb) * d.stride + d.col;
#pragma unroll
                    for (int i = 0; i < 64; ++i) {
                        if (tb + 2 * i < te) o[static_cast<size_t>(2 * i) * d.stride] = static_cast<uint16_t>(res[i] & 0xFFFFu);
                        if (tb + 2 * i + 1 < te) o[static_cast<size_t>(2 * i + 1) * d.stride] = static_cast<uint16_t>(res[i] >> 16);
                    }
                }
            }
            if (!ok && lane == 0) {
                *abort_flag = 1;
                record_dev_err(err, kDevErrTimeout);
            }
        }
    } else {
        // ------------------------------------------------ split K: every pair owns a slice of the tokens
        // Pair p finishes tokens [p w, (p + 1) w) of the tile.  Once all MMAs of the cluster are
        // complete (its X rings are idle), each CTA writes its f32 partials of the other pairs'
        // slices into the ring of the CTA that owns the same features there, slot by slot
        // [slot][token][128 features]; then each CTA adds its slice in the order of the splits.
        const int w = (nt / 8 + nsplit - 1) / nsplit * 8;
        bool ok = true;
        if (warp >= kWarpEpi0) {
            ok = __all_sync(0xFFFFFFFFu, wait_full(bar(B_ACCFULL), 0u, abort_flag));
            if (!ok && lane == 0) {
                *abort_flag = 1;
                record_dev_err(err, kDevErrTimeout);
            }
            tc_fence_after();
        }
        __syncwarp();
        cluster_sync();
        if (warp >= kWarpEpi0 && ok) {
            for (int p = 0; p < nsplit; ++p) {
                if (p == part) continue;
                const int slot = part < p ? part : part - 1;
                const uint32_t peer = mapa_shared(base + L::OFF_X, static_cast<uint32_t>(2 * p + half));
                for (int j = 8 * eh; j < w && p * w + j < nt; j += 16) {
                    uint32_t r[8];
                    tmem_ld8(tmem + lane_row + kTmAcc + static_cast<uint32_t>(p * w + j), r);
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        st_dsmem_f32(peer + static_cast<uint32_t>(((slot * w + j + e) * 128 + fl) * 4), r[e]);
                }
            }
        }
        __syncwarp();
        cluster_sync();
        if (warp >= kWarpEpi0 && ok) {
            const int ft = u0 / n_tt, tt = u0 - ft * n_tt;
            const int n = ft * kBF + 128 * half + fl;
            const float* slots = reinterpret_cast<const float*>(gb + L::OFF_X);
            for (int j = 8 * eh; j < w && part * w + j < nt; j += 16) {
                uint32_t r[8];
                tmem_ld8(tmem + lane_row + kTmAcc + static_cast<uint32_t>(part * w + j), r);
                tmem_wait_ld();
                const int t = tt * nt + part * w + j;
                if (n < N) {
                    const Dst d = dst_of(epi, y, N, n);
                    // (all loads of the chunk before its stores: h may be x, so no load may move past one)
                    float v[8], res[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        res[e] = epi.residual != nullptr && t + e < T
                                     ? __uint_as_float(static_cast<uint32_t>(epi.residual[static_cast<size_t>(t + e) * N + n]) << 16)
                                     : 0.f;
                    for (int p = 0; p < nsplit; ++p) {
                        const int slot = p < part ? p : p - 1;
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float a = p == part ? __uint_as_float(r[e]) : slots[(slot * w + j + e) * 128 + fl];
                            v[e] = p == 0 ? a : v[e] + a;
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (t + e < T)
                            d.p[static_cast<size_t>(t + e) * d.stride + d.col] = __bfloat16_as_ushort(
                                __float2bfloat16_rn(epi.residual != nullptr ? v[e] + res[e] : v[e]));
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync();  // no CTA leaves while its pair's MMAs, commits or partials may still reach it
    if (warp == kWarpMma) {
        tc_fence_after();
        tmem_dealloc2(tmem, kTmemCols);
    }
}

// RMSNorm rows: one CTA per row of K values, so that a chunk of a few hundred tokens fills the
// device and a thread's 16-byte loads are all in flight (500 rows of 4096 under the profiler: 8.7
// us with a warp per row, 4.1 with this).  Per-thread float sums of squares over the chunks in order, a shuffle tree, then the
// warps in order (a fixed order); a thread keeps its first kRmsKeep chunks in registers and
// re-reads the rest (L1/L2) to write bf16((x * r) * gamma).
constexpr int kRmsThreads = 128, kRmsKeep = 8;
__global__ void __launch_bounds__(kRmsThreads) rmsnorm_rows_kernel(const uint16_t* __restrict__ x,
                                                                   const uint16_t* __restrict__ gamma, float eps, int T,
                                                                   int K, uint16_t* __restrict__ xn) {
    __shared__ float part[kRmsThreads / 32];
    const int tid = threadIdx.x, row = blockIdx.x;
    griddep_wait();  // a dependent launch, as is the GEMM that follows
    griddep_launch_dependents();
    const uint4* xr = reinterpret_cast<const uint4*>(x + static_cast<size_t>(row) * K);
    const int nchunk = K / 8;
    auto squares = [](float ss, const uint4& v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float a = __uint_as_float(w[e] << 16), b = __uint_as_float(w[e] & 0xFFFF0000u);
            ss = fmaf(a, a, ss);
            ss = fmaf(b, b, ss);
        }
        return ss;
    };
    uint4 keep[kRmsKeep];
#pragma unroll
    for (int i = 0; i < kRmsKeep; ++i)
        keep[i] = tid + i * kRmsThreads < nchunk ? xr[tid + i * kRmsThreads] : make_uint4(0u, 0u, 0u, 0u);
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < kRmsKeep; ++i) ss = squares(ss, keep[i]);
    for (int i = tid + kRmsKeep * kRmsThreads; i < nchunk; i += kRmsThreads) ss = squares(ss, xr[i]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
    if ((tid & 31) == 0) part[tid >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kRmsThreads / 32; ++w) tot += part[w];
    const float r = 1.0f / sqrtf(tot / static_cast<float>(K) + eps);
    const uint4* gr = reinterpret_cast<const uint4*>(gamma);
    uint4* out = reinterpret_cast<uint4*>(xn + static_cast<size_t>(row) * K);
    auto write = [&](int i, const uint4& v) {
        const uint4 g = gr[i];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w}, gw[4] = {g.x, g.y, g.z, g.w};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float lo = (__uint_as_float(w[e] << 16) * r) * __uint_as_float(gw[e] << 16);
            const float hi = (__uint_as_float(w[e] & 0xFFFF0000u) * r) * __uint_as_float(gw[e] & 0xFFFF0000u);
            o[e] = pack_bf16x2(lo, hi);
        }
        out[i] = make_uint4(o[0], o[1], o[2], o[3]);
    };
#pragma unroll
    for (int i = 0; i < kRmsKeep; ++i)
        if (tid + i * kRmsThreads < nchunk) write(tid + i * kRmsThreads, keep[i]);
    for (int i = tid + kRmsKeep * kRmsThreads; i < nchunk; i += kRmsThreads) write(i, xr[i]);
}

std::mutex g_mutex;
PFN_encodeTiled g_encode = nullptr;
constexpr int kMaxDevices = 64;
bool g_configured[kMaxDevices] = {};
int g_clusters[kMaxDevices][kMaxSplit + 1] = {};  // clusters of 2 S CTAs resident at once, by S

// How a product of T tokens x N features x K inputs is cut: tokens per tile and pairs per tile.
struct Plan {
    int nt, split, n_tt, units;
};

// The cheapest plan by a model of the busiest cluster, in microseconds as measured on a GB300
// (calls one after another; K = 2048, 4096 and 11008, N = 3072 .. 22016, every nt and split):
// a 128-input group costs its MMAs (0.526 at nt = 256) and at least the chain of the issuing
// warp (0.28 at nt = 32, 0.35 at 128); a further tile of a pair 1.4; a launch 4.7; a split its
// cluster barriers and the exchange of its partials.
// What it weighs up, T x N at K = 4096: 8 x 6144 split 2 9.7, whole 13.6; 256 x 4096 128
// tokens split 2 12.8, 256 whole 22.6; 500 x 4096 in tiles of 128 17.1, of 256 22.8;
// 1024 x 6144 in tiles of 192 32.9, of 256 41.2.
Plan make_plan(int T, int N, int K, const int* clusters) {
    const int ngroup = K / 128, ft = (N + kBF - 1) / kBF;
    Plan best = {};
    double best_c = 1e300;
    for (int split = 1; split <= std::min(kMaxSplit, ngroup); ++split) {
        const int n_tt0 = (T + kMaxNt - 1) / kMaxNt;
        for (int n_tt = n_tt0; n_tt <= (T + 31) / 32; ++n_tt) {
            const int nt = ((T + n_tt - 1) / n_tt + 31) / 32 * 32;
            if ((T + nt - 1) / nt != n_tt) continue;
            const long long units = static_cast<long long>(ft) * n_tt;
            const long long rounds = (units + clusters[split] - 1) / clusters[split];
            // (narrower tiles only while they fill idle SMs; a split only where SMs are idle)
            if ((n_tt > n_tt0 && rounds > 1 && nt < 64) || units > (split > 1 ? 4096 : 1LL << 29)) break;
            const double group = std::max(0.526 * nt / kMaxNt, 0.265 + 0.00067 * nt) * ((ngroup + split - 1) / split);
            const double c = split == 1 ? 4.7 + rounds * group + (rounds - 1) * 1.4
                                        : rounds * (group + 5.2 + 0.022 * (nt - 32));
            if (c < best_c * 0.999) {
                best_c = c;
                best = {nt, split, n_tt, static_cast<int>(units)};
            }
        }
    }
    return best;
}

// Plans of the last shapes per device, so that a loop over the same products plans once.
Plan find_plan(int dev, int T, int N, int K, const int* clusters) {
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, int>, Plan> cache;
    std::lock_guard<std::mutex> lock(mu);
    const auto key = std::make_tuple(dev, T, N, K);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    if (cache.size() >= 4096) cache.clear();
    return cache[key] = make_plan(T, N, K, clusters);
}

cudaError_t configure(int dev) {
    cudaError_t e = cudaFuncSetAttribute(w4_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::ALLOC);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(w4_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::ALLOC);
    for (int s = 1; s <= kMaxSplit && e == cudaSuccess; ++s) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(2 * s));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = L::ALLOC;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = static_cast<unsigned>(2 * s);
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        e = s == 1 ? cudaOccupancyMaxActiveClusters(&n, w4_gemm_kernel<false>, &cfg)
                   : cudaOccupancyMaxActiveClusters(&n, w4_gemm_kernel<true>, &cfg);
        if (e == cudaSuccess && n < 1) e = cudaErrorInvalidConfiguration;
        g_clusters[dev][s] = n;
    }
    return e;
}

// The current device, configured, and the plan of a product there.
cudaError_t device_plan(int T, int N, int K, int* dev_out, Plan* plan) {
    cudaError_t e = cudaGetDevice(dev_out);
    const int dev = *dev_out;
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (g_encode == nullptr) {
            cudaDriverEntryPointQueryResult qres;
            void* fn = nullptr;
            e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qres);
            if (e != cudaSuccess) return e;
            if (qres != cudaDriverEntryPointSuccess || fn == nullptr) return cudaErrorNotSupported;
            g_encode = reinterpret_cast<PFN_encodeTiled>(fn);
        }
        if (!g_configured[dev]) {
            e = configure(dev);
            if (e != cudaSuccess) return e;
            g_configured[dev] = true;
        }
    }
    *plan = find_plan(dev, T, N, K, g_clusters[dev]);
    return plan->units < 1 ? cudaErrorInvalidValue : cudaSuccess;
}

}  // namespace

cudaError_t launch_rmsnorm_rows(const uint16_t* x, const uint16_t* gamma, float eps, int T, int K, uint16_t* xn,
                                cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(T));
    cfg.blockDim = dim3(kRmsThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, rmsnorm_rows_kernel, x, gamma, eps, T, K, xn);
}

cudaError_t launch_w4_gemm(const uint8_t* tiles, const uint16_t* x, int T, int N, int K, uint16_t* y, int* err,
                           cudaStream_t st, const W4GemmEpi* epi_in) {
    int dev = 0;
    Plan plan;
    const cudaError_t e = device_plan(T, N, K, &dev, &plan);
    if (e != cudaSuccess) return e;
    CUtensorMap map, map_wc, map_ws;
    {
        const cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(T)};
        const cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
        const cuuint32_t box[2] = {64, static_cast<cuuint32_t>(plan.nt / 2)};
        const cuuint32_t estr[2] = {1, 1};
        const CUresult r = g_encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(x), dims, strides,
                                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    // The tile stream as two views: record (row tile t, group g) at (t * K/128 + g) * 1072 bytes.
    //   codes  [row tile][group][16 rows][64 bytes]  (16-bit elements, box 32 x 16 x 1 x 16)
    //   scales and zero points [row tile][group][48 bytes] from byte 1024 of each record
    const cuuint64_t ng = static_cast<cuuint64_t>(K / 128), nt = static_cast<cuuint64_t>(N / 16);
    {
        const cuuint64_t dims[4] = {32, 16, ng, nt};
        const cuuint64_t strides[3] = {64, kRecBytes, kRecBytes * ng};
        const cuuint32_t box[4] = {32, 16, 1, static_cast<cuuint32_t>(kRecs)};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        const CUresult r = g_encode(&map_wc, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, const_cast<uint8_t*>(tiles), dims,
                                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[3] = {24, ng, nt};
        const cuuint64_t strides[2] = {kRecBytes, kRecBytes * ng};
        const cuuint32_t box[3] = {24, 1, static_cast<cuuint32_t>(kRecs)};
        const cuuint32_t estr[3] = {1, 1, 1};
        const CUresult r = g_encode(&map_ws, CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, const_cast<uint8_t*>(tiles) + 1024,
                                    dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                    CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    W4GemmEpi epi = {N, N, nullptr, nullptr, nullptr};
    if (epi_in != nullptr) epi = *epi_in;
    const int csize = 2 * plan.split;
    const int ncl = plan.split > 1 ? plan.units : std::min(plan.units, g_clusters[dev][1]);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(ncl * csize));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = L::ALLOC;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(csize);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, plan.split > 1 ? w4_gemm_kernel<true> : w4_gemm_kernel<false>, map, map_wc, map_ws,
                              plan.nt, plan.split, plan.n_tt, plan.units, T, N, K, y, err, epi);
}

cudaError_t w4_gemm_plan(int T, int N, int K, int out[4]) {
    int dev = 0;
    Plan plan;
    const cudaError_t e = device_plan(T, N, K, &dev, &plan);
    if (e != cudaSuccess) return e;
    out[0] = plan.nt;
    out[1] = plan.split;
    out[2] = plan.units;
    out[3] = plan.split > 1 ? plan.units : std::min(plan.units, g_clusters[dev][1]);
    return cudaSuccess;
}

}  // namespace attn
