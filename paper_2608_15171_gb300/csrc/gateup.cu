// Gate-up projection of the decoder MLP with the gated activation fused in:
//   Y[t, i] = silu(X[t] . W_gate[i]) * (X[t] . W_up[i])
// (the GEMM profiled beside attention in Section 6.1), on the tcgen05 tensor
// cores.
//
// The weights are packed once (gateup_pack_kernel) so that every 256-row
// block holds 128 gate rows followed by the 128 up rows of the same
// features.  One output tile is 256 tokens x 128 features, worked by a pair of
// CTAs (cta_group::2): M 256 (128 tokens in each CTA) x N 256 (gate products
// left, up products right), so the epilogue combines them without leaving
// the SM and the [T, 2I] intermediate never reaches HBM.  Each CTA of the pair
// loads its own tokens and half of the weight rows: 32 KB of L2 traffic for 64
// columns of K and 512 tensor cycles.  A CTA by itself with the same 128 x 256
// share needs 48 KB, 96 B/clk on every SM, which L2 does not deliver.  Hidden
// 2048, inter 11008, 128-token tiles of single CTAs and now, us; a run of a few
// ms, and back to back for 150 ms (the GPU is then at its power limit):
//   256 tokens  34.0 -> 24.7, 33.8 -> 24.7     2056  119.3 -> 105.8, 128.8 -> 122.0
//   512         43.3 -> 32.0, 43.1 -> 35.3    16384  818 -> 721, 908 -> 854
//   1024        66.5 -> 54.5, 68.2 -> 62.4
// Tokens are padded to 256 instead of 128, so that calls of few rounds whose
// last 128 tokens are all padding can be slower than those tiles were: 520
// tokens 43.3 -> 44.1, 770 56.4 -> 58.7 (hidden 4096, inter 14336: 520 tokens 105.0
// -> 108.5); most counts are faster (260 31.7 -> 30.2, 1030 76.6 -> 72.0).
//
// Persistent kernel, one CTA per SM, 192 threads:
//   warp 0      TMA producer: X tile (128 x 64) and W tile (128 x 64) per
//               64-wide K block, 128-byte swizzle, 6-stage ring; both CTAs'
//               bytes are counted by the leader's barrier
//   warp 1      allocates TMEM; the leader's issues the pair's MMAs (4 x K16 per
//               K block) into one of two 256-column accumulators, and its
//               commits release the ring and fill the accumulators in both CTAs
//   warps 2-5   epilogue: each thread owns one token row (its TMEM lane),
//               reads 32 gate and 32 up columns at a time, writes bf16
// The producer and MMA warps run their loops as whole warps and only issue
// under elect_one(), which keeps descriptors and addresses in uniform
// registers (2-2.5 % against loops of lane 0).
// Tiles are visited in groups of 16 M blocks with the M block fastest, so
// the pairs running at one time share a few weight tiles and keep a few MB of
// X tiles hot in L2 (groups of 8: 2056 tokens 114.5 against 112.9 us).
// Calls of at most few_tokens() tokens take another kernel, below.
#include <algorithm>

#include "ppas_device.cuh"
#include "ppas_internal.h"

namespace ppas {
namespace {

constexpr int kGM = 256;   // tokens per tile: 128 in each CTA of a pair
constexpr int kGN = 256;   // accumulator columns: 128 gate + 128 up
constexpr int kGK = 64;    // K per stage (128 bytes of bf16: one swizzle row)
constexpr int kGStages = 6;
constexpr int kGroupM = 16;  // M blocks per raster group
constexpr uint32_t kABytes = kGM / 2 * kGK * 2;  // 16 KB in each CTA
constexpr uint32_t kBBytes = kGN / 2 * kGK * 2;  // 16 KB in each CTA
constexpr uint32_t kStage = kABytes + kBBytes;
constexpr uint32_t kOffBarG = kGStages * kStage;
enum : int {
    G_FULL = 0,
    G_EMPTY = G_FULL + kGStages,
    G_ACCFULL = G_EMPTY + kGStages,  // [2]
    G_ACCEMPTY = G_ACCFULL + 2,      // [2]
    G_DRAIN = G_ACCEMPTY + 2,
    G_COUNT = G_DRAIN + 1
};
constexpr uint32_t kOffTmemG = kOffBarG + G_COUNT * 8;
constexpr uint32_t kOffAbortG = kOffTmemG + 4;   // set in both CTAs of a pair
constexpr uint32_t kOffIssuedG = kOffAbortG + 4;  // K blocks whose copies this CTA issued
constexpr uint32_t kSmemG = kOffBarG + 256 + 1024;  // + alignment slack
static_assert(kOffIssuedG + 4 <= kOffBarG + 256, "barrier area");
static_assert(kSmemG <= 232448, "shared memory per CTA");
constexpr int kGThreads = 192;

// One item of a pair: a tile, or one of `cut` equal column slices of it.
struct GateUpItem {
    int mb, nb;     // m block, n block (128 features)
    int f0, width;  // the slice's first feature within the block, and its features
};

// tile index -> (m block, n block), M fastest within groups of kGroupM
__device__ __forceinline__ void tile_mn(int t, int m_blocks, int n_blocks, int &mb, int &nb) {
    const int per_group = kGroupM * n_blocks;
    const int grp = t / per_group, rem = t - grp * per_group;
    const int gm = min(kGroupM, m_blocks - grp * kGroupM);
    nb = rem / gm;
    mb = grp * kGroupM + rem % gm;
}

__device__ __forceinline__ void tmem_ld16_sync(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

// item t of the launch: the first n_full are whole tiles, the others slices
__device__ __forceinline__ GateUpItem gateup_item(const GateUpParams &p, int t, int m_blocks, int n_blocks) {
    GateUpItem it;
    const int u = t - p.n_full;
    const int tile = u < 0 ? t : p.n_full + u / p.cut;
    tile_mn(tile, m_blocks, n_blocks, it.mb, it.nb);
    it.width = u < 0 ? kGN / 2 : kGN / 2 / p.cut;
    it.f0 = u < 0 ? 0 : (u % p.cut) * it.width;
    return it;
}

}  // namespace

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGThreads, 1)
    gateup_swiglu_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                         const __grid_constant__ CUtensorMap tm_cut, const __grid_constant__ GateUpParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t sb = (raw_s + 1023u) & ~1023u;
    uint8_t *const sg = smem_raw + (sb - raw_s);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (uniform)
    auto bar = [&](int i) { return sb + kOffBarG + 8u * static_cast<uint32_t>(i); };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sg + kOffAbortG);

    const int m_blocks = (p.n_tokens + kGM - 1) / kGM;
    const int n_blocks = p.inter / (kGN / 2);
    const int n_items = p.n_items;
    const int k_blocks = p.hidden / kGK;
    const uint32_t rank = cluster_ctarank();  // 0: the pair's leader
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    // a wait ran out: both CTAs of the pair are told
    auto give_up = [&]() {
        *abort_flag = 1;
        dsmem_st_s32(dsmem_addr(sb + kOffAbortG, rank ^ 1u), 1);
    };

    if (warp == 1) {
        tmem_alloc_pair(sb + kOffTmemG, 512);
        tmem_relinquish_pair();
    }
    if (tid == 0) {
        for (int s = 0; s < kGStages; ++s) {
            mbar_init(bar(G_FULL + s), 1);
            mbar_init(bar(G_EMPTY + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(G_ACCFULL + b), 1);
            mbar_init(bar(G_ACCEMPTY + b), 8);  // one arrive per epilogue warp of the pair
        }
        mbar_init(bar(G_DRAIN), 1);
        *abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tm_x);
        prefetch_tmap(&tm_w);
        prefetch_tmap(&tm_cut);
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();  // both CTAs' barriers and TMEM are there
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(sg + kOffTmemG), 0);
    // the set-up above overlaps the kernel before this one on the stream
    grid_dep_wait();

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        // each CTA loads its 128 tokens and its half of the weight rows (rank
        // 0: the gate rows, rank 1: the up rows); all of a stage's bytes
        // are counted by the leader's barrier
        int q = 0;  // K blocks issued by this CTA
        bool ok = true;
        for (int t = pair; ok && t < n_items; t += n_pairs) {
            const GateUpItem item = gateup_item(p, t, m_blocks, n_blocks);
            const int x_row = item.mb * kGM + static_cast<int>(rank) * (kGM / 2);
            const int w_row = item.nb * kGN + static_cast<int>(rank) * (kGN / 2) + item.f0;
            const CUtensorMap *tw = t < p.n_full ? &tm_w : &tm_cut;
            const uint32_t bytes = kABytes + static_cast<uint32_t>(item.width) * kGK * 2;
            for (int kb = 0; kb < k_blocks; ++kb, ++q) {
                const int s = q % kGStages;
                if (q >= kGStages && !mbar_wait_warp(bar(G_EMPTY + s), ((q / kGStages) & 1) ^ 1, p.err)) {
                    ok = false;
                    break;
                }
                const uint32_t full = dsmem_addr(bar(G_FULL + s), 0);
                if (elect_one()) {
                    const uint32_t dst = sb + s * kStage;
                    if (rank == 0) mbar_expect_tx(bar(G_FULL + s), 2 * bytes);
                    tma_load_2d_pair(dst, &tm_x, kb * kGK, x_row, full);
                    tma_load_2d_pair(dst + kABytes, tw, kb * kGK, w_row, full);
                }
                __syncwarp();
            }
            if (__any_sync(0xffffffffu, *abort_flag)) ok = false;
        }
        // the leader's last releases of the ring have reached this CTA before it leaves
        for (int j = max(0, q - kGStages); ok && j < q; ++j)
            ok = mbar_wait_warp(bar(G_EMPTY + j % kGStages), (j / kGStages) & 1, p.err);
        if (!ok) give_up();
        if (lane == 0) *reinterpret_cast<volatile int *>(sg + kOffIssuedG) = q;
        // every MMA of the pair has completed, and this CTA has been told
        mbar_wait_warp(bar(G_DRAIN), 0, p.err);
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer (the leader's)
        if (rank == 0) {
            const uint64_t da0 = smem_desc_sw128(sb, 16, 1024);
            const uint64_t db0 = smem_desc_sw128(sb + kABytes, 16, 1024);
            int q = 0, it = 0;
            bool ok = true;
            for (int t = pair; ok && t < n_items; t += n_pairs, ++it) {
                const int buf = it & 1;
                const uint32_t d = tmem + buf * kGN;
                const uint32_t idesc = t < p.n_full ? idesc_bf16_f32(kGM, kGN, false, false)
                                                    : idesc_bf16_f32(kGM, kGN / p.cut, false, false);
                // both epilogues have drained this accumulator (two tiles ago)
                if (it >= 2 && !mbar_wait_warp(bar(G_ACCEMPTY + buf), ((it >> 1) & 1) ^ 1, p.err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                for (int kb = 0; kb < k_blocks; ++kb, ++q) {
                    const int s = q % kGStages;
                    if (!mbar_wait_warp(bar(G_FULL + s), (q / kGStages) & 1, p.err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t da = da0 + ((s * kStage) >> 4), db = db0 + ((s * kStage) >> 4);
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kGK / 16; ++kk)
                            umma_bf16_pair(d, da + (kk * 2), db + (kk * 2), idesc, (kb > 0 || kk > 0) ? 1u : 0u);
                        umma_commit_pair(bar(G_EMPTY + s));
                        if (kb == k_blocks - 1) umma_commit_pair(bar(G_ACCFULL + buf));
                    }
                    __syncwarp();
                }
            }
            if (!ok) give_up();
            if (elect_one()) umma_commit_pair(bar(G_DRAIN));
        }
    } else {
        // ---------------------------------------------------------------- epilogue
        const int wq = warp & 3;  // TMEM lane quarter of this warp
        const uint32_t t_lane = tmem + (static_cast<uint32_t>(wq * 32) << 16);
        int it = 0;
        for (int t = pair; t < n_items; t += n_pairs, ++it) {
            const int buf = it & 1;
            const bool ok = mbar_wait_warp(bar(G_ACCFULL + buf), (it >> 1) & 1, p.err) &&
                            !__any_sync(0xffffffffu, *abort_flag);
            if (!ok) {
                give_up();
                break;
            }
            tc_fence_after();
            const GateUpItem item = gateup_item(p, t, m_blocks, n_blocks);
            const int row0 = item.mb * kGM + static_cast<int>(rank) * (kGM / 2) + wq * 32;  // the warp's first token
            __nv_bfloat16 *out = p.y + static_cast<int64_t>(row0) * p.inter + item.nb * (kGN / 2) + item.f0;
#pragma unroll 1
            for (int c = 0; c < item.width / 32; ++c) {
                float gv[32], uv[32];
                tmem_ld32_sync(t_lane + buf * kGN + c * 32, gv);
                tmem_ld32_sync(t_lane + buf * kGN + item.width + c * 32, uv);
                if (row0 + lane < p.n_tokens) {
                    uint4 *dst = reinterpret_cast<uint4 *>(out + static_cast<int64_t>(lane) * p.inter + c * 32);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t w4[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int e = 8 * i + 2 * k;
                            const float y0 = __fdividef(gv[e], 1.f + __expf(-gv[e])) * uv[e];
                            const float y1 = __fdividef(gv[e + 1], 1.f + __expf(-gv[e + 1])) * uv[e + 1];
                            w4[k] = pack_bf16x2(y0, y1);
                        }
                        dst[i] = make_uint4(w4[0], w4[1], w4[2], w4[3]);
                    }
                }
            }
            // the accumulator is free: its reads have completed, and nothing else
            // is handed over.  (With a cluster-scope release here every tile waited
            // for its own stores: 8000 tokens, hidden 64, inter 6912 73.7 us, 47.8
            // without; hidden 512 92.9 and 80.4; 2056, hidden 2048, inter 11008
            // 121.1 and 120.2.)
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(dsmem_addr(bar(G_ACCEMPTY + buf), 0));
        }
    }

    // neither CTA frees its TMEM or leaves while the other's MMAs, copies or
    // arrivals may still reach it
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, 512);
    }
    if (*abort_flag) {  // (the same in both CTAs)
        // a wait ran out: nor while copies are in flight.  The leader, whose
        // barriers count both CTAs' bytes, waits for the newest block of each
        // stage, and arms what only the other CTA issued.  (After the release of
        // TMEM: before it, calls of 10 us took 0.05 more.)
        if (rank == 0 && warp == 0) {
            const int q0 = *reinterpret_cast<volatile int *>(sg + kOffIssuedG);
            const int q1 = dsmem_ld_s32(dsmem_addr(sb + kOffIssuedG, 1));
            const RingPairNewest nw =
                lane < kGStages ? ring_pair_newest(q0, q1, lane, kGStages) : RingPairNewest{-1, false};
            if (nw.arm) {
                const GateUpItem item = gateup_item(p, pair + nw.block / k_blocks * n_pairs, m_blocks, n_blocks);
                mbar_expect_tx(bar(G_FULL + lane), kABytes + static_cast<uint32_t>(item.width) * kGK * 2);
            }
            if (nw.block >= 0) mbar_wait(bar(G_FULL + lane), (nw.block / kGStages) & 1, nullptr);
            __syncwarp();
        }
        cluster_sync_all();
    }
}

// ---------------------------------------------------------------- few tokens
// At most few_tokens tokens (a decode iteration): the projection is bound by
// streaming the weights, so the operands change sides.  A = weights, 64 gate
// rows and the 64 up rows of the same features as one M128 tile; B = all the
// tokens (N = tokens rounded up to 16).  One CTA per 64 features.  Where those
// are more than the SMs, two share one, so that at inter = 11008 all 172 CTAs
// stream at once (tiles of 128 tokens x 128 features are 86, and pad the tokens
// to 128 rows of MMA work); else each has an SM, and its memory, to itself.
// 192 threads: warp 0 TMA, warp 1 MMA, warps 2-5 epilogue: gate and up
// accumulators of a feature lie 64 TMEM lanes apart, so both go through shared
// memory (the ring, once the last MMA has completed).
// Hidden 2048, inter 11008 (90 MB of weights): see launch_gateup_few.
constexpr int kFF = 64;  // features per CTA
constexpr uint32_t kFewA = 128 * kGK * 2;  // weight tile of a K block: 16 KB
constexpr uint32_t kFewRing = 112640;      // ring bytes at most where two CTAs share an SM
constexpr uint32_t kFewRingAlone = 225280; // and where no SM gets a second CTA
constexpr int kFewMaxStages = 12;

// accumulator columns to allocate: a power of two, at least 32
__host__ __device__ constexpr int few_cols(int n) { return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : 256; }
__host__ __device__ constexpr uint32_t few_stage(int n) { return kFewA + static_cast<uint32_t>(n) * kGK * 2; }
__host__ __device__ constexpr int few_stages(int n, uint32_t ring) {
    return static_cast<int>(ring / few_stage(n)) < kFewMaxStages ? static_cast<int>(ring / few_stage(n))
                                                                 : kFewMaxStages;
}
static_assert(few_stages(kFewTokens, kFewRing) >= 3, "ring depth");
static_assert(kFewTokens * 128 * 4 <= few_stages(kFewTokens, kFewRing) * few_stage(kFewTokens),
              "epilogue buffer in the ring");
static_assert(few_stages(kFewTokensAlone, kFewRingAlone) >= 3 && kFewTokensAlone <= 256 &&
                  kFewTokensAlone * 128 * 4 <= few_stages(kFewTokensAlone, kFewRingAlone) * few_stage(kFewTokensAlone),
              "the same where a CTA is alone");

__global__ void __launch_bounds__(kGThreads, 2)
    gateup_few_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                      const __grid_constant__ GateUpParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kFewMaxStages + 1];
    __shared__ uint32_t tmem_base;
    __shared__ int abort_word;
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t sb = (raw_s + 1023u) & ~1023u;
    float *const buf = reinterpret_cast<float *>(smem_raw + (sb - raw_s));  // [128 rows][n] after the MMAs
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (uniform)
    auto full = [&](int s) { return smem_u32(bars) + 8u * static_cast<uint32_t>(s); };
    auto empty = [&](int s) { return smem_u32(bars) + 8u * static_cast<uint32_t>(kFewMaxStages + s); };
    const uint32_t done = smem_u32(bars) + 8u * (2 * kFewMaxStages);
    volatile int *abort_flag = &abort_word;

    const int n = (p.n_tokens + 15) & ~15;
    const uint32_t stage = few_stage(n);
    // (computed: as a parameter of the launch, calls of 5 us took 0.1 more)
    const int stages = few_stages(n, p.alone ? kFewRingAlone : kFewRing);
    const int k_blocks = p.hidden / kGK;
    const int f0 = blockIdx.x * kFF;                       // first feature
    const int w_row = (f0 / 128) * 256 + (f0 % 128);       // its gate row in the packed weight; up: + 128

    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_base), few_cols(n));
        tmem_relinquish();
    }
    if (tid < stages) {
        mbar_init(full(tid), 1);
        mbar_init(empty(tid), 1);
        if (tid == 0) {
            mbar_init(done, 1);
            *abort_flag = 0;
            prefetch_tmap(&tm_x);
            prefetch_tmap(&tm_w);
        }
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *const_cast<volatile uint32_t *>(&tmem_base), 0);
    // the set-up above overlaps the kernel before this one on the stream
    grid_dep_wait();
    grid_dep_launch();

    if (warp == 0) {
        int kb = 0;
        for (int s = 0, round = 0; kb < k_blocks; ++kb) {
            if (round > 0 && !mbar_wait_warp(empty(s), (round - 1) & 1, p.err)) {
                *abort_flag = 1;
                break;
            }
            if (elect_one()) {
                const uint32_t dst = sb + s * stage;
                mbar_expect_tx(full(s), stage);
                tma_load_2d(dst, &tm_w, kb * kGK, w_row, full(s));
                tma_load_2d(dst + kFewA / 2, &tm_w, kb * kGK, w_row + 128, full(s));
                tma_load_2d(dst + kFewA, &tm_x, kb * kGK, 0, full(s));
            }
            __syncwarp();
            if (++s == stages) {
                s = 0;
                ++round;
            }
        }
        ring_land(full(0), kb, stages, lane);
    } else if (warp == 1) {
        const uint64_t da0 = smem_desc_sw128(sb, 16, 1024);
        const uint64_t db0 = smem_desc_sw128(sb + kFewA, 16, 1024);
        const uint32_t idesc = idesc_bf16_f32(128, 16, false, false) +
                               (static_cast<uint32_t>((n - 16) >> 3) << 17);  // N = n
        bool ok = true;
        for (int kb = 0, s = 0, round = 0; kb < k_blocks; ++kb) {
            if (!mbar_wait_warp(full(s), round & 1, p.err)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint64_t da = da0 + ((s * stage) >> 4), db = db0 + ((s * stage) >> 4);
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < kGK / 16; ++kk)
                    umma_bf16(tmem, da + kk * 2, db + kk * 2, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
                umma_commit(empty(s));
            }
            __syncwarp();
            if (++s == stages) {
                s = 0;
                ++round;
            }
        }
        if (!ok) *abort_flag = 1;
        // every MMA issued so far has completed once `done` is set
        if (elect_one()) umma_commit(done);
        __syncwarp();
        mbar_wait(done, 0, p.err);
    } else {
        const int wq = warp & 3;  // TMEM lane quarter: rows 0-63 gate, 64-127 up
        const bool ok = mbar_wait_warp(done, 0, p.err) && !__any_sync(0xffffffffu, *abort_flag);
        tc_fence_after();
        const uint32_t t_lane = tmem + (static_cast<uint32_t>(wq * 32) << 16);
        if (ok)
            for (int c = 0; c < n; c += 16) {
                uint32_t v[16];
                tmem_ld16_sync(t_lane + c, v);
#pragma unroll
                for (int i = 0; i < 16; ++i) buf[(c + i) * 128 + wq * 32 + lane] = __uint_as_float(v[i]);
            }
        nbar_sync(1, 128);
        if (ok) {
            // one warp per token: a lane's two features
            for (int t = wq; t < p.n_tokens; t += 4) {
                const float2 g = *reinterpret_cast<const float2 *>(buf + t * 128 + 2 * lane);
                const float2 u = *reinterpret_cast<const float2 *>(buf + t * 128 + 64 + 2 * lane);
                const float y0 = __fdividef(g.x, 1.f + __expf(-g.x)) * u.x;
                const float y1 = __fdividef(g.y, 1.f + __expf(-g.y)) * u.y;
                *reinterpret_cast<uint32_t *>(p.y + static_cast<int64_t>(t) * p.inter + f0 + 2 * lane) =
                    pack_bf16x2(y0, y1);
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, few_cols(n));
    }
}

// W [2I, H] (gate rows, then up rows) -> packed: block j of 256 rows holds
// gate rows 128j .. 128j+127 then up rows I+128j .. I+128j+127.
__global__ void gateup_pack_kernel(const uint4 *__restrict__ w, uint4 *__restrict__ wp, int hidden, int inter) {
    const int vec_per_row = hidden / 8;
    const int64_t total = static_cast<int64_t>(2 * inter) * vec_per_row;
    for (int64_t v = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; v < total;
         v += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t prow = v / vec_per_row;
        const int col = static_cast<int>(v - prow * vec_per_row);
        const int64_t blk = prow / 256, within = prow % 256;
        const int64_t src_row = within < 128 ? blk * 128 + within : inter + blk * 128 + (within - 128);
        wp[v] = w[src_row * vec_per_row + col];
    }
}

cudaError_t launch_gateup(const CUtensorMap &tm_x, const CUtensorMap &tm_w, const CUtensorMap &tm_cut,
                          const GateUpParams &p, int pairs, cudaStream_t st) {
    static std::atomic<uint64_t> smem_set{0};
    const cudaError_t e = ensure_smem_limit(gateup_swiglu_kernel, static_cast<int>(kSmemG), smem_set);
    if (e != cudaSuccess) return e;
    PdlLaunch l(dim3(2 * pairs), dim3(kGThreads), kSmemG, st);
    return cudaLaunchKernelEx(&l.cfg, gateup_swiglu_kernel, tm_x, tm_w, tm_cut, p);
}

// Times on one GB300, with 128-token tiles before and now (hidden 2048,
// inter 11008, 90 MB of weights): 1 token 26.5 -> 18.1 us, 8: 25.3 -> 17.8,
// 32: 22.3 -> 16.9, 64: 22.7 -> 18.6, 128: 23.4 -> 20.5 (the copy bandwidth
// takes 13.4); hidden 4096, inter 14336 (235 MB), 4 tokens: 55.1 -> 37.7.  Against
// the kernel above: 129 tokens 24.1 there, 20.4 here, 160 tokens 24.2 and 21.1
// (inter 14336: 45.9 and 43.8; hidden 8192, inter 28672: 157 on both).  Past
// 160 the ring falls below three stages and the epilogue's buffer outgrows it:
// those calls take the kernel above.
//
// With no more CTAs than SMs (inter <= 9728) each has an SM to itself: fewer SMs
// stream, so each has to keep more bytes in flight, and gets the longer ring.
// Times with kFewRing and with kFewRingAlone: hidden 4096, inter 4096 (67 MB,
// 64 CTAs): 24 tokens 16.8 -> 14.1 us, 64: 20.6 -> 14.8, 128: 24.8 -> 17.9 (the
// kernel above: 19.0, 19.2, 19.8); hidden 2048, inter 5632: 24 tokens 11.5 ->
// 10.7, 128: 16.0 -> 12.7; hidden 1024, inter 2816: 128 tokens 6.7 -> 6.1, 24
// tokens 4.9 and 4.9.  This ring has five stages at 224 tokens; past 160, the
// kernel above and this one: hidden 2048, inter 5632: 176 tokens 16.3 and 14.2,
// 192: 16.3, 14.6, 224: 16.4, 15.6, 256: 16.7, 18.7; inter 9728: 192 tokens 19.9,
// 18.2, 224: 20.0, 19.0; hidden 4096, inter 9728, 224 tokens: 31.8, 31.6.  With
// fewer than half the SMs streaming it loses there: hidden 4096, inter 4096, 176
// tokens: 20.1, 21.5.
cudaError_t launch_gateup_few(const CUtensorMap &tm_x, const CUtensorMap &tm_w, const GateUpParams &p, int sms,
                              cudaStream_t st) {
    static std::atomic<uint64_t> smem_set{0};
    const cudaError_t e =
        ensure_smem_limit(gateup_few_kernel, static_cast<int>(kFewRingAlone + 1024), smem_set);
    if (e != cudaSuccess) return e;
    const int n = (p.n_tokens + 15) & ~15;
    GateUpParams fp = p;
    fp.alone = p.inter / kFF <= sms;
    const int stages = few_stages(n, fp.alone ? kFewRingAlone : kFewRing);
    PdlLaunch l(dim3(p.inter / kFF), dim3(kGThreads), stages * few_stage(n) + 1024, st);
    return cudaLaunchKernelEx(&l.cfg, gateup_few_kernel, tm_x, tm_w, fp);
}

cudaError_t launch_gateup_pack(const void *w, void *wp, int hidden, int inter, cudaStream_t st) {
    const int64_t total = static_cast<int64_t>(2 * inter) * (hidden / 8);
    const int grid = static_cast<int>(std::min<int64_t>((total + 255) / 256, 152 * 16));
    gateup_pack_kernel<<<grid, 256, 0, st>>>(static_cast<const uint4 *>(w), static_cast<uint4 *>(wp), hidden,
                                             inter);
    return cudaGetLastError();
}

}  // namespace ppas
