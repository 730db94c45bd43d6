#pragma once

// Decode-row attention (one query token per sequence), split over the context:
// the body of one decode CTA, shared by the decode kernel and the single
// launch of a mixed step.
//
// A decode row is bandwidth-bound: every K/V byte is read once and used by
// the group's q-heads only.  One CTA takes one (row, kv-head, split): its
// pages are fetched by TMA (two 16x64 boxes per page and matrix, 128-byte
// swizzle) into a 3-stage ring per warp (eight warps, so eight threads issue
// copies; one issuing thread alone moves only ~7 B/clk); the split's page ids
// are staged in shared memory first.  Each warp computes
//   S^T[16 keys x heads] = K_page[16 x 128] . Q^T        (mma.sync m16n8k16)
//   online softmax per head (fp32, exp2 domain)
//   O^T[128 x heads] += V_page^T[128 x 16 keys] . P^T     (mma.sync m16n8k16)
// with the group's q-heads as the MMA's 8 columns (columns >= group are zero):
// 16 MMAs a page.  With the heads as its 16 rows, half of them always empty, a
// page took 48, and a step bound by one SM's rate (few rows, or decode rows
// beside prefill items) waited for them: 1 row x 25k (16/2 heads) 13.0 -> 12.6
// us a layer, 8 rows 36.8 -> 36.1, 16 rows x 30k (32/8) 283.5 -> 281.3, 4 x 512
// with 8 decodes 134.5 -> 131.5.  The
// warps merge their (m, l, O) in shared memory; with several splits the
// partial goes to the workspace and the last CTA of the (row, kv-head) to
// finish merges all splits:
//   o = sum_i 2^(m_i - M) o_i / sum_i 2^(m_i - M) l_i,  M = max_i m_i.
// The splits count their arrivals in a 64-bit ticket per (row, kv-head)
// that carries the launch's tag (tags increase from launch to launch), so
// tickets never need clearing before a launch; the kernel is launched with
// programmatic stream serialization and touches global memory only after
// grid_dep_wait().
// A step of one row is a chain of latencies once its 26 MB have streamed (at
// 5.8 of its 13.3 us, per-CTA timestamps), so the tail is kept short: the
// ticket is claimed before the merges by a reduction nobody waits for, one
// thread fences instead of all, the heads of a merge are independent
// loads, and the last CTA merges up to 20 partials in one round, weights in
// registers.  One row x 25k, 16/2 heads, append + attention: 14.3 -> 12.8 us
// a layer; 8 rows x 25k 37.4 -> 36.8.  (Claiming at entry cost
// the page loop 1 %: 96 rows of 17-4100 tokens 135.4 -> 137.3 us a layer.)
#include <math.h>

#include "ppas_device.cuh"
#include "ppas_internal.h"

namespace ppas {
namespace decode_detail {

constexpr uint32_t kBox = 2048;                     // 16 rows x 128 B
constexpr uint32_t kStageBytes = 4 * kBox;          // K lo, K hi, V lo, V hi
constexpr uint32_t kRingBytes = kDecodeStages * kStageBytes;
constexpr uint32_t kOffBar = kDecodeWarps * kRingBytes;
constexpr uint32_t kOffFlag = kOffBar + kDecodeWarps * kDecodeStages * 8;
constexpr uint32_t kOffIds = kOffFlag + 16;   // page ids of this split
// a cluster's merge: rank 0's slots for the cluster's CTA partials
// ([rank][group][128] O, then [rank][group][2] (m, l)), outside the rings,
// which a slower CTA of the cluster may still be streaming through when a
// faster one writes its partial
constexpr int kMaxCluster = 4;
constexpr uint32_t kOffClusterRecv = kOffIds + kDecodeMaxPagesPerSplit * 4;
constexpr uint32_t kClusterRecvBytes = kMaxCluster * 8 * (kHeadDim + 2) * 4;
constexpr uint32_t kSmemBytes = kOffClusterRecv + kClusterRecvBytes + 1024;
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
// merge scratch (aliases the rings once every warp is done)
constexpr int kMaxGroup = 8;
// a warp's O rows in the merge scratch: four floats apart from 128, so that
// the accumulators' columns fall into different banks
constexpr int kCoStride = kHeadDim + 4;
static_assert(kDecodeWarps * kMaxGroup * (2 + kCoStride) * 4 <= static_cast<int>(kOffBar), "merge scratch");
static_assert(2 * kMaxDecodeSplitsPerRow * kMaxGroup * 4 <= static_cast<int>(kOffBar), "split weights");
static_assert(kDecodeWarps >= kMaxGroup, "the split merge gives each head of a group one warp");
static_assert(kClusterRecvBytes == kMaxCluster * kMaxGroup * (kHeadDim + 2) * 4, "cluster slots");

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// transposes an 8 x 8 matrix of 16-bit values held one row to four lanes
__device__ __forceinline__ uint32_t movmatrix_t(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}

// byte offset of 16-byte chunk `chunk` (0..15 over 128 columns) of `row` in
// a page stored as two 16-row x 128 B halves with the 128-byte swizzle
__device__ __forceinline__ uint32_t swz(int row, int chunk) {
    return static_cast<uint32_t>((chunk >> 3) * kBox + row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
}

}  // namespace decode_detail

constexpr int kDecodeThreads = kDecodeWarps * 32;
constexpr uint32_t kDecodeSmemBytes = decode_detail::kSmemBytes;

// The CTA-wide barrier of the decode body: all threads of a decode launch,
// or the kDecodeThreads threads that run it inside a larger CTA (named
// barrier 1).
template <bool kPartial>
__device__ __forceinline__ void decode_cta_sync() {
    if constexpr (kPartial)
        nbar_sync(1, kDecodeThreads);
    else
        __syncthreads();
}

// One (row, kv-head, split) of a step's decode rows: CTA `bid` of the decode
// plan in p, run by threads 0 .. kDecodeThreads - 1 of the CTA (kPartial:
// the CTA has more threads, which do not take part).
template <bool kPartial, class P>
__device__ __forceinline__ void decode_cta(const CUtensorMap &tm_k, const CUtensorMap &tm_v, const P &p, int bid) {
    // in a cluster launch every CTA announces that it has started; the
    // matching wait comes before the first store into another CTA's shared
    // memory (the barrier phases of every CTA: this one, then one after
    // the stores, on every path)
    if constexpr (!kPartial)
        if (cluster_nctarank() > 1) cluster_arrive_relaxed();
    using namespace decode_detail;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t sb = (raw_s + 1023u) & ~1023u;
    uint8_t *const sg = smem_raw + (sb - raw_s);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (uniform)

    // ---- which (row, kv-head, split)
    int lo = 0, hi = p.n_rows - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.rows[mid].cta_base <= bid) lo = mid; else hi = mid - 1;
    }
    const DecodeRow row = p.rows[lo];
    const int local = bid - row.cta_base;
    const int kvh = local / row.n_splits, sp = local % row.n_splits;
    const int g = p.group;
    const int n_pages = (row.ctx_len + kPage - 1) / kPage;
    const int pg0 = sp * row.pages_per_split;
    const int pg1 = min(pg0 + row.pages_per_split, n_pages);
    const int my_count = max(0, (pg1 - pg0 - warp + kDecodeWarps - 1) / kDecodeWarps);
    const int32_t *table = p.block_tables + static_cast<int64_t>(row.table_row) * p.table_stride;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sg + kOffFlag);

    const uint32_t ring = sb + warp * kRingBytes;
    auto bar = [&](int st) { return sb + kOffBar + (warp * kDecodeStages + st) * 8u; };
    int32_t *ids = reinterpret_cast<int32_t *>(sg + kOffIds);
    if (lane == 0) {
        for (int st = 0; st < kDecodeStages; ++st) mbar_init(bar(st), 1);
        fence_mbar_init();
    }
    if (tid == 0) {
        *abort_flag = 0;
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
    }
    // the set-up above overlaps the kernel before this one on the stream;
    // global memory (page ids, Q, pages, workspace, output) only after it
    grid_dep_wait();
    // the split's page ids, loaded once by every thread in parallel
    for (int i = tid; i < pg1 - pg0; i += kDecodeThreads) ids[i] = __ldg(table + pg0 + i);
    decode_cta_sync<kPartial>();

    // A whole warp runs this and one elected lane issues: the copies' operands
    // stay uniform, where a lane 0 branch moved each through ordinary
    // registers between two pages' math.  (16 rows x 30k, 32/8 heads:
    // 287.2 -> 281.4 us a layer, 7.0 TB/s; 96 rows of 17-4100 tokens: 138.2 ->
    // 134.1; 8 rows x 25k, 16/2 heads: 38.2 -> 37.4.)
    auto issue = [&](int i) {
        const int st = i % kDecodeStages;
        const int pg = pg0 + warp + kDecodeWarps * i;
        int blk = ids[pg - pg0];
        if (blk < 0 || blk >= p.num_blocks) {
            if (lane == 0) report_error(p.err, PPAS_DEVERR_BAD_INDEX);
            blk = 0;
        }
        const int r = __shfl_sync(0xffffffffu, (blk * p.n_kv_heads + kvh) * kPage, 0);
        if (elect_one()) {
            const uint32_t dst = ring + st * kStageBytes, b = bar(st);
            mbar_expect_tx(b, kStageBytes);
            tma_load_2d(dst, &tm_k, 0, r, b);
            tma_load_2d(dst + kBox, &tm_k, 64, r, b);
            tma_load_2d(dst + 2 * kBox, &tm_v, 0, r, b);
            tma_load_2d(dst + 3 * kBox, &tm_v, 64, r, b);
        }
        __syncwarp();
    };
    for (int i = 0; i < min(kDecodeStages, my_count); ++i) issue(i);

    // ---- Q as the B operand: n = the group's heads, k = head dims
    const int hr = lane >> 2, c = lane & 3;
    uint32_t qb[8][2];
    {
        const bool valid = hr < g;
        const uint32_t *qrow = reinterpret_cast<const uint32_t *>(
            p.q + (static_cast<int64_t>(row.q_row) * p.n_q_heads + kvh * g + (valid ? hr : 0)) * kHeadDim);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            qb[kk][0] = valid ? __ldg(qrow + kk * 8 + c) : 0u;
            qb[kk][1] = valid ? __ldg(qrow + kk * 8 + 4 + c) : 0u;
        }
    }

    // accumulators: this lane has tokens hr and hr + 8 of a page's S, head
    // dims 16 n + hr and 16 n + hr + 8 of O, and heads 2c, 2c + 1 of both
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;  // l: over this lane's tokens
    float o[8][4];
#pragma unroll
    for (int n = 0; n < 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    const float sl2 = p.scale_log2;
    int consumed = 0;

    for (int i = 0; i < my_count; ++i) {
        const int st = i % kDecodeStages;
        const bool ok = mbar_wait_warp(bar(st), (i / kDecodeStages) & 1, p.err);
        if (!ok) {
            *abort_flag = 1;
            break;
        }
        consumed = i + 1;
        const int pg = pg0 + warp + kDecodeWarps * i;
        const int valid = min(kPage, row.ctx_len - pg * kPage);
        const uint32_t kb = ring + st * kStageBytes, vb = kb + 2 * kBox;
        if (valid < kPage) {
            // tokens past the context: zero their V rows so that 0 * V stays 0
            uint8_t *vg = sg + (vb - sb);
            const int n = (kPage - valid) * 8;
            for (int x = lane; x < 2 * n; x += 32) {
                const int half = x / n, rr = valid + (x % n) / 8, ch = x % 8;
                *reinterpret_cast<uint4 *>(vg + half * kBox + rr * 128 + ch * 16) = make_uint4(0, 0, 0, 0);
            }
            fence_proxy_async_smem();
            __syncwarp();
        }
        // S^T = K Q^T: 16 tokens x 8 heads, k over the head dims (two chains)
        float sa[4] = {0.f, 0.f, 0.f, 0.f}, sc[4] = {0.f, 0.f, 0.f, 0.f};
        const int mi = lane >> 3, ri = lane & 7;
#pragma unroll
        for (int kk = 0; kk < 8; kk += 2) {
            uint32_t a[4];
            ldsm_x4(kb + swz((mi & 1) * 8 + ri, kk * 2 + (mi >> 1)), a[0], a[1], a[2], a[3]);
            mma_bf16_16816(sa, a, qb[kk][0], qb[kk][1]);
            ldsm_x4(kb + swz((mi & 1) * 8 + ri, kk * 2 + 2 + (mi >> 1)), a[0], a[1], a[2], a[3]);
            mma_bf16_16816(sc, a, qb[kk + 1][0], qb[kk + 1][1]);
        }
        const float x0 = hr < valid ? (sa[0] + sc[0]) * sl2 : -INFINITY;  // (token hr, head 2c)
        const float x1 = hr < valid ? (sa[1] + sc[1]) * sl2 : -INFINITY;
        const float x2 = hr + 8 < valid ? (sa[2] + sc[2]) * sl2 : -INFINITY;  // (token hr + 8, head 2c)
        const float x3 = hr + 8 < valid ? (sa[3] + sc[3]) * sl2 : -INFINITY;
        float mx0 = fmaxf(x0, x2), mx1 = fmaxf(x1, x3);
#pragma unroll
        for (int o_ = 4; o_ <= 16; o_ <<= 1) {
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o_));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o_));
        }
        mx0 = fmaxf(m0, mx0);
        mx1 = fmaxf(m1, mx1);
        const float al0 = ex2(m0 - mx0), al1 = ex2(m1 - mx1);
        m0 = mx0;
        m1 = mx1;
        const float e0 = ex2(x0 - m0), e1 = ex2(x1 - m1), e2 = ex2(x2 - m0), e3 = ex2(x3 - m1);
        l0 = l0 * al0 + (e0 + e2);
        l1 = l1 * al1 + (e1 + e3);
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            o[n][0] *= al0;
            o[n][1] *= al1;
            o[n][2] *= al0;
            o[n][3] *= al1;
        }
        // O^T += V^T P^T: 16 head dims x 8 heads at a time, k over the tokens
        const uint32_t p0 = movmatrix_t(pack_bf16x2(e0, e1)), p1 = movmatrix_t(pack_bf16x2(e2, e3));
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            uint32_t a[4];
            ldsm_x4_t(vb + swz((mi >> 1) * 8 + ri, n * 2 + (mi & 1)), a[0], a[1], a[2], a[3]);
            mma_bf16_16816(o[n], a, p0, p1);
        }
        __syncwarp();
        if (i + kDecodeStages < my_count) issue(i + kDecodeStages);
    }
    // copies still in flight (only after an abort)
    if (lane == 0)
        for (int i = consumed; i < min(consumed + kDecodeStages, my_count); ++i)
            mbar_wait(bar(i % kDecodeStages), (i / kDecodeStages) & 1, nullptr);

    // CTAs per thread-block cluster: 1 unless the launch groups the splits of
    // a (row, kv-head) into clusters (steps of decode rows only)
    const uint32_t nct = kPartial ? 1u : cluster_nctarank();
    const uint32_t crank = nct > 1 ? cluster_ctarank() : 0u;

    // The splits of a (row, kv-head) count their arrivals in a ticket =
    // (tag << 16) | arrivals.  Tags grow from launch to launch, so a maximum
    // turns a word left by an earlier launch (or reset to 0) into this
    // launch's tag with no arrivals, and leaves a word this launch already
    // owns alone.  The split claims the word here, without waiting for an
    // answer, and adds its arrival (one atomic) when its partial is written.
    unsigned long long *const ctr = p.counters + lo * p.n_kv_heads + kvh;
    const unsigned long long ticket0 = p.launch_tag << 16;
    if (tid == 0 && row.n_splits > 1 && crank == 0) atomicMax(ctr, ticket0);

#pragma unroll
    for (int o_ = 4; o_ <= 16; o_ <<= 1) {
        l0 += __shfl_xor_sync(0xffffffffu, l0, o_);
        l1 += __shfl_xor_sync(0xffffffffu, l1, o_);
    }

    decode_cta_sync<kPartial>();  // rings are free from here on
    float *cm = reinterpret_cast<float *>(sg);
    float *cl = cm + kDecodeWarps * kMaxGroup;
    float *co = cl + kDecodeWarps * kMaxGroup;
    // this lane's heads 2c, 2c + 1 (those past the group are left out)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int hh = 2 * c + x;
        if (hh < g) {
            if (hr == 0) {
                cm[warp * kMaxGroup + hh] = x ? m1 : m0;
                cl[warp * kMaxGroup + hh] = x ? l1 : l0;
            }
            float *dst = co + (warp * kMaxGroup + hh) * kCoStride + hr;
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                dst[16 * n] = o[n][x];
                dst[16 * n + 8] = o[n][2 + x];
            }
        }
    }
    decode_cta_sync<kPartial>();
    // (in a cluster an aborted CTA carries on to the cluster barrier below)
    if (nct == 1 && *abort_flag) return;
    // rank 0's slot for this CTA's partial (cluster launches only)
    const uint32_t recv = sb + kOffClusterRecv;
    const uint32_t slot_o = nct > 1 ? dsmem_addr(recv + crank * (kMaxGroup * kHeadDim * 4), 0) : 0u;
    const uint32_t slot_ml =
        nct > 1 ? dsmem_addr(recv + kMaxCluster * kMaxGroup * kHeadDim * 4 + crank * (kMaxGroup * 2 * 4), 0) : 0u;
    if (nct > 1) cluster_wait();  // every CTA of the cluster has started (its arrive at entry)

    // thread -> (head-dim column, first head); the CTA's threads cover
    // kDecodeThreads / 128 heads at a time, all of a group's in one round of
    // independent loads
    const int t = tid & (kHeadDim - 1);
    constexpr int hstep = kDecodeThreads / kHeadDim, kHeads = kMaxGroup / hstep;
    const int h0 = tid / kHeadDim;
    float Mh[kHeads], Lh[kHeads], Oh[kHeads];
#pragma unroll
    for (int i = 0; i < kHeads; ++i) {
        const int hh = h0 + i * hstep;
        if (hh >= g) break;
        float m[kDecodeWarps];
        Mh[i] = -INFINITY;
#pragma unroll
        for (int w = 0; w < kDecodeWarps; ++w) {
            m[w] = cm[w * kMaxGroup + hh];
            Mh[i] = fmaxf(Mh[i], m[w]);
        }
        Lh[i] = Oh[i] = 0.f;
#pragma unroll
        for (int w = 0; w < kDecodeWarps; ++w) {
            // a warp without keys (or a split past its row's pages, which a
            // cluster plan may hold) has m = -inf and weight 0
            const float f = m[w] == -INFINITY ? 0.f : ex2(m[w] - Mh[i]);
            Lh[i] += f * cl[w * kMaxGroup + hh];
            Oh[i] += f * co[(w * kMaxGroup + hh) * kCoStride + t];
        }
    }
#pragma unroll
    for (int i = 0; i < kHeads; ++i) {
        const int hh = h0 + i * hstep;
        if (hh >= g) break;
        const int head = kvh * g + hh;
        if (row.n_splits == 1) {
            const int64_t oi = (static_cast<int64_t>(row.q_row) * p.n_q_heads + head) * kHeadDim + t;
            if (p.out_fp32) static_cast<float *>(p.out)[oi] = Oh[i] / Lh[i];
            else static_cast<__nv_bfloat16 *>(p.out)[oi] = __float2bfloat16_rn(Oh[i] / Lh[i]);
        } else if (nct > 1) {
            dsmem_st_f32(slot_o + static_cast<uint32_t>(hh * kHeadDim + t) * 4u, Oh[i]);
            if (t == 0) {
                dsmem_st_f32(slot_ml + static_cast<uint32_t>(hh * 2) * 4u, Mh[i]);
                dsmem_st_f32(slot_ml + static_cast<uint32_t>(hh * 2 + 1) * 4u, Lh[i]);
            }
        } else {
            const int64_t pi = static_cast<int64_t>(row.part_base + sp) * p.n_q_heads + head;
            p.part_o[pi * kHeadDim + t] = Oh[i];
            if (t == 0) {
                p.part_ml[pi * 2] = Mh[i];
                p.part_ml[pi * 2 + 1] = Lh[i];
            }
        }
    }
    if (row.n_splits == 1) return;
    int n_parts = row.n_splits;  // partial slots of this (row, kv-head)
    if constexpr (!kPartial) {
        if (nct > 1) {
            // The cluster's CTAs are consecutive splits sp0 .. sp0 + nct - 1
            // of this (row, kv-head) (sp0 a multiple of nct, rank = sp -
            // sp0).  Each has stored its partial into rank 0's slots above;
            // after the barrier (every CTA reaches it, an aborted one too)
            // rank 0 merges them from its own shared memory into partial
            // slot sp0 / nct, and the others are done.
            cluster_sync_all();
            if (crank != 0) return;
            const float *ro = reinterpret_cast<const float *>(sg + kOffClusterRecv);
            const float *rml = ro + kMaxCluster * kMaxGroup * kHeadDim;
#pragma unroll
            for (int i = 0; i < kHeads; ++i) {
                const int hh = h0 + i * hstep;
                if (hh >= g) break;
                float m[kMaxCluster];
                Mh[i] = -INFINITY;
#pragma unroll
                for (int r = 0; r < kMaxCluster; ++r) {
                    m[r] = r < static_cast<int>(nct) ? rml[(r * kMaxGroup + hh) * 2] : -INFINITY;
                    Mh[i] = fmaxf(Mh[i], m[r]);
                }
                Lh[i] = Oh[i] = 0.f;
#pragma unroll
                for (int r = 0; r < kMaxCluster; ++r)
                    if (m[r] != -INFINITY) {
                        const float f = ex2(m[r] - Mh[i]);
                        Lh[i] += f * rml[(r * kMaxGroup + hh) * 2 + 1];
                        Oh[i] += f * ro[(r * kMaxGroup + hh) * kHeadDim + t];
                    }
            }
#pragma unroll
            for (int i = 0; i < kHeads; ++i) {
                const int hh = h0 + i * hstep;
                if (hh >= g) break;
                const int64_t pi =
                    static_cast<int64_t>(row.part_base + sp / static_cast<int>(nct)) * p.n_q_heads + kvh * g + hh;
                p.part_o[pi * kHeadDim + t] = Oh[i];
                if (t == 0) {
                    p.part_ml[pi * 2] = Mh[i];
                    p.part_ml[pi * 2 + 1] = Lh[i];
                }
            }
            n_parts = row.n_splits / static_cast<int>(nct);
        }
    }

    // ---- the last CTA of this (row, kv-head) merges every split
    decode_cta_sync<kPartial>();
    __shared__ int s_last;
    if (tid == 0) {
        __threadfence();  // the whole CTA's partials (ordered before this by the barrier), then the arrival
        unsigned long long old = atomicAdd(ctr, 1ull);
        int prev = (old >> 16) == p.launch_tag ? static_cast<int>(old & 0xFFFFull) : -1;
        // a word with a larger tag (memory nothing of this process wrote):
        // the splits that met it count themselves again, from one of them on
        unsigned long long cur = old + 1;
        for (int it = 0; prev < 0 && it < (1 << 20); ++it) {
            if ((cur >> 16) == p.launch_tag) {
                old = atomicAdd(ctr, 1ull);
                prev = static_cast<int>(old & 0xFFFFull);
            } else {
                const unsigned long long got = atomicCAS(ctr, cur, ticket0 + 1);
                if (got == cur) prev = 0;
                cur = got;
            }
        }
        if (prev < 0) report_error(p.err, PPAS_DEVERR_TIMEOUT);  // the word was never claimed
        s_last = (prev == n_parts - 1);
        __threadfence();
    }
    decode_cta_sync<kPartial>();
    if (!s_last) return;
    if (tid == 0) *ctr = 0;  // ready for a replay with the same tag (a captured graph)
    // Warp hh merges head hh on its own (lane: 4 columns)
    const int ns = n_parts;
    const int hh = warp, c4 = lane;
    if (hh >= g) return;
    const int head = kvh * g + hh;
    const float4 *po = reinterpret_cast<const float4 *>(p.part_o) + c4;
    const float2 *pml = reinterpret_cast<const float2 *>(p.part_ml);
    auto part_index = [&](int s_) { return static_cast<int64_t>(row.part_base + s_) * p.n_q_heads + head; };
    auto warp_max = [](float x) {
#pragma unroll
        for (int o_ = 16; o_ >= 1; o_ >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o_));
        return x;
    };
    auto warp_sum = [](float x) {
#pragma unroll
        for (int o_ = 16; o_ >= 1; o_ >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o_);
        return x;
    };
    // partials a round: as many as the registers hold beside the rest (4 each).
    // A one-row step in clusters of 4 has 18 with 2 kv-heads (one round), 36 with
    // 1 (two, by the other path), fewer with more.
    constexpr int kBatch = 20;
    float4 ov[kBatch];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float L;
    auto load_o = [&](int s0) {
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
            ov[k] = s0 + k < ns ? __ldcg(po + part_index(s0 + k) * (kHeadDim / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto add_o = [&](int k, float f) {
        acc = make_float4(acc.x + f * ov[k].x, acc.y + f * ov[k].y, acc.z + f * ov[k].z, acc.w + f * ov[k].w);
    };
    if (ns <= kBatch) {
        // one round: lane s holds split s's (m, l) and weight w = 2^(m - M); its
        // load goes first, so the weights are there when the O are
        const float2 ml = lane < ns ? __ldcg(pml + part_index(lane)) : make_float2(-INFINITY, 0.f);
        load_o(0);
        const float M = warp_max(ml.x);
        const float f = ml.x == -INFINITY ? 0.f : ex2(ml.x - M);
        L = warp_sum(f * ml.y);
#pragma unroll
        for (int k = 0; k < kBatch; ++k) add_o(k, __shfl_sync(0xffffffffu, f, k));
    } else {
        // the first splits' O go out before the weights are known, so their
        // latency hides that of the (m, l) round; the weights stay in a
        // shared-memory row of the warp (the rings are free)
        load_o(0);
        float *wm = reinterpret_cast<float *>(sg) + hh * 2 * kMaxDecodeSplitsPerRow;  // [ns] m, then w
        float *wl = wm + kMaxDecodeSplitsPerRow;                                     // [ns] l
        float M = -INFINITY;
        for (int s_ = lane; s_ < ns; s_ += 32) {
            const float2 ml = __ldcg(pml + part_index(s_));
            wm[s_] = ml.x;
            wl[s_] = ml.y;
            M = fmaxf(M, ml.x);
        }
        M = warp_max(M);
        L = 0.f;
        for (int s_ = lane; s_ < ns; s_ += 32) {
            const float m = wm[s_];
            const float f = m == -INFINITY ? 0.f : ex2(m - M);
            wm[s_] = f;
            L += f * wl[s_];
        }
        L = warp_sum(L);
        __syncwarp();
        for (int s0 = 0; s0 < ns; s0 += kBatch) {
            if (s0 > 0) load_o(s0);
#pragma unroll
            for (int k = 0; k < kBatch; ++k) add_o(k, s0 + k < ns ? wm[s0 + k] : 0.f);
        }
    }
    const float inv_l = 1.f / L;
    acc = make_float4(acc.x * inv_l, acc.y * inv_l, acc.z * inv_l, acc.w * inv_l);
    const int64_t oi = (static_cast<int64_t>(row.q_row) * p.n_q_heads + head) * kHeadDim + 4 * c4;
    if (p.out_fp32) {
        *reinterpret_cast<float4 *>(static_cast<float *>(p.out) + oi) = acc;
    } else {
        *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(p.out) + oi) =
            make_uint2(pack_bf16x2(acc.x, acc.y), pack_bf16x2(acc.z, acc.w));
    }
}

}  // namespace ppas
