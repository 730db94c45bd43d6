// Prefill-chunk attention on the 5th-generation tensor cores (tcgen05),
// as a persistent kernel.
//
// One CTA runs on each SM and works through a list of items, each one
// 128-token query tile of two q-heads of the same kv-head (one head when the
// group size is 1) over a range of 128-key KV tiles; both Q tiles share every
// K/V tile the CTA loads.  Per Q tile t the work is a chain
// S_t = Q_t K^T -> softmax -> P_t (bf16, in TMEM) -> O_t += P_t V, and the
// two tiles' chains interleave on the tensor core.
// TMEM, the barriers and the K/V rings live across items, so an item's
// epilogue overlaps the next item's first Q K^T and its K/V loads.
// TMEM (512 columns) holds one S of 128 columns, which the two tiles use in
// turn, and apart from it P_0, P_1 (64 each) and O_0, O_1 (128 each).  A
// softmax thread takes its whole S row into registers first, so S is free
// for the other tile's Q K^T ~200 cycles after it is complete, long before
// P of the row exists; with P over S's own columns (two S buffers of 128,
// no room apart) Q K^T had to wait for the P V that reads P, and the chain
// softmax -> P V -> Q K^T set the pace: 4340 cycles a KV tile of both Q
// tiles (2048 of them MMA), the two softmax warpgroups held apart by a turn
// barrier.  Now they overlap.  The MMA and TMA warps run their loops as
// whole warps and only issue under elect_one(): with a loop of lane 0 the
// operands of every MMA and copy went through ordinary registers, and 8
// MMAs with their commits and the loop around them took the issuing thread
// about 1400 cycles instead of the tensor core's 512.
// Warp roles (512 threads, four warpgroups):
//   warps 0-3   TMA producers: warps 0/1 fetch pages 0-3 / 4-7 of each K
//               tile (3-stage ring), warps 2/3 those of each V tile (2
//               stages), through the block table.  One issuing thread moves
//               only ~7 B/clk of small TMA boxes on GB300, so every tile is
//               fetched by two threads.
//   warp 4      Q K^T issuer: S = Q_t K^T (A = Q in shared
//               memory) for t = 0, 1, as soon as S has been read out.
//   warp 5      P V issuer: O_t += P_t V (A = P in TMEM).  A batch goes
//               out behind the Q K^T batch after the next one (see there).
//   warp 6      Q loader: Q_t of the next item once the last Q K^T of the
//               current item on tile t has completed.
//   warps 8-11  softmax for tile 0, warps 12-15 for tile 1: each thread owns
//               one query row (its TMEM lane), loads its S row, masks by
//               absolute position, runs the online softmax in fp32 (exp2
//               domain) and stores P back to TMEM; at the end of an item it
//               writes O (or a piece's partial).
// Registers move from the producer/MMA warpgroups to the softmax warpgroups
// with setmaxnreg.  The running max is only raised (and O rescaled in TMEM)
// when it grows by more than 2^8; until then the stale max keeps every
// exponent <= 2^8, and the final O / l is exact either way.
// 16384 tokens over an empty prefix, 16/2 heads, 1.0996 TFLOP of causal work:
// 922 us with P over S, 735 with S apart, 620-640 issued by whole warps (565 us,
// 1.95 PFLOP/s, in the first 50 ms of a run; after that the GPU lowers its
// clock, as under a cuBLAS GEMM).  What bounds it now is the tensor core, and
// in a long run the power it draws.
// The host plan may cut a long (query tile, head slot) unit into pieces on
// consecutive CTAs (stream-K): each piece writes its partial (m, l, O) to the
// workspace, and prefill_merge_kernel, launched after this kernel, combines
// the pieces of every cut unit.
// The same CTA body serves the mixed step's single launch (mixed_attn_kernel
// below), whose CTAs past the prefill ones run decode splits
// (attn_decode_body.cuh).
// The kernel is launched with programmatic stream serialization: its set-up
// (TMEM allocation, barriers, tensor-map prefetch) overlaps the kernel before
// it on the stream, and global memory is touched only after grid_dep_wait().
#include <math.h>

#include "attn_decode_body.cuh"
#include "ppas_device.cuh"
#include "ppas_internal.h"

namespace ppas {
namespace {

constexpr int kKT = kPrefillKT;              // keys per KV tile (128)
constexpr int kPagesPerTile = kKT / kPage;   // 8
constexpr int kNK = 3;                       // K ring depth
constexpr int kNV = 2;                       // V ring depth
constexpr uint32_t kBox = 2048;              // one TMA box: 16 rows x 128 B
constexpr uint32_t kHalf = 16384;            // 128 rows x 128 B (64 columns)
constexpr uint32_t kTileBytes = 2 * kHalf;   // a Q, K or V tile: 128 rows x 256 B

constexpr uint32_t kOffQ = 0;
constexpr uint32_t kOffK = kOffQ + 2 * kTileBytes;
constexpr uint32_t kOffV = kOffK + kNK * kTileBytes;
constexpr uint32_t kOffBar = kOffV + kNV * kTileBytes;
enum : int {
    B_Q = 0,                   // [tile]
    B_QEMPTY = B_Q + 2,        // [tile]
    B_KFULL = B_QEMPTY + 2,
    B_KEMPTY = B_KFULL + kNK,
    B_VFULL = B_KEMPTY + kNK,
    B_VEMPTY = B_VFULL + kNV,
    B_SFULL = B_VEMPTY + kNV,  // [tile]
    B_SFREE = B_SFULL + 2,     // the S columns have been read out
    B_PFULL = B_SFREE + 1,     // [tile]
    B_ODONE = B_PFULL + 2,     // [tile]
    B_QKI = B_ODONE + 2,       // [4]: Q K^T batch n, issued (n mod 4)
    B_DRAIN = B_QKI + 4,
    B_COUNT = B_DRAIN + 1
};
constexpr uint32_t kOffTmem = kOffBar + B_COUNT * 8;
constexpr uint32_t kOffAbort = kOffTmem + 4;
static_assert(kOffAbort + 4 <= kOffBar + 256, "barrier area");
constexpr uint32_t kSmemBytes = kOffBar + 256 + 1024;  // + alignment slack
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0;    // one S (128 columns) that the two tiles use in turn
constexpr uint32_t kColP = 128;  // P of tile t at kColP + 64 t
constexpr uint32_t kColO = 256;  // O of tile t at kColO + 128 t
constexpr float kRescaleThreshold = 8.0f;  // log2 units
constexpr int kThreads = 512;
constexpr int kMmaWarp = 4;       // warps 4..7 form the MMA warpgroup
constexpr int kQWarp = 6;         // loads Q (warps 4, 5 issue MMAs)
constexpr int kSoftmaxWarp0 = 8;  // warps 8..11 tile 0, 12..15 tile 1
// register split: 8 warps x 56 + 8 warps x 200 = 512 threads x 128 at launch
constexpr int kRegsSmall = 56;
constexpr int kRegsLarge = 200;
static_assert(8 * 32 * kRegsSmall + 8 * 32 * kRegsLarge <= kThreads * 128, "register split");

constexpr uint32_t kIdescQK = idesc_bf16_f32(128, kKT, false, false);  // B = K rows (K-major)
constexpr uint32_t kIdescPV = idesc_bf16_f32(128, 128, false, true);   // B = V rows (MN-major)

// A row of S: 128 TMEM columns of this warp's lanes (one row per thread) in four
// loads under one wait.  One statement: a load's registers hold nothing before
// the wait, so the compiler must not come to move or spill them in between.
__device__ __forceinline__ void tmem_ld128_sync(uint32_t taddr, float (&r)[128]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
        "%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%128];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
        "%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,"
        "%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%129];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
        "%64,%65,%66,%67,%68,%69,%70,%71,%72,%73,%74,%75,%76,%77,%78,%79,"
        "%80,%81,%82,%83,%84,%85,%86,%87,%88,%89,%90,%91,%92,%93,%94,%95}, [%130];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
        "%96,%97,%98,%99,%100,%101,%102,%103,%104,%105,%106,%107,%108,%109,%110,%111,"
        "%112,%113,%114,%115,%116,%117,%118,%119,%120,%121,%122,%123,%124,%125,%126,%127}, [%131];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
          "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15]),
          "=f"(r[16]), "=f"(r[17]), "=f"(r[18]), "=f"(r[19]), "=f"(r[20]), "=f"(r[21]), "=f"(r[22]), "=f"(r[23]),
          "=f"(r[24]), "=f"(r[25]), "=f"(r[26]), "=f"(r[27]), "=f"(r[28]), "=f"(r[29]), "=f"(r[30]), "=f"(r[31]),
          "=f"(r[32]), "=f"(r[33]), "=f"(r[34]), "=f"(r[35]), "=f"(r[36]), "=f"(r[37]), "=f"(r[38]), "=f"(r[39]),
          "=f"(r[40]), "=f"(r[41]), "=f"(r[42]), "=f"(r[43]), "=f"(r[44]), "=f"(r[45]), "=f"(r[46]), "=f"(r[47]),
          "=f"(r[48]), "=f"(r[49]), "=f"(r[50]), "=f"(r[51]), "=f"(r[52]), "=f"(r[53]), "=f"(r[54]), "=f"(r[55]),
          "=f"(r[56]), "=f"(r[57]), "=f"(r[58]), "=f"(r[59]), "=f"(r[60]), "=f"(r[61]), "=f"(r[62]), "=f"(r[63]),
          "=f"(r[64]), "=f"(r[65]), "=f"(r[66]), "=f"(r[67]), "=f"(r[68]), "=f"(r[69]), "=f"(r[70]), "=f"(r[71]),
          "=f"(r[72]), "=f"(r[73]), "=f"(r[74]), "=f"(r[75]), "=f"(r[76]), "=f"(r[77]), "=f"(r[78]), "=f"(r[79]),
          "=f"(r[80]), "=f"(r[81]), "=f"(r[82]), "=f"(r[83]), "=f"(r[84]), "=f"(r[85]), "=f"(r[86]), "=f"(r[87]),
          "=f"(r[88]), "=f"(r[89]), "=f"(r[90]), "=f"(r[91]), "=f"(r[92]), "=f"(r[93]), "=f"(r[94]), "=f"(r[95]),
          "=f"(r[96]), "=f"(r[97]), "=f"(r[98]), "=f"(r[99]), "=f"(r[100]), "=f"(r[101]), "=f"(r[102]), "=f"(r[103]),
          "=f"(r[104]), "=f"(r[105]), "=f"(r[106]), "=f"(r[107]), "=f"(r[108]), "=f"(r[109]), "=f"(r[110]), "=f"(r[111]),
          "=f"(r[112]), "=f"(r[113]), "=f"(r[114]), "=f"(r[115]), "=f"(r[116]), "=f"(r[117]), "=f"(r[118]), "=f"(r[119]),
          "=f"(r[120]), "=f"(r[121]), "=f"(r[122]), "=f"(r[123]), "=f"(r[124]), "=f"(r[125]), "=f"(r[126]), "=f"(r[127])
        : "r"(taddr), "r"(taddr + 32), "r"(taddr + 64), "r"(taddr + 96)
        : "memory");
}

// 16 TMEM columns of this warp's lanes
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t *r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

__device__ __forceinline__ void tmem_st32_f(uint32_t taddr, const float (&v)[32]) {
    uint32_t r[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(v[i]);
    tmem_st32(taddr, r);
}

// two fp32 lanes at once (Blackwell packed FP32 pipe)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Stores 32 consecutive output columns of the warp's 32 rows, scaled by inv_l
// (v: this thread's row; first_row: the warp's first row of the tile, whose
// first rows_valid rows exist; dst: column 0 of the chunk in the warp's first
// row, `stride` elements a row).  A thread holds a row, so bf16 stores of its
// own 64 bytes would touch 32 rows an instruction; the four lanes of a quad
// first trade 16-byte chunks (a 4 x 4 transpose by shuffles), after which an
// instruction covers 8 rows x 64 bytes.  (One item of 16 KV tiles after the
// other, 512 queries over 2048 keys: 25.3 us a layer with direct stores, 24.2
// with the exchange; the same through a shared-memory buffer measured 23.8 but
// would take a stage of the K ring.)
__device__ __forceinline__ void store_rows(void *dst, bool fp32, int64_t stride, int lane, int first_row,
                                           int rows_valid, const float (&v)[32], float inv_l) {
    if (fp32) {
        if (first_row + lane >= rows_valid) return;
        float4 *d = reinterpret_cast<float4 *>(static_cast<float *>(dst) + lane * stride);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            d[i] = make_float4(v[4 * i] * inv_l, v[4 * i + 1] * inv_l, v[4 * i + 2] * inv_l, v[4 * i + 3] * inv_l);
        return;
    }
    uint32_t w[4][4];  // [chunk of 8 columns][pair]; afterwards [row of the quad][pair] of chunk lane & 3
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i >> 2][i & 3] = pack_bf16x2(v[2 * i] * inv_l, v[2 * i + 1] * inv_l);
#pragma unroll
    for (int step = 1; step <= 2; ++step) {
        const bool hi = (lane & step) != 0;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int k0 = step == 1 ? 2 * x : x, k1 = k0 + step;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, hi ? w[k0][e] : w[k1][e], step);
                w[k0][e] = hi ? got : w[k0][e];
                w[k1][e] = hi ? w[k1][e] : got;
            }
        }
    }
    const int quad = lane & ~3;
    __nv_bfloat16 *d = static_cast<__nv_bfloat16 *>(dst) + quad * stride + (lane & 3) * 8;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (first_row + quad + i < rows_valid)
            *reinterpret_cast<uint4 *>(d + i * stride) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// The parts of a work item each role needs (read from the kernel parameters).
struct ItemView {
    const int32_t *table;  // the sequence's block-table row
    int ctx_len;
    int kvh;               // kv-head of the item's head slot
    int kt0, n_kt;         // KV tiles [kt0, kt0 + n_kt)
};

template <class P>
__device__ __forceinline__ ItemView item_view(const P &p, int w) {
    const PrefillWork wk = p.work[w];
    const PrefillSeq sq = p.seqs[wk.seq];
    ItemView v;
    v.table = p.block_tables + static_cast<int64_t>(sq.table_row) * p.table_stride;
    v.ctx_len = sq.ctx_len;
    v.kvh = wk.slot * p.heads_per_cta / p.group;
    v.kt0 = wk.kt0;
    v.n_kt = wk.kt1 - wk.kt0;
    return v;
}

// pages of KV tile j that hold at least one context key
__device__ __forceinline__ int pages_in(int ctx_len, int j) {
    return min(kPagesPerTile, (ctx_len - j * kKT + kPage - 1) / kPage);
}

}  // namespace

// The work of prefill CTA `cta` of the plan in p (all 512 threads).
template <class P>
__device__ __forceinline__ void prefill_cta(const CUtensorMap &tm_q, const CUtensorMap &tm_k,
                                            const CUtensorMap &tm_v, const P &p, int cta) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t sb = (raw_s + 1023u) & ~1023u;  // 1024-aligned for the 128-byte swizzle
    uint8_t *const sg = smem_raw + (sb - raw_s);

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (uniform)
    const int hpc = p.heads_per_cta;
    // this CTA's items, in order
    const int w_beg = p.cta_begin[cta], w_end = p.cta_begin[cta + 1];

    auto bar = [&](int i) { return sb + kOffBar + 8u * static_cast<uint32_t>(i); };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sg + kOffAbort);

    if (warp == kMmaWarp) {
        tmem_alloc(sb + kOffTmem, kTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int t = 0; t < 2; ++t) {
            mbar_init(bar(B_Q + t), 1);
            mbar_init(bar(B_QEMPTY + t), 1);
        }
        for (int s = 0; s < kNK; ++s) {
            mbar_init(bar(B_KFULL + s), 2);      // two producer threads per tile
            mbar_init(bar(B_KEMPTY + s), 1);
        }
        for (int s = 0; s < kNV; ++s) {
            mbar_init(bar(B_VFULL + s), 2);
            mbar_init(bar(B_VEMPTY + s), 1);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(bar(B_SFULL + t), 1);
            mbar_init(bar(B_PFULL + t), 4);
            mbar_init(bar(B_ODONE + t), 1);
        }
        mbar_init(bar(B_SFREE), 4);
        for (int i = 0; i < 4; ++i) mbar_init(bar(B_QKI + i), 1);
        mbar_init(bar(B_DRAIN), 2);
        *abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tm_q);
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(sg + kOffTmem), 0);
    // the set-up above overlaps the previous kernel of the stream; global
    // memory (KV pages, Q, block tables, outputs) only after it has completed
    grid_dep_wait();
    // KV tiles whose copies this producer has issued; the Q loader's Q tiles (tile n
    // of them has the barrier B_Q + n % hpc)
    int issued = 0;

    if (warp < 4) {
        // ------------------------------------------------------------ K/V producers
        // The rings run on across item boundaries: tile g of this CTA (over
        // all its items) goes to stage g % depth.
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsSmall));
        if (w_beg < w_end) {
            const bool is_v = warp >= 2;
            const int pg_lo = (warp & 1) * (kPagesPerTile / 2);  // this warp's pages of each tile
            const int ns = is_v ? kNV : kNK;
            const CUtensorMap *tm = is_v ? &tm_v : &tm_k;
            const uint32_t ring = sb + (is_v ? kOffV : kOffK);
            const int full0 = is_v ? B_VFULL : B_KFULL, empty0 = is_v ? B_VEMPTY : B_KEMPTY;
            const int pg = pg_lo + (lane & 3);  // lane i (mod 4) looks after page pg_lo + i
            // page ids of the next tile are loaded while the current one is issued
            int id = 0;
            auto load_id = [&](const ItemView &v, int jj) {
                const int j = v.kt0 + jj;
                id = pg < pages_in(v.ctx_len, j) ? __ldg(v.table + j * kPagesPerTile + pg) : 0;
            };
            int w = w_beg, jj = 0;
            ItemView cur = item_view(p, w);
            load_id(cur, 0);
            for (;;) {
                const int g = issued;
                const int s = g % ns;
                const int np = max(0, min(kPagesPerTile / 2, pages_in(cur.ctx_len, cur.kt0 + jj) - pg_lo));
                if (pg - pg_lo < np && (id < 0 || id >= p.num_blocks)) {
                    if (lane < 4) report_error(p.err, PPAS_DEVERR_BAD_INDEX);
                    id = 0;  // keep the barrier's byte count consistent
                }
                const int row = (id * p.n_kv_heads + cur.kvh) * kPage;
                // the next tile: this item's, else the next item's first
                int jn = jj + 1, wn = w;
                if (jn == cur.n_kt) {
                    jn = 0;
                    ++wn;
                }
                const bool more = wn < w_end;
                const ItemView nxt = (more && wn != w) ? item_view(p, wn) : cur;
                if (more) load_id(nxt, jn);
                if (g >= ns && !mbar_wait_warp(bar(empty0 + s), ((g / ns) & 1) ^ 1, p.err)) {
                    *abort_flag = 1;
                    break;
                }
                int rows[kPagesPerTile / 2];
#pragma unroll
                for (int i = 0; i < kPagesPerTile / 2; ++i) rows[i] = __shfl_sync(0xffffffffu, row, i);
                if (elect_one()) {
                    const uint32_t b = bar(full0 + s);
                    mbar_expect_tx(b, static_cast<uint32_t>(np) * 2 * kBox);
                    const uint32_t dst = ring + s * kTileBytes + pg_lo * kBox;
#pragma unroll
                    for (int i = 0; i < kPagesPerTile / 2; ++i)
                        if (i < np) {
                            tma_load_2d(dst + i * kBox, tm, 0, rows[i], b);
                            tma_load_2d(dst + kHalf + i * kBox, tm, 64, rows[i], b);
                        }
                }
                __syncwarp();
                ++issued;
                if (!more) break;
                w = wn;
                jj = jn;
                cur = nxt;
            }
        }
    } else if (warp < kSoftmaxWarp0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsSmall));
        if (warp == kMmaWarp && w_beg < w_end) {
            // -------------------------------------------------------- Q K^T issuer
            // descriptors are built once; advancing one operand by b bytes
            // adds b >> 4 to the start-address field (no carry: < 256 KB)
            const uint64_t dq0 = smem_desc_sw128(sb + kOffQ, 16, 1024);
            const uint64_t dk0 = smem_desc_sw128(sb + kOffK, 16, 1024);
            bool ok = true;
            int g = 0;  // KV tiles of this CTA so far
            int n = 0;  // S tiles so far (hpc per KV tile)
            for (int w = w_beg, i = 0; ok && w < w_end; ++w, ++i) {
                const ItemView v = item_view(p, w);
                for (int jj = 0; ok && jj < v.n_kt; ++jj, ++g) {
                    const int sk = g % kNK;
                    if (!mbar_wait_warp(bar(B_KFULL + sk), (g / kNK) & 1, p.err)) { ok = false; break; }
                    const uint64_t dk = dk0 + ((sk * kTileBytes) >> 4);
                    for (int t = 0; t < hpc; ++t, ++n) {
                        if (jj == 0 && !mbar_wait_warp(bar(B_Q + t), i & 1, p.err)) { ok = false; break; }
                        // the S columns, once the softmax before has read them out
                        if (n >= 1 && !mbar_wait_warp(bar(B_SFREE), (n - 1) & 1, p.err)) { ok = false; break; }
                        tc_fence_after();
                        const uint64_t dq = dq0 + ((t * kTileBytes) >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk) {
                                const uint32_t o = (kk >> 2) * kHalf + (kk & 3) * 32;
                                umma_bf16(tmem + kColS, dq + (o >> 4), dk + (o >> 4), kIdescQK, kk > 0 ? 1u : 0u);
                            }
                            umma_commit(bar(B_SFULL + t));
                            mbar_arrive(bar(B_QKI + (n & 3)));  // P V (n - hpc) may follow
                            if (t == hpc - 1) umma_commit(bar(B_KEMPTY + sk));
                            // the item's last Q K^T frees Q_t for the next item
                            if (jj == v.n_kt - 1) umma_commit(bar(B_QEMPTY + t));
                        }
                        __syncwarp();
                    }
                }
            }
            if (!ok) *abort_flag = 1;
            // every MMA issued so far completes before TMEM is released
            if (elect_one()) umma_commit(bar(B_DRAIN));
            __syncwarp();
            mbar_wait(bar(B_DRAIN), 0, p.err);
        } else if (warp == kMmaWarp + 1 && w_beg < w_end) {
            // -------------------------------------------------------- P V issuer
            const uint64_t dv0 = smem_desc_sw128(sb + kOffV, kHalf, 1024);
            bool ok = true;
            int g = 0;
            for (int w = w_beg; ok && w < w_end; ++w) {
                const ItemView v = item_view(p, w);
                for (int jj = 0; ok && jj < v.n_kt; ++jj, ++g) {
                    const int sv = g % kNV;
                    if (!mbar_wait_warp(bar(B_VFULL + sv), (g / kNV) & 1, p.err)) { ok = false; break; }
                    const uint64_t dv = dv0 + ((sv * kTileBytes) >> 4);
                    const int chunks = pages_in(v.ctx_len, v.kt0 + jj);
                    for (int t = 0; t < hpc; ++t) {
                        if (!mbar_wait_warp(bar(B_PFULL + t), g & 1, p.err)) { ok = false; break; }
                        // P V (n) goes out behind Q K^T (n + hpc): P V (n) and
                        // the read-out of S (n + hpc - 1), which lets that
                        // Q K^T start, are ready at about the same time, and
                        // the tensor core would work on both batches in turn
                        // while the softmax waits for S (16384 tokens: 695 us
                        // without this rule, 623 with it).  Not for the last KV
                        // tile of an item: the Q K^T after it may wait for the
                        // epilogues.
                        // Q K^T runs at most n + 2 hpc ahead of P V (n) (the
                        // softmax stores P (n + hpc) only after P V (n)), so
                        // four barriers keep its phases apart.
                        if (jj + 1 < v.n_kt) {
                            const int gate = (g + 1) * hpc + t;
                            if (!mbar_wait_warp(bar(B_QKI + (gate & 3)), (gate >> 2) & 1, p.err)) { ok = false; break; }
                        }
                        tc_fence_after();
                        // O_t += P_t V(j), P_t from TMEM; the item's first tile overwrites O_t
                        const uint32_t d_p = tmem + kColP + t * 64, d_o = tmem + kColO + t * 128;
                        if (elect_one()) {
                            if (chunks == kPagesPerTile) {
#pragma unroll
                                for (int kk = 0; kk < kPagesPerTile; ++kk)
                                    umma_bf16_ts(d_o, d_p + kk * 8, dv + ((kk * 2048) >> 4), kIdescPV,
                                                 (jj > 0 || kk > 0) ? 1u : 0u);
                            } else {
                                for (int kk = 0; kk < chunks; ++kk)
                                    umma_bf16_ts(d_o, d_p + kk * 8, dv + ((kk * 2048) >> 4), kIdescPV,
                                                 (jj > 0 || kk > 0) ? 1u : 0u);
                            }
                            umma_commit(bar(B_ODONE + t));
                            if (t == hpc - 1) umma_commit(bar(B_VEMPTY + sv));
                        }
                        __syncwarp();
                    }
                }
            }
            if (!ok) *abort_flag = 1;
            if (elect_one()) umma_commit(bar(B_DRAIN));
            __syncwarp();
            mbar_wait(bar(B_DRAIN), 0, p.err);
        } else if (warp == kQWarp) {
            // -------------------------------------------------------- Q loader
            // Q tile t of item i is loaded once the last Q K^T of item i-1 on
            // that tile has completed.
            for (int w = w_beg, i = 0; w < w_end; ++w, ++i) {
                const PrefillWork wk = p.work[w];
                const int qrow = p.seqs[wk.seq].q_start + wk.qt * kTileQ;
                const int h0 = wk.slot * hpc;
                bool ok = true;
                for (int t = 0; t < hpc; ++t) {
                    if (i > 0 && !mbar_wait_warp(bar(B_QEMPTY + t), (i - 1) & 1, p.err)) {
                        ok = false;
                        break;
                    }
                    if (elect_one()) {
                        mbar_expect_tx(bar(B_Q + t), kTileBytes);
                        tma_load_3d(sb + kOffQ + t * kTileBytes, &tm_q, 0, h0 + t, qrow, bar(B_Q + t));
                        tma_load_3d(sb + kOffQ + t * kTileBytes + kHalf, &tm_q, 64, h0 + t, qrow, bar(B_Q + t));
                    }
                    __syncwarp();
                    ++issued;
                }
                if (!ok) {
                    *abort_flag = 1;
                    break;
                }
            }
        }
    } else {
        // ------------------------------------------------------------ softmax warpgroups
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsLarge));
      if ((warp - kSoftmaxWarp0) / 4 < hpc) {
        const int t = (warp - kSoftmaxWarp0) / 4;
        const int wq = warp & 3;
        const int r = wq * 32 + lane;  // query row == TMEM lane
        const uint32_t t_lane = tmem + (static_cast<uint32_t>(wq * 32) << 16);
        const uint32_t t_s = t_lane + kColS, t_p = t_lane + kColP + t * 64, t_o = t_lane + kColO + t * 128;
        const float sl2 = p.scale_log2;
        bool ok = true;
        int g = 0;  // KV tiles of this CTA so far

        for (int w = w_beg; w < w_end; ++w) {
            // what the KV loop needs (the epilogue reads the rest again)
            int pos, min_pos, kt0, n_kt, last_j, ctx_len;
            {
                const PrefillWork wk = p.work[w];
                const PrefillSeq sq = p.seqs[wk.seq];
                const int t0 = wk.qt * kTileQ;
                const int prefix = sq.ctx_len - sq.q_len;
                ctx_len = sq.ctx_len;
                pos = min(prefix + t0 + r, ctx_len - 1);  // last key this row may see
                min_pos = prefix + t0;
                last_j = (prefix + t0 + min(kTileQ, sq.q_len - t0) - 1) / kKT;  // last KV tile of the causal range
                kt0 = wk.kt0;
                n_kt = wk.kt1 - wk.kt0;
            }
            float m_used = -INFINITY, l_run = 0.f;

            for (int jj = 0; ok && jj < n_kt; ++jj, ++g) {
                const int j = kt0 + jj;  // absolute KV tile
                ok = mbar_wait_warp(bar(B_SFULL + t), g & 1, p.err);
                if (!ok) break;
                tc_fence_after();
                float s[kKT];
                tmem_ld128_sync(t_s, s);
                // S is in registers: the other tile's Q K^T may overwrite it
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_SFREE));
                const int first_key = j * kKT;
                if (first_key + kKT - 1 > min_pos) {
                    // one bit per visible key: a row sees keys up to pos
                    const int lim = pos - first_key;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int n = min(max(lim - 32 * q + 1, 0), 32);
                        const uint32_t seen = static_cast<uint32_t>((1ull << n) - 1);
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (!((seen >> i) & 1u)) s[32 * q + i] = -INFINITY;
                    }
                }
                // four independent chains over the 128 scores, two new ones per max3
                float mx0 = fmaxf(s[0], s[4]), mx1 = fmaxf(s[1], s[5]);
                float mx2 = fmaxf(s[2], s[6]), mx3 = fmaxf(s[3], s[7]);
#pragma unroll
                for (int i = 8; i < kKT; i += 8) {
                    mx0 = max3(mx0, s[i], s[i + 4]);
                    mx1 = max3(mx1, s[i + 1], s[i + 5]);
                    mx2 = max3(mx2, s[i + 2], s[i + 6]);
                    mx3 = max3(mx3, s[i + 3], s[i + 7]);
                }
                const float m_cand = max3(fmaxf(mx0, mx1), mx2, mx3) * sl2;
                const bool need = m_cand > m_used + kRescaleThreshold;
                float alpha = 1.f;
                if (need) {
                    alpha = ex2(m_used - m_cand);
                    m_used = m_cand;
                }
                // a row whose keys in this range are all masked keeps m = -inf and p = 0
                const float neg_m = m_used == -INFINITY ? 0.f : -m_used;
                const float2 sl2x2 = make_float2(sl2, sl2), negx2 = make_float2(neg_m, neg_m);
                float2 ra = make_float2(0.f, 0.f), rb = make_float2(0.f, 0.f);
                // P (bf16 pairs, lower key in the low half), packed as the
                // exponentials come.  (The pass alone, two warpgroups at work:
                // 1799 cycles with each x64 load awaited by itself and packing
                // after the last exponential, 1392 with all loads issued
                // together and packing in this loop.)
                uint32_t pk[4][16];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
#pragma unroll
                    for (int i = 0; i < 32; i += 4) {
                        const float *v = s + 32 * q + i;
                        const float2 xa = fma2(make_float2(v[0], v[1]), sl2x2, negx2);
                        const float2 xb = fma2(make_float2(v[2], v[3]), sl2x2, negx2);
                        const float2 ea = make_float2(ex2(xa.x), ex2(xa.y)), eb = make_float2(ex2(xb.x), ex2(xb.y));
                        ra = add2(ra, ea);
                        rb = add2(rb, eb);
                        pk[q][i / 2] = pack_bf16x2(ea.x, ea.y);
                        pk[q][i / 2 + 1] = pack_bf16x2(eb.x, eb.y);
                    }
                }
                // P V (g-1) has read the P before and O is stable
                if (g >= 1) {
                    ok = mbar_wait_warp(bar(B_ODONE + t), (g - 1) & 1, p.err);
                    if (!ok) break;
                    tc_fence_after();
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_st16(t_p + 16 * q, pk[q]);
                l_run = l_run * alpha + ((ra.x + ra.y) + (rb.x + rb.y));
                if (j == last_j) {
                    // rows of the last page past the context may hold anything:
                    // zero them in V so that P = 0 times V stays 0.  Each tile's
                    // warpgroup does it before releasing its own P, so both P V
                    // products are ordered after it (the second writes the same
                    // zeros again)
                    const int keys_here = min(kKT, ctx_len - first_key);
                    if (keys_here & (kPage - 1)) {
                        const int s_idx = g % kNV;
                        ok = __all_sync(0xffffffffu, mbar_wait(bar(B_VFULL + s_idx), (g / kNV) & 1, p.err));
                        if (!ok) break;
                        const int pg = keys_here / kPage, from = keys_here & (kPage - 1);
                        const int n = (kPage - from) * 8;  // 16-byte chunks per half
                        uint8_t *vb = sg + kOffV + s_idx * kTileBytes + pg * kBox + from * 128;
                        for (int c = r; c < 2 * n; c += 128)
                            *reinterpret_cast<uint4 *>(vb + (c / n) * kHalf + (c % n) * 16) = make_uint4(0, 0, 0, 0);
                        fence_proxy_async_smem();
                    }
                }
                if (jj >= 1 && __any_sync(0xffffffffu, need)) {
#pragma unroll 1
                    for (int c4 = 0; c4 < 4; ++c4) {
                        float v[32];
                        tmem_ld32_sync(t_o + c4 * 32, v);
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] *= alpha;
                        tmem_st32_f(t_o + c4 * 32, v);
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_PFULL + t));
            }

            // ---- epilogue of the item: O_t after its last P V
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(bar(B_ODONE + t), (g - 1) & 1, p.err));
            const PrefillWork wk = p.work[w];
            const PrefillSeq sq = p.seqs[wk.seq];
            const int t0 = wk.qt * kTileQ;
            const int rows_valid = min(kTileQ, sq.q_len - t0);
            if (wk.part == kNoPart) {
                if (ok) {
                    tc_fence_after();
                    const float inv_l = 1.f / l_run;
                    const int64_t stride = static_cast<int64_t>(p.n_q_heads) * kHeadDim;
                    const int64_t at = (sq.q_start + t0 + wq * 32) * stride + (wk.slot * hpc + t) * kHeadDim;
                    uint8_t *dst = static_cast<uint8_t *>(p.out) + at * (p.out_fp32 ? 4 : 2);
                    // (not unrolled: this code runs cold, so its length is its cost)
#pragma unroll 1
                    for (int c4 = 0; c4 < 4; ++c4) {
                        float v[32];
                        tmem_ld32_sync(t_o + c4 * 32, v);
                        store_rows(dst + c4 * (p.out_fp32 ? 128 : 64), p.out_fp32 != 0, stride, lane, wq * 32, rows_valid,
                                   v, inv_l);
                    }
                }
            } else if (ok) {
                // a piece of a split unit: this range's (m, l, O) for the row;
                // the merge kernel combines the unit's pieces after this
                // launch.  Partial O of one (piece, head) is stored as 32
                // chunks of [128 rows][4 floats], so that a store instruction
                // of a warp writes 512 contiguous bytes.
                tc_fence_after();
                const int64_t b = static_cast<int64_t>(wk.part) * hpc + t;
                float4 *dst = reinterpret_cast<float4 *>(p.part_o) + b * (kHeadDim / 4) * kTileQ + r;
#pragma unroll 1
                for (int c4 = 0; c4 < 4; ++c4) {
                    float v[32];
                    tmem_ld32_sync(t_o + c4 * 32, v);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        __stcg(dst + (c4 * 8 + i) * kTileQ, make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
                }
                // two scalar stores: the paired float2 store costs the softmax loop
                // register spills at its 200-register budget
                __stcg(p.part_ml + (b * kTileQ + r) * 2, m_used);
                __stcg(p.part_ml + (b * kTileQ + r) * 2 + 1, l_run);
            }
        }
        if (!ok) *abort_flag = 1;
      }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
    // a wait ran out: the copies in flight land before the CTA leaves.  (Last, and
    // once for all rings: before the release of TMEM, or by each producer at its
    // end, it cost a step of short items, or a long one, 0.3-1 %.)
    if (*abort_flag && issued > 0) {
        const bool q = warp == kQWarp, v = warp >= 2;
        ring_land(bar(q ? B_Q : v ? B_VFULL : B_KFULL), issued, q ? hpc : v ? kNV : kNK, lane);
    }
}

__global__ void __launch_bounds__(kThreads, 1)
    prefill_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                        const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ PrefillParams p) {
    prefill_cta(tm_q, tm_k, tm_v, p, blockIdx.x);
}

// A whole mixed step in one launch: CTAs [0, p.pf.n_ctas) run the prefill
// items, the CTAs after them the decode splits (one (row, kv-head, split)
// each, on warps 0-7; warps 8-15 hand their registers to them and leave).
// The block scheduler starts CTAs in index order, so the first wave holds
// every prefill CTA and fills the SMs left to the decode rows.
__global__ void __launch_bounds__(kThreads, 1)
    mixed_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                      const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ MixedParams p) {
    if (static_cast<int>(blockIdx.x) < p.pf.n_ctas) {
        prefill_cta(tm_q, tm_k, tm_v, p.pf, blockIdx.x);
        return;
    }
    if ((threadIdx.x >> 5) >= kDecodeWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsSmall));
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsLarge));
    decode_cta<true>(tm_k, tm_v, p.dc, static_cast<int>(blockIdx.x) - p.pf.n_ctas);
}
static_assert(kDecodeThreads == 8 * 32 && kDecodeSmemBytes <= kSmemBytes,
              "decode CTAs of a mixed launch: warps 0-7 of the CTA, within its shared memory");

// Combines the pieces of a split unit:
//   o = sum_i 2^(m_i - M) o_i / sum_i 2^(m_i - M) l_i,  M = max_i m_i
// (m in log2 units), taking the pieces four at a time with the running
// maximum (exact up to rounding).  CTA (unit, head t, 32 rows, 64 columns); a
// warp takes the 32 rows (a lane a row) and 8 columns, so a load of a partial
// is 512 contiguous bytes, a lane has up to 12 loads in flight, and a bf16
// store is 16 bytes.  Bound by the latency of its rounds of four pieces and by
// L2.  With one float4 a thread and four rows a warp it took 5.2 us of a
// 512-token layer's 19.6 and 7.7 of the 4 x 512 step's 137; the layers now take
// 18.5-18.8 and 134 (16 columns a lane: 18.7 and 135.4; 4: 18.6 and 135.6;
// eight pieces a round: 19.6 and 136.8), 128 tokens over 25,000 (19 pieces a
// unit) 28.3 -> 25.6.
__global__ void __launch_bounds__(256) prefill_merge_kernel(const __grid_constant__ MergeParams p) {
    grid_dep_wait();  // the partials come from the prefill launch before this one
    const int hpc = p.heads_per_cta;
    const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) + 8 * (blockIdx.x & 1);
    const int r = ((blockIdx.x >> 1) & 3) * 32 + lane;
    int rest = blockIdx.x >> 3;
    const int t = rest % hpc;
    const MergeUnit mu = p.units[rest / hpc];
    const int ns = mu.n_splits;
    constexpr int kC = 2;  // 16-byte chunks of a lane
    float M = -INFINITY, L = 0.f;
    float4 acc[kC];
#pragma unroll
    for (int c = 0; c < kC; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i0 = 0; i0 < ns; i0 += 4) {
        float2 ml[4];
        float4 o[4][kC];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t b = (static_cast<int64_t>(mu.part) + i0 + k) * hpc + t;
            ml[k] = i0 + k < ns ? __ldcg(reinterpret_cast<const float2 *>(p.part_ml + (b * kTileQ + r) * 2))
                                : make_float2(-INFINITY, 0.f);
#pragma unroll
            for (int c = 0; c < kC; ++c)
                o[k][c] = i0 + k < ns ? __ldcg(reinterpret_cast<const float4 *>(p.part_o) +
                                               (b * (kHeadDim / 4) + warp * kC + c) * kTileQ + r)
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const float mn = fmaxf(fmaxf(M, fmaxf(ml[0].x, ml[1].x)), fmaxf(ml[2].x, ml[3].x));
        if (mn == -INFINITY) continue;  // every key of these pieces is masked for this row
        const float sc = M == -INFINITY ? 0.f : ex2(M - mn);
        L *= sc;
#pragma unroll
        for (int c = 0; c < kC; ++c) acc[c] = make_float4(acc[c].x * sc, acc[c].y * sc, acc[c].z * sc, acc[c].w * sc);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float f = ml[k].x == -INFINITY ? 0.f : ex2(ml[k].x - mn);
            L += f * ml[k].y;
#pragma unroll
            for (int c = 0; c < kC; ++c)
                acc[c] = make_float4(acc[c].x + f * o[k][c].x, acc[c].y + f * o[k][c].y, acc[c].z + f * o[k][c].z,
                                     acc[c].w + f * o[k][c].w);
        }
        M = mn;
    }
    if (r >= mu.rows_valid) return;
    const float inv_l = 1.f / L;
    const int64_t orow = static_cast<int64_t>(mu.out_row0 + r) * p.n_q_heads + mu.head0 + t;
    const int64_t col = orow * kHeadDim + warp * (4 * kC);
    if (p.out_fp32) {
        float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(p.out) + col);
#pragma unroll
        for (int c = 0; c < kC; ++c)
            dst[c] = make_float4(acc[c].x * inv_l, acc[c].y * inv_l, acc[c].z * inv_l, acc[c].w * inv_l);
    } else {
        uint4 *dst = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(p.out) + col);
#pragma unroll
        for (int c = 0; c < kC; c += 2)
            dst[c / 2] = make_uint4(pack_bf16x2(acc[c].x * inv_l, acc[c].y * inv_l),
                                    pack_bf16x2(acc[c].z * inv_l, acc[c].w * inv_l),
                                    pack_bf16x2(acc[c + 1].x * inv_l, acc[c + 1].y * inv_l),
                                    pack_bf16x2(acc[c + 1].z * inv_l, acc[c + 1].w * inv_l));
    }
}

cudaError_t launch_prefill_merge(const MergeParams &p, cudaStream_t st) {
    if (p.n_units <= 0) return cudaSuccess;
    PdlLaunch l(dim3(p.n_units * p.heads_per_cta * 8), dim3(256), 0, st);
    return cudaLaunchKernelEx(&l.cfg, prefill_merge_kernel, p);
}

static std::atomic<uint64_t> g_prefill_smem_set{0};
static std::atomic<uint64_t> g_mixed_smem_set{0};

cudaError_t prepare_prefill() {
    return ensure_smem_limit(prefill_attn_kernel, static_cast<int>(kSmemBytes), g_prefill_smem_set);
}

cudaError_t prepare_mixed() {
    return ensure_smem_limit(mixed_attn_kernel, static_cast<int>(kSmemBytes), g_mixed_smem_set);
}

cudaError_t launch_prefill(const CUtensorMap &tm_q, const CUtensorMap &tm_k, const CUtensorMap &tm_v,
                           const PrefillParams &p, cudaStream_t st) {
    const cudaError_t e = prepare_prefill();
    if (e != cudaSuccess) return e;
    if (p.n_ctas <= 0) return cudaSuccess;
    PdlLaunch l(dim3(p.n_ctas), dim3(kThreads), kSmemBytes, st);
    return cudaLaunchKernelEx(&l.cfg, prefill_attn_kernel, tm_q, tm_k, tm_v, p);
}

cudaError_t launch_mixed(const CUtensorMap &tm_q, const CUtensorMap &tm_k, const CUtensorMap &tm_v,
                         const MixedParams &p, cudaStream_t st) {
    const cudaError_t e = prepare_mixed();
    if (e != cudaSuccess) return e;
    const int grid = p.pf.n_ctas + p.dc.n_ctas;
    if (grid <= 0) return cudaSuccess;
    PdlLaunch l(dim3(grid), dim3(kThreads), kSmemBytes, st);
    return cudaLaunchKernelEx(&l.cfg, mixed_attn_kernel, tm_q, tm_k, tm_v, p);
}

}  // namespace ppas
