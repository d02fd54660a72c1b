// Tensor-core chunked prefill for sm_103a: the full attention of Eq. 3 for the query rows of a
// chunk of new tokens, over the paged Value-Only Cache, under the causal mask.
//
// One CTA per (query head h, sequence b, block of 128 query rows); head_dim 128. The rows of the
// block sit at consecutive positions p0 .. p0 + 127 of the sequence (the chunk is the tail of the
// cached rows), so the CTA walks the cache tiles 0 .. p_last / 128 and masks only the last ones.
// Small chunks share more (kShared): a block's 128 rows hold several heads of a group, which read
// the same tiles, and while the blocks leave SMs idle, a cluster of up to 8 CTAs splits a block's
// tiles and merges the states through distributed shared memory. (Chunk append and prefill, back to
// back: 4 sequences of 4000 tokens, 16-token chunks, 12 heads: 52 -> 17 us; 2 of 8000 tokens, 100-token
// chunks, 32 heads: 93 -> 51.)
//
//   routing  Q_r = Q . W^R[w(h)]                      M = 128 rows, N = 128, K = 128 (Section 2.2)
//   scores   S   = Q_hi . V_t^T + Q_lo . V_t^T        M = 128 rows, N = 128 tokens, K = 2 x 128
//   output   O  += P . V_t                             M = 128 rows, N = 128 dims,  K = 128
//
// Each cached tile V_t [128 tokens x 128 dims] arrives once by TMA (one box per page) and feeds
// both products from the same shared-memory copy: as the K-major B operand of the score MMAs
// (bf16, as it landed) and, once the softmax warps have converted it to fp16 in place, as the
// MN-major B operand of the output MMAs. Everything else lives in TMEM (512 columns): 256 columns
// of scores, O (128), and the routed query Q_hi | Q_lo (64 + 64). Q and P enter the MMAs as A
// operands straight from TMEM, so the only operand the tensor cores read from shared memory is
// the cache tile.
//
// The pipeline's unit is a half tile u of 64 tokens: its scores go to one of four 64-column
// buffers as soon as the output MMAs of half tile u - 4 have read that buffer's weights, the
// softmax writes P over the buffer's first 32 columns, and the output MMAs follow. Two groups of
// four softmax warps take alternate half tiles, so a half tile's chain (scores, maximum,
// exponentials, weights, output, about 2600 cycles) is spread over four in flight. With whole
// tiles and two buffers that chain set the pace; so did the issuing threads, which are held until
// their MMAs start and then paid warp-wide waits before the next ones: each issuer's loop now
// runs in one elected lane. 32K-token prompt (12 heads) 3335 -> 3000 us, 512-token chunks on 8192
// (8 x 32 heads) 595 -> 543 us (whole tiles and half tiles timed in turn; single boxes give 2980 to
// 3140 us for the prompt); the issued MMAs, 1.5 times the useful ones, then run at 1.58 to 1.66
// PFLOP/s under the power cap, where cuBLAS sustains 1.73.
//
// Precision: the routed query (times scale * log2 e) is carried as a pair of bf16 operands,
// x = hi + lo, about 16 significant bits where one bf16 operand keeps 8; the softmax weights
// are one fp16 operand (11 bits) against the tile in fp16. A CPU replay of these roundings on
// the parity cases (peaked rows at the start of a prompt, scores of tens of units, 1 % outlier
// values x20) puts the worst error at 0.40 of |err| <= 2e-3 + 1e-2 |ref|; with one bf16 operand
// for the weights it is 1.0-2.5 times the bound, with one fp16 operand for the query 2-5 times.
// So each tile costs three 128 x 128 x 128 MMAs instead of the four of a pair on both sides.
// bf16 values convert to fp16 exactly from 2^-14 to 65280 (smaller ones round to fp16's
// subnormal grid, an absolute error below 2^-25); a cached value of magnitude 65536 or more has
// no finite fp16 form and makes the outputs of the rows whose tiles hold it non-finite. The
// epilogue raises KL_FLAG_RANGE for any non-finite output.
//
// Softmax (thread = query row = TMEM lane): scores arrive already scaled by scale * log2 e (the
// routed query is scaled before its bf16 rounding), so p = 2^(s - m). The reference maximum m of
// a row only moves when a half tile's maximum exceeds it by more than 7 (a factor 128): then the row's
// O in TMEM and its running sum l are rescaled; otherwise p may reach 2^7, well inside fp16 and
// fp32 range, and the final O / l is unchanged because O and l share the same reference. The first
// reference covers the first 128 tokens (two half tiles, one of each softmax group): the row's largest
// weight is then more often exactly 1 and free of rounding. (With the first 64 alone fp32 outputs
// were further off from 64 bits: rms 1.56e-4 instead of 1.49e-4 on rows of 200 tokens, 1.060e-4
// instead of 1.044e-4 on a 4096-token prompt.) A reference that moves within a tile sees only its half
// of the tile, so with the limit of 8 that suits whole tiles rows with outlier values were further
// off as well, 1.19e-4 against 1.12e-4 (100-token chunks on 200 to 2000 tokens); with 7 they are at
// 1.09e-4, for 1 to 2 % of the time of such inputs (4 x 512 rows on 4096 tokens 187 -> 191 us).
//
// Roles (352 threads, one CTA per SM):
//   warps 0-7  softmax and epilogue: warp w serves TMEM lane quarter w % 4 (its 32 query rows)
//              and the half tiles of parity w / 4; in the prologue and the epilogue warps w and
//              w + 4 split the 128 columns of the routed query and of O between them
//   warp 8     producer: TMA of W^R and the query block (ring position 0), then cache tiles
//   warp 9     routing and score MMA issuer (one elected lane) and TMEM owner
//   warp 10    output MMA issuer: a thread of its own, so that a half tile's output MMAs need
//              not queue behind the next scores
// Every wait is bounded (about one second); a wait that runs out raises KL_FLAG_TIMEOUT, makes
// every role leave its loop, drains outstanding copies and MMAs and frees TMEM.
#include <cudaTypedefs.h>
#include <math.h>

#include "kl_internal.cuh"
#include "kl_prefill_plan.cuh"
#include "kl_tc_ptx.cuh"

namespace kl {
namespace {

constexpr int kD = 128;
constexpr int kBM = kPrefillRows;                 // query rows per CTA
constexpr int kBN = kPrefillTile;                 // cache rows per tile
constexpr int kBS = 64;                           // cache rows per half tile
constexpr int kSub = 4;                           // half tiles in flight (score buffers)
constexpr int kStages = 5;
constexpr int kComputeWarps = 8;                  // two per TMEM lane quarter
constexpr int kProducerWarp = 8;
constexpr int kMmaWarp = 9;                       // routing and score MMAs; TMEM owner
constexpr int kPvWarp = 10;                       // output MMAs
constexpr int kThreads = 11 * 32;
constexpr uint32_t kTileBytes = kBN * kD * 2;     // 32 KiB
constexpr uint32_t kHalfBytes = kTileBytes / 2;   // one 64-column half: 128 rows x 128 B
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0;                     // S of half tile u: 64 (u % 4) .. + 63 (then
                                                  // its P, fp16 pairs, in the first 32); the
                                                  // routed query first lands in 0 .. 127
constexpr uint32_t kColO = 256;                   // O: columns 256 .. 383
constexpr uint32_t kColQ = 384;                   // Q_hi: 384 .. 447, Q_lo: 448 .. 511
constexpr uint32_t kLoCols = 64;                  // hi -> lo of a packed bf16 operand
constexpr float kRescaleLog2 = 7.f;
constexpr uint64_t kTimeoutNs = 1000000000ull;

struct __align__(1024) PrefillSmem {
    // The query block (A operand of the routing MMA); K-major, 128B-swizzled:
    // [64-dim half][128 rows][128 B].
    uint8_t q[kBM * kD * 2];
    // Ring of 32 KiB slots: W^R[w(h)] at position 0 ([64-column half][128 k rows][128 B]), then
    // the cache tiles ([64-dim half][128 tokens][128 B]); all 128B-swizzled.
    uint8_t tiles[kStages][kTileBytes];
    uint64_t full[kStages], empty[kStages];
    uint64_t s_full[kSub], s_free[kSub], p_full[kSub];
    uint64_t turn[4][2];       // per lane quarter and parity: the references after a half tile
    uint64_t first[4];         // per lane quarter: the maxima of half tile 1 are in lsum[1]
    uint64_t r_full, qr_ready, drain, drain2;
    float mref[2][kBM];        // the rows' references after the last half tile of each parity
    float lsum[2][kBM];        // the two groups' shares of the row sums, for the epilogue (before:
                               // [1] the maxima of half tile 1, for the first reference)
    float2 ml[kBM];            // the rows' references and sums, for the cluster's merge
    uint32_t tmem_base;
    int abort;
};

// Bounded wait. Warp-collective (every lane calls it in uniform control flow and gets the same
// answer), or by one lane alone (one(): the MMA issuers, whose successful waits must cost little).
// False when the CTA is aborting or the wait ran out (about 1 s).
struct Waiter {
    volatile int *abort;
    int32_t *err;
    __device__ bool slow(uint64_t *bar, uint32_t parity) const {
        const uint64_t t0 = ptx::globaltimer();
        while (true) {
            if (ptx::mbar_try_wait(bar, parity)) return true;
            if (*abort) return false;
            if (ptx::globaltimer() - t0 > kTimeoutNs) {
                *abort = 1;
                raise_flag(err, KL_FLAG_TIMEOUT);
                return false;
            }
        }
    }
    __device__ bool one(uint64_t *bar, uint32_t parity) const {
        return ptx::mbar_try_wait(bar, parity) || slow(bar, parity);
    }
    __device__ bool operator()(uint64_t *bar, uint32_t parity) const {
        return __all_sync(0xffffffffu, one(bar, parity));
    }
};

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// x = hi + lo with hi = bf16(x), lo = bf16(x - hi), for two values packed as bf16 pairs.
__device__ __forceinline__ void split2(float x0, float x1, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - hf.x, x1 - hf.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// Instruction descriptor of kind::f16 with fp16 A and B (A and B formats 0), fp32 accumulator,
// operand majorness (0 = K-major, 1 = MN-major), N and M.
__host__ __device__ constexpr uint32_t idesc_f16(uint32_t M, uint32_t N, bool a_mn, bool b_mn) {
    return (1u << 4) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((N >> 3) << 17) |
           ((M >> 4) << 24);
}

// max(a, b, c): the three-operand PTX max.
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Packed fp32 pair arithmetic (one instruction for two lanes of data).
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\t"
        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
        "add.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\t"
        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
        "sub.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float f) {
    return make_float2(a.x * f, a.y * f);
}

// Two values as an fp16 pair (a in the low half), round to nearest even.
__device__ __forceinline__ uint32_t pack_f16(float a, float b) {
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

__device__ __forceinline__ void ld_shared_v4(uint32_t addr, uint32_t *v) {
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c,
                                             uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
                 "r"(d)
                 : "memory");
}

// kShared: several heads per block or CTAs per cluster (a.hp, a.rpb, a.cs); otherwise one head per
// block and one CTA per block, as constants.
template <bool kShared>
__global__ void __launch_bounds__(kThreads, 1)
    prefill_tc_kernel(const __grid_constant__ CUtensorMap vmap,
                      const __grid_constant__ CUtensorMap wmap,
                      const __grid_constant__ CUtensorMap qmap, const PrefillArgs a) {
    extern __shared__ uint8_t smem_raw[];
    PrefillSmem &sm = *reinterpret_cast<PrefillSmem *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const Geometry &geo = a.geo;
    const int cs = kShared ? a.cs : 1, hp = kShared ? a.hp : 1, rpb = kShared ? a.rpb : kBM;
    const int rank = blockIdx.x % cs, hg = blockIdx.x / cs, b = blockIdx.y;
    const int mblk = (int)gridDim.z - 1 - (int)blockIdx.z;   // the longest blocks start first
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    grid_dep_wait();
    const int q0 = a.cu_q[b], q1 = a.cu_q[b + 1];
    const int L = a.seq_lens[b];
    const int n = q1 - q0;
    if (q0 < 0 || n < 0 || q1 > a.total_q || L < n || L > geo.max_pages * geo.P) {
        if (tid == 0 && blockIdx.x == 0 && mblk == 0) raise_flag(a.err, KL_FLAG_BAD_LENGTH);
        return;
    }
    // The block: query rows m0 .. m0 + rows - 1 of the chunk, heads h .. h + hn - 1; row r of the
    // 128 is query row r / hp of head r % hp.
    const int m0 = mblk * rpb;
    if (m0 >= n) return;
    const int rows = min(rpb, n - m0);
    const int nhg = (geo.G + hp - 1) / hp;       // blocks of heads per value head
    const int g = hg / nhg, h = g * geo.G + (hg % nhg) * hp;
    const int hn = min(hp, (g + 1) * geo.G - h);
    const int wsel = geo.wr_per_qh ? h : g;      // (one W^R per query head: hp is 1)
    const int pos0 = L - n + m0;                 // position of row 0
    const int pos_last = pos0 + rows - 1;        // <= L - 1
    // The cluster's CTAs take consecutive shares of the block's cache tiles; this one's are tiles
    // tile0 .. tile0 + n_tiles - 1, half tiles 0 .. n_sub - 1 from there (none for the last ranks
    // of a short sequence).
    const int all_tiles = pos_last / kBN + 1;
    const int share = (all_tiles + cs - 1) / cs;
    const int tile0 = min(all_tiles, rank * share);
    const int n_tiles = min(share, all_tiles - tile0);
    const int n_sub = max(0, min(2 * n_tiles, pos_last / kBS + 1 - 2 * tile0));

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            ptx::mbar_init(&sm.full[s], 1);
            ptx::mbar_init(&sm.empty[s], 1);
        }
        // One completion per half tile u of its buffer b = u % kSub on s_full[b] (its scores),
        // p_full[b] (its weights and the converted rows) and s_free[b] (its output MMAs are done:
        // O holds it, and the buffer may be written), and per lane quarter on turn[.][u % 2].
        // Every wait names the completion it needs: MMAs that write different TMEM ranges are
        // not assumed to complete in issue order.
        for (int b2 = 0; b2 < kSub; ++b2) {
            ptx::mbar_init(&sm.s_full[b2], 1);
            ptx::mbar_init(&sm.s_free[b2], 1);
            ptx::mbar_init(&sm.p_full[b2], kComputeWarps / 2);
        }
        for (int q = 0; q < 4; ++q) {
            for (int b2 = 0; b2 < 2; ++b2) ptx::mbar_init(&sm.turn[q][b2], 1);
            ptx::mbar_init(&sm.first[q], 1);
        }
        ptx::mbar_init(&sm.r_full, 1);
        ptx::mbar_init(&sm.qr_ready, kComputeWarps);
        ptx::mbar_init(&sm.drain, 1);
        ptx::mbar_init(&sm.drain2, 1);
        sm.abort = 0;
        ptx::fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        ptx::tmem_alloc(&sm.tmem_base, kTmemCols);
        ptx::tmem_relinquish();
    }
    // rows of the query block that its box does not fill
    if (kShared) {
        for (int i = tid; i < (kBM - hp * rpb) * 16; i += kThreads)
            *reinterpret_cast<uint4 *>(sm.q + (i & 8 ? kHalfBytes : 0) + (hp * rpb + (i >> 4)) * 128 +
                                       (i & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
        ptx::fence_proxy_async_smem();
    }
    if (warp == kProducerWarp && lane == 0) {
        ptx::prefetch_tensormap(&vmap);
        ptx::prefetch_tensormap(&wmap);
        ptx::prefetch_tensormap(&qmap);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    // (No early signal to the kernel behind: a chunk append that came to sit under the last wave
    // made batches of short sequences slower, 16 x 16 heads of 100 to 3000 tokens 203 -> 230 us.)

    const uint32_t tmem = sm.tmem_base;
    const Waiter wait{&sm.abort, a.err};

    const int qd = warp & 3, hf = warp >> 2;     // softmax warps: lane quarter and group
    const int r = qd * 32 + lane;                // query row = TMEM lane
    if (kShared && n_sub == 0) {
        // no share of the cache: an empty state
        if (warp < 4) sm.ml[r] = make_float2(-INFINITY, 0.f);
    } else if (warp == kProducerWarp) {
        // ------------------------------------------------------------------ producer ----
        const int P = geo.P;
        const int ppt = kBN / P;                          // pages per tile (<= 8)
        const int seq_pages = (L + P - 1) / P;
        const uint32_t page_bytes = (uint32_t)P * 128u;  // one half of one page
        const int32_t *bt = a.block_table + (size_t)b * geo.max_pages;
        int issued = 0;
        bool bad = false;
        // position 0: W^R[w(h)] (B operand of the routing MMA) and the query block
        if (lane == 0) {
            ptx::mbar_arrive_expect_tx(&sm.full[0], kTileBytes + hp * rpb * kD * 2);
            ptx::tma_load_2d(sm.tiles[0], &wmap, &sm.full[0], 0, wsel * kD);
            ptx::tma_load_2d(sm.tiles[0] + kHalfBytes, &wmap, &sm.full[0], 64, wsel * kD);
            ptx::tma_load_3d(sm.q, &qmap, &sm.full[0], 0, h, q0 + m0);
            ptx::tma_load_3d(sm.q + kHalfBytes, &qmap, &sm.full[0], 64, h, q0 + m0);
        }
        __syncwarp();
        issued = 1;
        for (int i = 0; i < n_tiles; ++i) {
            const int r = i + 1, s = r % kStages;
            const int pg = (tile0 + i) * ppt + lane;      // page index within the sequence
            const bool exists = lane < ppt && pg < seq_pages;
            const int page = exists ? bt[pg] : -1;
            if (r >= kStages && !wait(&sm.empty[s], ((r / kStages) & 1) ^ 1)) break;
            const bool in_range = exists && page >= 0 && page < geo.num_pages;
            if (exists && !in_range) bad = true;
            const unsigned mask = __ballot_sync(0xffffffffu, in_range);
            if (lane == 0) ptx::mbar_arrive_expect_tx(&sm.full[s], __popc(mask) * page_bytes * 2u);
            __syncwarp();
            if (in_range) {
                const int row = (page * geo.Hkv + g) * P;
                uint8_t *dst = sm.tiles[s] + lane * page_bytes;
                ptx::tma_load_2d(dst, &vmap, &sm.full[s], 0, row);
                ptx::tma_load_2d(dst + kHalfBytes, &vmap, &sm.full[s], 64, row);
            }
            issued = r + 1;
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) raise_flag(a.err, KL_FLAG_BAD_PAGE);
        if (sm.abort) {
            // copies still in flight land before the CTA's shared memory goes away
            for (int i = max(0, issued - kStages); i < issued; ++i) {
                const uint64_t t0 = ptx::globaltimer();
                while (!ptx::mbar_try_wait(&sm.full[i % kStages], (i / kStages) & 1) &&
                       ptx::globaltimer() - t0 < kTimeoutNs) {
                }
            }
        }
    } else if (warp == kMmaWarp || warp == kPvWarp) {
        // ---------------------------------------------------------------- MMA issuers ----
        // K-major SW128 operands step 32 B per 16 columns inside a 64-column half and jump a
        // half (kHalfBytes) every 4 steps; MN-major SW128 operands step 16 rows = 2 KiB; TMEM
        // A operands step 8 columns (16 packed 16-bit values).
        constexpr uint32_t idesc_qk = ptx::idesc_bf16(128, kBS, false, false);
        constexpr uint32_t idesc_route = ptx::idesc_bf16(128, 128, false, true);
        constexpr uint32_t idesc_pv = idesc_f16(128, 128, false, true);   // (mma_bf16_ts issues
        // the kind::f16 MMA; this descriptor makes both of its operands fp16)
        const uint64_t q_desc = ptx::smem_desc(ptx::smem_addr(sm.q), 16, 1024, ptx::kSwizzle128B);
        const uint64_t k_desc = ptx::smem_desc(ptx::smem_addr(sm.tiles[0]), 16, 1024, ptx::kSwizzle128B);
        const uint64_t mn_desc =
            ptx::smem_desc(ptx::smem_addr(sm.tiles[0]), kHalfBytes, 1024, ptx::kSwizzle128B);
        auto kstep = [](int kk) -> uint32_t { return ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4; };
        bool ok = true;
        if (warp == kMmaWarp) {
            // routing, then the score MMAs of every tile
            ok = wait(&sm.full[0], 0);
            if (ok) {
                ptx::tc_fence_after();
                if (ptx::elect_one()) {
                    // Q_r = Q . W^R: A = query block (K-major), B = W^R (N = output dim j,
                    // MN-major)
#pragma unroll
                    for (int kk = 0; kk < kD / 16; ++kk)
                        ptx::mma_bf16(tmem + kColS, q_desc + kstep(kk), mn_desc + ((kk * 2048) >> 4),
                                      idesc_route, kk > 0);
                    ptx::mma_commit(&sm.empty[0]);
                    ptx::mma_commit(&sm.r_full);
                }
                __syncwarp();
            }
            ok = ok && wait(&sm.qr_ready, 0);
            // (the whole loop by one lane: a warp-wide wait between two half tiles left the
            // tensor cores idle, since the issuing thread is held until its MMAs start)
            if (ok && ptx::elect_one()) {
                ptx::tc_fence_after();
                for (int u = 0; u < n_sub; ++u) {
                    const int r = (u >> 1) + 1, s = r % kStages, sb = u % kSub;
                    if (!wait.one(&sm.full[s], (r / kStages) & 1)) break;
                    // the output MMAs of half tile u - kSub have read buffer sb (its P)
                    if (u >= kSub && !wait.one(&sm.s_free[sb], (u / kSub - 1) & 1)) break;
                    ptx::tc_fence_after();
                    // S = Q_hi . V^T + Q_lo . V^T: A = Q_r in TMEM, B = 64 rows of the tile
                    // (N = tokens, K-major)
                    const uint64_t b0 = k_desc + ((s * kTileBytes + (u & 1) * kBS * 128) >> 4);
#pragma unroll
                    for (int kk = 0; kk < 2 * kD / 16; ++kk)
                        ptx::mma_bf16_ts(tmem + kColS + sb * kBS,
                                         tmem + kColQ + (kk >= 8 ? kLoCols : 0u) + (kk & 7) * 8,
                                         b0 + kstep(kk & 7), idesc_qk, kk > 0);
                    ptx::mma_commit(&sm.s_full[sb]);
                }
            }
        } else if (ptx::elect_one()) {
            // the output MMAs of every half tile: O += P . V, fp16; A = P in TMEM (the first 32
            // columns of its score buffer), B = 64 rows of the tile (N = dims, MN-major),
            // converted to fp16 by the softmax warps before they arrive on p_full
            for (int u = 0; u < n_sub; ++u) {
                const int s = ((u >> 1) + 1) % kStages, sb = u % kSub;
                if (!wait.one(&sm.p_full[sb], (u / kSub) & 1)) break;
                ptx::tc_fence_after();
                const uint64_t b0 = mn_desc + ((s * kTileBytes + (u & 1) * kBS * 128) >> 4);
                const uint32_t pa = tmem + kColS + sb * kBS;
#pragma unroll
                for (int kk = 0; kk < kBS / 16; ++kk)
                    ptx::mma_bf16_ts(tmem + kColO, pa + kk * 8, b0 + ((kk * 2048) >> 4), idesc_pv,
                                     (u > 0 || kk > 0) ? 1u : 0u);
                ptx::mma_commit(&sm.s_free[sb]);
                if ((u & 1) || u == n_sub - 1) ptx::mma_commit(&sm.empty[s]);
            }
        }
        __syncwarp();
        // every MMA this warp issued completes before TMEM is freed
        uint64_t *drain = warp == kMmaWarp ? &sm.drain : &sm.drain2;
        if (ptx::elect_one()) ptx::mma_commit(drain);
        __syncwarp();
        const uint64_t t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(drain, 0) && ptx::globaltimer() - t0 < kTimeoutNs) {
        }
    } else {
        // --------------------------------------------------------- softmax, epilogue ----
        // Two groups of four warps: warp w serves the 32 query rows of lane quarter w % 4
        // (thread = row = TMEM lane), group w / 4 the half tiles of that parity, so that one
        // group's softmax runs while the tensor cores and the other group work on the half tiles
        // around it. The groups share each row's reference (and O): the owner of half tile u takes
        // the reference that u - 1 left, and passes its own on (turn) before its exponentials. In
        // the prologue and the epilogue the two warps of a lane quarter split the 128 columns.
        const int c0 = hf * 64;                              // this warp's columns
        const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
        const uint32_t pair_bar = 1 + qd;
        // rows past the block's end take the last valid position: finite, never stored
        const int pos_r = min(pos0 + r / hp, pos_last);
        const float sl2 = geo.scale * kLog2e;
        bool ok = wait(&sm.r_full, 0);

        // Routed query row, this warp's 64 columns: Q_r * scale * log2 e as hi + lo bf16 pairs
        // into the Q columns (32 packed columns each).
        if (ok) {
            ptx::tc_fence_after();
            uint32_t u0[32], u1[32];
            ptx::tmem_ld32(tmem + kColS + c0 + lane_base, u0);
            ptx::tmem_ld32(tmem + kColS + c0 + 32 + lane_base, u1);
            ptx::tmem_wait_ld();
            ptx::reg_fence(u0);
            ptx::reg_fence(u1);
            uint32_t hi[32], lo[32];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                split2(__uint_as_float(u0[2 * e]) * sl2, __uint_as_float(u0[2 * e + 1]) * sl2,
                       hi[e], lo[e]);
                split2(__uint_as_float(u1[2 * e]) * sl2, __uint_as_float(u1[2 * e + 1]) * sl2,
                       hi[16 + e], lo[16 + e]);
            }
            ptx::tmem_st32(tmem + kColQ + c0 / 2 + lane_base, hi);
            ptx::tmem_st32(tmem + kColQ + kLoCols + c0 / 2 + lane_base, lo);
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm.qr_ready);
        }

        float m_used = -INFINITY;  // the reference of this thread's share of the row sum
        // this group's share of sum 2^(s - m_used), in two packed pairs of partial sums
        float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
        bool okl = ok;
        for (int u = hf; okl && u < n_sub; u += 2) {
            const int t0 = tile0 * kBN + u * kBS, k = u >> 1, sb = u % kSub;
            const uint32_t sbuf = tmem + kColS + (uint32_t)sb * kBS + lane_base;   // S, then P
            // This thread's half (64 dims) of a cache row of the half tile as fp16, formed while
            // the scores are still on their way: the output MMAs read the tile as fp16. Rows at
            // or past the sequence's end (an unwritten page tail, or a page slot no TMA filled)
            // become zeros, so that 0-weights never meet a non-finite value. The lanes start at
            // different 16-byte chunks so that a warp's accesses spread over all banks.
            const int stage = (k + 1) % kStages;
            okl = wait(&sm.full[stage], ((k + 1) / kStages) & 1);
            if (!okl) break;
            const uint32_t v_s = ptx::smem_addr(sm.tiles[stage]) + (r >> 6) * kHalfBytes +
                                 (hf * kBS + (r & 63)) * 128;
            uint32_t vr[32];
            if (t0 + (r & 63) < L) {
#pragma unroll
                for (int c = 0; c < 8; ++c) ld_shared_v4(v_s + ((c + lane) & 7) * 16, vr + 4 * c);
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    vr[e] = pack_f16(__uint_as_float(vr[e] << 16), __uint_as_float(vr[e] & 0xffff0000u));
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) vr[e] = 0u;
            }
            okl = wait(&sm.s_full[sb], (u / kSub) & 1);
            if (!okl) break;
            ptx::tc_fence_after();
            uint32_t s0[32], s1[32];
            ptx::tmem_ld32(sbuf, s0);
            ptx::tmem_ld32(sbuf + 32, s1);
            // the score MMAs have read these rows: their fp16 form takes their place
#pragma unroll
            for (int c = 0; c < 8; ++c)
                st_shared_v4(v_s + ((c + lane) & 7) * 16, vr[4 * c], vr[4 * c + 1], vr[4 * c + 2],
                             vr[4 * c + 3]);
            ptx::tmem_wait_ld();
            ptx::reg_fence(s0);
            ptx::reg_fence(s1);
            // causal mask: token t0 + c is visible to the row when it is <= pos_r
            if (t0 + kBS - 1 > pos0) {
                const int lim = pos_r - t0;
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    if (c > lim) s0[c] = 0xff800000u;
                    if (c + 32 > lim) s1[c] = 0xff800000u;
                }
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                mx[0] = max3(mx[0], __uint_as_float(s0[c]), __uint_as_float(s0[c + 1]));
                mx[1] = max3(mx[1], __uint_as_float(s0[c + 2]), __uint_as_float(s0[c + 3]));
                mx[2] = max3(mx[2], __uint_as_float(s1[c]), __uint_as_float(s1[c + 1]));
                mx[3] = max3(mx[3], __uint_as_float(s1[c + 2]), __uint_as_float(s1[c + 3]));
            }
            float mt = max3(mx[0], mx[1], fmaxf(mx[2], mx[3]));
            float m_ref = -INFINITY;
            if (u == 0) {
                // the row's first reference is the maximum of its first two half tiles
                if (n_sub > 1) {
                    okl = wait(&sm.first[qd], 0);
                    if (!okl) break;
                    mt = fmaxf(mt, sm.lsum[1][r]);
                }
            } else {
                if (u == 1) {
                    sm.lsum[1][r] = mt;
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&sm.first[qd]);
                }
                okl = wait(&sm.turn[qd][hf ^ 1], ((u - 1) >> 1) & 1);
                if (!okl) break;
                m_ref = sm.mref[hf ^ 1][r];
            }
            // a new reference when the maximum grew by more than 2^7 (or is the first finite)
            const float m_new = fmaxf(m_ref, mt);
            if (__any_sync(0xffffffffu, m_new > m_ref + kRescaleLog2)) {
                const float f = (m_new == -INFINITY || m_ref == -INFINITY) ? 0.f : ptx::ex2(m_ref - m_new);
                if (u > 0) {
                    // O holds half tiles 0 .. u - 1 once the output MMAs of u - 1 are done
                    okl = wait(&sm.s_free[(u - 1) % kSub], ((u - 1) / kSub) & 1);
                    if (!okl) break;
                    ptx::tc_fence_after();
#pragma unroll
                    for (int c = 0; c < 128; c += 32) {
                        uint32_t o[32];
                        ptx::tmem_ld32(tmem + kColO + c + lane_base, o);
                        ptx::tmem_wait_ld();
                        ptx::reg_fence(o);
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * f);
                        ptx::tmem_st32(tmem + kColO + c + lane_base, o);
                    }
                    ptx::tmem_wait_st();
                }
                m_ref = m_new;
            }
            sm.mref[hf][r] = m_ref;
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm.turn[qd][hf]);
            // the group's sums move to this reference
            if (__any_sync(0xffffffffu, m_ref != m_used)) {
                const float f = m_used == -INFINITY ? 0.f : ptx::ex2(m_used - m_ref);
                la = mul2(la, f);
                lb = mul2(lb, f);
                m_used = m_ref;
            }
            // the row's 64 weights -> 32 packed fp16 columns of P (in pairs: s - m, 2^x, the
            // running sums, the fp16 pack)
            const float mr = m_ref == -INFINITY ? 0.f : m_ref;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float2 d = sub2(make_float2(__uint_as_float(s0[2 * e]), __uint_as_float(s0[2 * e + 1])),
                                      make_float2(mr, mr));
                const float2 pe = make_float2(ptx::ex2(d.x), ptx::ex2(d.y));
                if (e & 1) lb = add2(lb, pe); else la = add2(la, pe);
                s0[e] = pack_f16(pe.x, pe.y);
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float2 d = sub2(make_float2(__uint_as_float(s1[2 * e]), __uint_as_float(s1[2 * e + 1])),
                                      make_float2(mr, mr));
                const float2 pe = make_float2(ptx::ex2(d.x), ptx::ex2(d.y));
                if (e & 1) lb = add2(lb, pe); else la = add2(la, pe);
                s0[16 + e] = pack_f16(pe.x, pe.y);
            }
            // P over the first 32 columns of the buffer (the output MMAs of u - kSub, the last
            // reader of P there, finished before these scores were written)
            ptx::tmem_st32(sbuf, s0);
            ptx::tmem_wait_st();
            // the converted rows (generic-proxy stores) are read next by the output MMAs
            ptx::tc_fence_before();
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm.p_full[sb]);
        }

        // Epilogue: out = O / l, this warp's 64 output dims; l is the two groups' shares, at the
        // reference of the last half tile. A non-finite output (a cached value beyond fp16's range,
        // or a non-finite input) raises KL_FLAG_RANGE.
        const int last = n_sub - 1, lb2 = last & 1;
        if (okl && lb2 != hf) okl = wait(&sm.turn[qd][lb2], (last >> 1) & 1);
        const bool oke = okl && wait(&sm.s_free[last % kSub], (last / kSub) & 1);
        float l = (la.x + la.y) + (lb.x + lb.y);
        if (oke && lb2 != hf) {
            const float m_fin = sm.mref[lb2][r];
            l = m_used == -INFINITY ? 0.f : l * ptx::ex2(m_used - m_fin);
        }
        sm.lsum[hf][r] = l;
        const bool okp = ptx::bar_and(pair_bar, 64, oke);
        const float lt = l + sm.lsum[hf ^ 1][r];
        if (kShared && cs > 1) {
            if (hf == 0) sm.ml[r] = okp ? make_float2(sm.mref[lb2][r], lt) : make_float2(-INFINITY, 0.f);
        } else if (okp) {
            ptx::tc_fence_after();
            const float inv = lt > 0.f ? 1.f / lt : 0.f;
            float nf = 0.f;   // x * 0 is NaN exactly when x is not finite
            const int ri = r / hp, hh = r - ri * hp;
            const size_t orow = ((size_t)(q0 + m0 + ri) * geo.Hq + h + hh) * kD + c0;
#pragma unroll
            for (int c4 = 0; c4 < 2; ++c4) {
                uint32_t u[32];
                ptx::tmem_ld32(tmem + kColO + c0 + c4 * 32 + lane_base, u);
                ptx::tmem_wait_ld();
                ptx::reg_fence(u);
                if (ri < rows && hh < hn) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) nf = fmaf(__uint_as_float(u[e]), 0.f, nf);
                    if (a.out_dtype == KL_FP32) {
                        float4 *o = reinterpret_cast<float4 *>(static_cast<float *>(a.out) + orow + c4 * 32);
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            o[c] = make_float4(__uint_as_float(u[4 * c]) * inv, __uint_as_float(u[4 * c + 1]) * inv,
                                               __uint_as_float(u[4 * c + 2]) * inv, __uint_as_float(u[4 * c + 3]) * inv);
                    } else {
                        uint4 *o = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(a.out) + orow + c4 * 32);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            uint32_t w[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                w[e] = pack2(__uint_as_float(u[8 * c + 2 * e]) * inv,
                                             __uint_as_float(u[8 * c + 2 * e + 1]) * inv);
                            o[c] = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
            }
            if (__any_sync(0xffffffffu, nf != nf) && lane == 0) raise_flag(a.err, KL_FLAG_RANGE);
        }
    }

    if (kShared && cs > 1) {
        // Merge of the cluster's states (m, l, O) as kl_combine does: every CTA scales its O to the
        // cluster's maximum and sum and puts it into its idle ring; then CTA k adds up rows
        // 128 k / cs .. of all of them. Every thread takes part in every cluster barrier.
        constexpr uint32_t kXRow = kD * 4 + 16;   // bytes of a row in the ring
        const uint32_t xch = ptx::smem_addr(sm.tiles[0]);
        ptx::cluster_sync();
        if (warp < kComputeWarps) {
            const uint32_t mla = ptx::smem_addr(&sm.ml[r]);
            float2 v[8];
            float M = -INFINITY;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k < cs) {
                    v[k] = ptx::ld_cluster_v2(ptx::cluster_addr(mla, k));
                    if (v[k].y > 0.f) M = fmaxf(M, v[k].x);
                }
            }
            float z = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < cs && v[k].y > 0.f) z += v[k].y * ptx::ex2(v[k].x - M);
            const float2 own = sm.ml[r];
            // an empty state adds zeros; a NaN sum makes NaN outputs, as in an undivided block
            const bool none = n_sub == 0 || own.y == 0.f;
            const float w = own.y > 0.f ? ptx::ex2(own.x - M) / z : own.y;
            const int c0 = hf * 64;
#pragma unroll
            for (int c4 = 0; c4 < 2; ++c4) {
                uint32_t u[32];
                if (n_sub > 0) {
                    ptx::tc_fence_after();
                    ptx::tmem_ld32(tmem + kColO + c0 + c4 * 32 + ((uint32_t)(qd * 32) << 16), u);
                    ptx::tmem_wait_ld();
                    ptx::reg_fence(u);
                }
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    u[e] = none ? 0u : __float_as_uint(__uint_as_float(u[e]) * w);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    st_shared_v4(xch + r * kXRow + (c0 + c4 * 32 + 4 * c) * 4, u[4 * c], u[4 * c + 1],
                                 u[4 * c + 2], u[4 * c + 3]);
            }
        }
        ptx::cluster_sync();
        if (warp < kComputeWarps) {
            // one warp per row, 4 dims per lane
            const int per = kBM / cs;
            float nf = 0.f;
            for (int i = warp; i < per; i += kComputeWarps) {
                const int row = rank * per + i, ri = row / hp, hh = row - ri * hp;
                if (ri >= rows || hh >= hn) continue;
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (k < cs) {
                        const float4 x = ptx::ld_cluster_v4(ptx::cluster_addr(xch + row * kXRow + lane * 16, k));
                        o.x += x.x;
                        o.y += x.y;
                        o.z += x.z;
                        o.w += x.w;
                    }
                }
                nf = fmaf(o.x, 0.f, fmaf(o.y, 0.f, fmaf(o.z, 0.f, fmaf(o.w, 0.f, nf))));
                const size_t oi = ((size_t)(q0 + m0 + ri) * geo.Hq + h + hh) * kD + 4 * lane;
                if (a.out_dtype == KL_FP32)
                    *reinterpret_cast<float4 *>(static_cast<float *>(a.out) + oi) = o;
                else
                    *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(a.out) + oi) =
                        make_uint2(pack2(o.x, o.y), pack2(o.z, o.w));
            }
            if (__any_sync(0xffffffffu, nf != nf) && lane == 0) raise_flag(a.err, KL_FLAG_RANGE);
        }
        ptx::cluster_sync();      // no CTA leaves while another reads its ring
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
}

// Chunk append: row i of sequence b's chunk goes to position seq_lens[b] - n_b + i. One CTA per
// (16 chunk rows, sequence); 16-byte copies.
constexpr int kAppendRows = 16;

__global__ void __launch_bounds__(128) append_chunk_kernel(int Hkv, int D, int P, int num_pages,
                                                           int max_pages, int total_q,
                                                           const uint4 *v_new,
                                                           const int32_t *block_table,
                                                           const int32_t *seq_lens,
                                                           const int32_t *cu_q,
                                                           uint4 *v_cache, int32_t *err) {
    grid_dep_wait();
    grid_dep_launch();
    const int b = blockIdx.y;
    const int q0 = cu_q[b], n = cu_q[b + 1] - q0, L = seq_lens[b];
    if (q0 < 0 || n < 0 || q0 + n > total_q || L < n || L > max_pages * P) {
        if (threadIdx.x == 0 && blockIdx.x == 0) raise_flag(err, KL_FLAG_BAD_LENGTH);
        return;
    }
    const int i0 = blockIdx.x * kAppendRows;
    const int cpr = D / 8;   // 16-byte chunks per row
    const int per_row = Hkv * cpr;
    for (int k = threadIdx.x; k < kAppendRows * per_row; k += blockDim.x) {
        const int i = i0 + k / per_row;
        if (i >= n) break;
        const int gc = k % per_row, g = gc / cpr, c = gc % cpr;
        const int pos = L - n + i;
        const int page = block_table[(size_t)b * max_pages + pos / P];
        if (page < 0 || page >= num_pages) {
            raise_flag(err, KL_FLAG_BAD_PAGE);
            continue;
        }
        v_cache[(((size_t)page * Hkv + g) * P + pos % P) * cpr + c] =
            v_new[((size_t)(q0 + i) * Hkv + g) * cpr + c];
    }
}

// ------------------------------------------------------------------------ host side ------

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// bf16 tensor map of `rank` dimensions, innermost 128 elements (256-byte rows), box 64 x ...,
// 128-byte swizzle.
bool encode(CUtensorMap *map, const void *base, int rank, const cuuint64_t *dims,
            const cuuint64_t *strides, const cuuint32_t *box) {
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void *>(base), dims, strides,
              box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool prefill_tc_supported(const Geometry &g) {
    if (g.D != kD) return false;
    if (g.P != 16 && g.P != 32 && g.P != 64 && g.P != 128) return false;
    if ((int64_t)g.num_pages * g.Hkv * g.P >= ((int64_t)1 << 31)) return false;
    int dev = 0, major = 0, minor = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
    return major == 10 && minor == 3;
}

cudaError_t launch_prefill_tc(const PrefillArgs &a) {
    const Geometry &g = a.geo;
    if (g.B == 0 || a.total_q == 0 || a.max_q == 0) return cudaSuccess;
    PrefillArgs la = a;
    const PrefillPlan plan = plan_prefill(g.B, g.Hkv, g.G, a.max_q, (int64_t)g.max_pages * g.P,
                                          g.wr_per_qh != 0, device_sm_count());
    la.hp = plan.hp;
    la.rpb = plan.rpb;
    la.cs = plan.cs;
    CUtensorMap vmap, wmap, qmap;
    {
        // cache as [num_pages * Hkv * P rows][128], one box = one page of one head (64 dims)
        const cuuint64_t dims[2] = {kD, (cuuint64_t)g.num_pages * g.Hkv * g.P};
        const cuuint64_t strides[1] = {kD * 2};
        const cuuint32_t box[2] = {64, (cuuint32_t)g.P};
        if (!encode(&vmap, a.v_cache, 2, dims, strides, box)) return cudaErrorInvalidValue;
    }
    {
        // W^R as [Hw * 128 k rows][128 j], one box = a 64-column half of one matrix
        const cuuint64_t hw = g.wr_per_qh ? (cuuint64_t)g.Hq : (cuuint64_t)g.Hkv;
        const cuuint64_t dims[2] = {kD, hw * kD};
        const cuuint64_t strides[1] = {kD * 2};
        const cuuint32_t box[2] = {64, kD};
        if (!encode(&wmap, a.w_r, 2, dims, strides, box)) return cudaErrorInvalidValue;
    }
    {
        // q as [total_q][Hq][128], one box = rpb consecutive rows of hp heads (64 dims); rows past
        // total_q and heads past Hq read as zeros
        const cuuint64_t dims[3] = {kD, (cuuint64_t)g.Hq, (cuuint64_t)a.total_q};
        const cuuint64_t strides[2] = {kD * 2, (cuuint64_t)g.Hq * kD * 2};
        const cuuint32_t box[3] = {64, (cuuint32_t)la.hp, (cuuint32_t)la.rpb};
        if (!encode(&qmap, a.q, 3, dims, strides, box)) return cudaErrorInvalidValue;
    }
    const size_t smem = sizeof(PrefillSmem) + 1024;
    while (true) {
        const bool shared = la.hp > 1 || la.cs > 1;
        const auto kernel = shared ? prefill_tc_kernel<true> : prefill_tc_kernel<false>;
        static PerDeviceOnce once[2];
        cudaError_t e = once[shared].run([&] {
            return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        });
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(la.cs * g.Hkv * ((g.G + la.hp - 1) / la.hp), g.B, (a.max_q + la.rpb - 1) / la.rpb);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = a.stream;
        cudaLaunchAttribute attr[2];
        attr[0] = OverlapAttr(cfg).attr[0];
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)la.cs;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = la.cs > 1 ? 2 : 1;
        e = cudaLaunchKernelEx(&cfg, kernel, vmap, wmap, qmap, la);
        if (e == cudaSuccess || la.cs == 1) return e;
        // a context that may not use enough SMs of one GPC for the cluster: one CTA per block
        (void)cudaGetLastError();
        la.cs = 1;
    }
}

cudaError_t launch_append_chunk(const Geometry &g, int total_q, int max_q, const uint16_t *v_new,
                                const int32_t *block_table, const int32_t *seq_lens,
                                const int32_t *cu_q, uint16_t *v_cache, int32_t *err,
                                cudaStream_t stream) {
    if (g.B == 0 || total_q == 0 || max_q == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((max_q + kAppendRows - 1) / kAppendRows, g.B);
    cfg.blockDim = dim3(128);
    cfg.stream = stream;
    const OverlapAttr overlap(cfg);
    return cudaLaunchKernelEx(&cfg, append_chunk_kernel, g.Hkv, g.D, g.P, g.num_pages, g.max_pages,
                              total_q, reinterpret_cast<const uint4 *>(v_new), block_table, seq_lens,
                              cu_q, reinterpret_cast<uint4 *>(v_cache), err);
}

}  // namespace kl
