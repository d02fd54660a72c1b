// Tensor-core decode for groups of more than 8 query heads: one CTA per SM serves up to NH = 16
// or 32 heads of a group from one shared-memory copy of each cache tile.
//
// The products are those of kl_decode_tc_kernel.cuh (S^T = V [q_hi | q_lo]^T, O^T = V^T [p_hi |
// p_lo]) with N = 2 NH columns. What a tile costs the tensor core hardly depends on N: measured,
// a 128 x N x 16 MMA with both operands in shared memory takes 39 / 40 / 48 cycles at N = 16 /
// 32 / 64, so 32 heads cost one CTA 770 cycles per tile where four sibling CTAs of 8 heads spend
// 2500, against the 1460 cycles in which HBM delivers a tile to each SM.
//
// Two layouts (NG softmax groups of 8 compute warps per CTA):
//  NG = 2, one CTA per SM with a ring of 5 or 6 tiles: group 0 takes the even tiles and group 1
//    the odd ones, so that the tile chain (scores, softmax, weights) overlaps itself. Each group
//    keeps its own softmax state (reference, sums and an O accumulator in TMEM), so the groups
//    meet only at the end, where their two states are merged like two splits.
//  NG = 1, two CTAs per SM with a ring of 3 tiles, 16 heads: for launches of several waves, whose
//    start-ups and last wave then overlap and share HBM.
// After each tile the group adds the MMAs' O to its sum (fp32 columns in TMEM, rounded to nearest by
// the compute warps) and the next tile's MMAs start over, as the sibling CTAs do it: the tensor core's
// adds truncate. (fp32 outputs against 64 bits, 32 sequences of 300 to 8000 tokens, 128/8 heads:
// 2.65e-6, siblings 2.64e-6; with the MMAs adding up 4 tiles of a group 2.70e-6, a whole run 4.8e-6
// at 8192 tokens. Folding every tile instead of every fourth costs 1 to 3 %: 256 sequences of 32/1
// heads 105.3 -> 106.9 us, 64 of 1000 to 60000 tokens 173.5 -> 178.7.) The rare tile that moves a
// reference rescales both.
//
// Warps: group i = warps 8 i .. 8 i + 7: warp w of a group reads TMEM lane quarter w % 4 (thread =
// token of S and P, output dim of O) and takes the KH = NH / 2 heads KH (w / 4) ..; then the
// producer, the score-MMA issuer (TMEM owner) and the output-MMA issuer.
//
// Measured (back-to-back calls, 8192 tokens): 64 sequences of 128 heads over 8 value heads 252 us
// with sibling CTAs of 8 heads, 184 with NG = 2, 164 to 168 with NG = 1 (HBM floor 158); 256 sequences
// of 32 heads over one value head 248 us with siblings, 133 with NG = 1 (two CTAs per tile, bound by
// the ring's round trip), 107 with NH = 32 and NG = 2 (floor 80; the rest is the last, partly
// filled wave). One sequence of 100000 tokens, 128 / 8 heads: 49.0 us with NG = 1, 40.6 with
// NG = 2. Spills cost much, since the shared memory leaves next to no L1: 48 bytes more per thread
// and tile took the second case from 121 to 158 us, so the references live in shared memory and
// the weights are formed 8 heads at a time.
//
// Each wait is bounded as in kl_decode_tc_kernel.cuh.
#include "kl_decode_tc_kernel.cuh"

namespace kl {
namespace {

constexpr int kWideGroupThreads = 256;               // 8 compute warps per softmax group
constexpr uint32_t kBarGroup = 3;                    // + group: vote of one group's warps
constexpr int kWideMaxRuns = 256;                    // states merged per (b, g, head block)
// A reference moves when a weight 2^(s - m) passes this. Sums, O and the split-bf16 weights are
// floating point with fp32's exponent range, so the bound only keeps everything far from overflow. (Of
// the precision a stale reference costs only the chance that the largest weight is exactly 1: with a
// slack of 4 the fp32 error was 0.3 % smaller on two of nine inputs, the same on the others, and 64
// sequences of 1000 to 60000 tokens with outliers took 231 instead of 180 us.)
constexpr float kWideLazy = 1024.f;

// Warp roles and sizes for NH heads per CTA and NG softmax groups: NG = 2, one CTA per SM; NG = 1,
// two CTAs per SM.
template <int NH, int NG>
struct Wide {
    static constexpr int kStages = NG == 1 ? 3 : NH == 32 ? 5 : 6;
    static constexpr int kWarps = 8 * NG;                // compute warps
    static constexpr int kProducer = kWarps, kMma = kWarps + 1, kPv = kWarps + 2;
    static constexpr int kThreads = (kWarps + 3) * 32;
    static constexpr int kCtas = NG == 1 ? 2 : 1;        // per SM
    static constexpr uint32_t kTmemCols = 512 / kCtas;
};

template <int NH, int NG>
struct __align__(1024) WideSmem {
    static constexpr int kStages = Wide<NH, NG>::kStages;
    uint8_t tiles[kStages][kTileBytes];              // as Smem<false>::tiles
    uint8_t qr[2 * 2 * NH * 128];                    // routed query [half][hi | lo rows][128 B]
    uint8_t p[NG][kTile * 2 * NH * 2];               // per group: [16 groups of 8 tokens]
                                                     // [2 NH / 8 blocks][8 tokens][16 B]
    float red[NG][4][NH];                            // per group and lane quarter: maxima
    float lred[NG][4][NH];                           // ... row sums
    float mref[NG][NH];                              // per group: the heads' references (in
                                                     // shared memory to save registers)
    uint64_t full[kStages], empty[kStages];
    uint64_t s_full[2 * NG], s_empty[2 * NG], p_full[NG], o_full[NG];
    uint64_t qr_full, r_full, drain, drain2, merge_full;
    int is_last;
    uint32_t tmem_base;
    int abort;
};
// (228 KB per SM, of which each CTA takes 1 KB for the system)
static_assert(sizeof(WideSmem<16, 1>) <= 228 * 1024 / 2 - 1024, "two CTAs per SM");
static_assert(sizeof(WideSmem<32, 2>) <= 227 * 1024 && sizeof(WideSmem<16, 2>) <= 227 * 1024, "one");

// 8 consecutive columns at `a` and at `b` of the thread's TMEM lane, one wait.
__device__ __forceinline__ void tmem_ld_cols8(uint32_t a, uint32_t b, float (&x)[8], float (&y)[8]) {
    uint32_t u[8], v[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]),
          "=r"(u[7]), "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
          "=r"(v[6]), "=r"(v[7])
        : "r"(a), "r"(b)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        x[i] = __uint_as_float(u[i]);
        y[i] = __uint_as_float(v[i]);
    }
}

// 8 consecutive columns of the thread's TMEM lane (load and wait in one statement).
__device__ __forceinline__ void tmem_ld_col8(uint32_t a, float (&x)[8]) {
    uint32_t u[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]),
          "=r"(u[7])
        : "r"(a)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = __uint_as_float(u[i]);
}

// 8 consecutive columns of the thread's TMEM lane (complete with tmem_wait_st()).
__device__ __forceinline__ void tmem_st_cols8(uint32_t a, const float (&x)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(a),
                 "r"(__float_as_uint(x[0])), "r"(__float_as_uint(x[1])), "r"(__float_as_uint(x[2])),
                 "r"(__float_as_uint(x[3])), "r"(__float_as_uint(x[4])), "r"(__float_as_uint(x[5])),
                 "r"(__float_as_uint(x[6])), "r"(__float_as_uint(x[7]))
                 : "memory");
}

// Packed fp32 pairs: one instruction, each lane the scalar round-to-nearest operation.
struct F2 {
    float x, y;
};
__device__ __forceinline__ F2 f2(float a, float b) { return F2{a, b}; }
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
        "add.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
    F2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
        "sub.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
// max(a, b, c): the three-operand PTX max.
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Warp maximum through the integer reduction unit (the key of a float orders as the float does).
__device__ __forceinline__ float warp_max_redux(float f) {
    const int i = __float_as_int(f);
    const int k = __reduce_max_sync(0xffffffffu, i >= 0 ? i : i ^ 0x7FFFFFFF);
    return __int_as_float(k >= 0 ? k : k ^ 0x7FFFFFFF);
}

template <int NH, int NG, bool kExact>
__global__ void __launch_bounds__(Wide<NH, NG>::kThreads, Wide<NH, NG>::kCtas)
    decode_wide_kernel(const __grid_constant__ CUtensorMap vmap,
                       const __grid_constant__ CUtensorMap wmap,
                       const __grid_constant__ CUtensorMap qmap, const DecodeArgs a) {
    using S = WideSmem<NH, NG>;
    using W = Wide<NH, NG>;
    constexpr int NS = W::kStages, kWideWarps = W::kWarps, kWideComputeThreads = 32 * W::kWarps;
    constexpr int kWideProducer = W::kProducer, kWideMma = W::kMma, kWidePv = W::kPv;
    constexpr uint32_t kWideTmemCols = W::kTmemCols;
    constexpr int KH = NH / 2;                           // heads per compute warp
    constexpr int N = 2 * NH;                            // MMA columns: hi | lo
    constexpr uint32_t kQHalf = N * 128;                 // one 64-dim half of the query operand
    constexpr uint32_t kGroupBytes = N / 8 * 128;        // P: one group of 8 tokens
    // TMEM columns: two S buffers and the O of a tile of each group, N each; then each group's summed
    // O, NH each
    constexpr uint32_t kColS = 0, kColO = 2 * NG * N, kColF = 3 * NG * N;
    static_assert(kColF + NG * NH <= kWideTmemCols, "");
    // (aligned by declaration: with two CTAs per SM there is no room for slack)
    extern __shared__ __align__(1024) uint8_t smem_wide[];
    S &sm = *reinterpret_cast<S *>(smem_wide);

    const Geometry &geo = a.geo;
    const int hb = blockIdx.x % geo.nhb, cta = blockIdx.x / geo.nhb;
    const int g = blockIdx.y, b = blockIdx.z;
    const int split0 = cta * geo.spc;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int G = min(NH, geo.G - NH * hb);              // query heads of this CTA
    const int qh0 = g * geo.G + NH * hb;                 // its first query head
    const bool route = a.w_r != nullptr;                 // else q is the composed query
    const bool route_pq = route && geo.wr_per_qh;
    const int ro = !route ? 0 : route_pq ? G : 1;        // ring positions of W^R matrices

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            ptx::mbar_init(&sm.full[s], 1);
            ptx::mbar_init(&sm.empty[s], 1);
        }
        for (int i = 0; i < 2 * NG; ++i) {
            ptx::mbar_init(&sm.s_full[i], 1);
            ptx::mbar_init(&sm.s_empty[i], 8);
        }
        for (int i = 0; i < NG; ++i) {
            ptx::mbar_init(&sm.p_full[i], 8);
            ptx::mbar_init(&sm.o_full[i], 1);
        }
        ptx::mbar_init(&sm.qr_full, kWideWarps);
        ptx::mbar_init(&sm.r_full, 1);
        ptx::mbar_init(&sm.merge_full, 1);
        ptx::mbar_init(&sm.drain, 1);
        ptx::mbar_init(&sm.drain2, 1);
        sm.abort = 0;
        ptx::fence_mbar_init();
    }
    if (tid < NG * NH) (&sm.mref[0][0])[tid] = -INFINITY;
    if (warp == kWideMma) {
        ptx::tmem_alloc(&sm.tmem_base, kWideTmemCols);
        ptx::tmem_relinquish();
    }
    if (warp == kWideProducer && lane == 0) {
        ptx::prefetch_tensormap(&vmap);
        if (route) {
            ptx::prefetch_tensormap(&wmap);
            ptx::prefetch_tensormap(&qmap);
        }
    }
    grid_dep_wait();        // nothing above touched global memory
    const int L_raw = a.seq_lens[b];
    const int pos_raw = a.v_new ? a.positions[b] : -1;
    const int t_begin = split0 * geo.chunk;
    const int first_page = t_begin / geo.P;
    const int32_t *bt = a.block_table + (size_t)b * geo.max_pages;
    int bt_cur = -1, bt_nxt = -1;
    if (warp == kWideProducer) {
        if (first_page + lane < geo.max_pages) bt_cur = bt[first_page + lane];
        if (first_page + 32 + lane < geo.max_pages) bt_nxt = bt[first_page + 32 + lane];
    }
    // Ring position r < ro: W^R as the MN-major A operand [j half][128 k rows][128 B]; position 0
    // also brings the CTA's query rows, the K-major B operand, into the front of the q_r buffer.
    auto issue_route = [&](int r) {
        const int s = r % NS;
        if (lane == 0) {
            const int wrow = (route_pq ? qh0 + r : g) * kD;
            ptx::mbar_arrive_expect_tx(&sm.full[s],
                                       kTileBytes + (r == 0 ? 2u * (uint32_t)geo.qbox * 128u : 0u));
            ptx::tma_load_2d(sm.tiles[s], &wmap, &sm.full[s], 0, wrow);
            ptx::tma_load_2d(sm.tiles[s] + kHalfBytes, &wmap, &sm.full[s], 64, wrow);
            if (r == 0) {
                ptx::tma_load_2d(sm.qr, &qmap, &sm.full[s], 0, b * geo.Hq + qh0);
                ptx::tma_load_2d(sm.qr + kQHalf, &qmap, &sm.full[s], 64, b * geo.Hq + qh0);
            }
        }
        __syncwarp();
    };
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    grid_dep_launch();
    // the routing loads that fit the ring depend on nothing the CTA still reads
    const int early_route = ro < NS ? ro : NS;
    if (warp == kWideProducer)
        for (int r = 0; r < early_route; ++r) issue_route(r);

    int L = L_raw;
    if (L < 0 || L > geo.max_pages * geo.P) {
        if (tid == 0 && cta == 0 && g == 0) raise_flag(a.err, KL_FLAG_BAD_LENGTH);
        L = 0;
    }
    const int t_end = min(t_begin + geo.spc * geo.chunk, L);
    const int n_tiles = t_end > t_begin ? (t_end - t_begin + kTile - 1) / kTile : 0;
    const bool pos_ok = pos_raw >= 0 && pos_raw < geo.max_pages * geo.P;
    if (a.v_new && !pos_ok && tid == 0 && cta == 0 && g == 0) raise_flag(a.err, KL_FLAG_BAD_POSITION);
    const bool app_owner = a.v_new && pos_ok && pos_raw / (geo.chunk * geo.spc) == cta;

    // An empty run: the new row if it lies there, the zero output of an empty sequence, and no
    // part in the merge (which counts only the runs that hold tokens).
    if (n_tiles == 0) {
        if (app_owner && warp == 0) {
            const int page = bt[pos_raw / geo.P];
            if (page >= 0 && page < geo.num_pages) {
                const size_t off = (((size_t)page * geo.Hkv + g) * geo.P + pos_raw % geo.P) * kD;
                const uint16_t *src = a.v_new + ((size_t)b * geo.Hkv + g) * kD;
                reinterpret_cast<uint2 *>(a.cache_rw + off)[lane] = reinterpret_cast<const uint2 *>(src)[lane];
            } else if (lane == 0) {
                raise_flag(a.err, KL_FLAG_BAD_PAGE);
            }
        }
        if (tid < kD && L == 0 && cta == 0) {
            for (int h = 0; h < G; ++h) {
                const size_t oi = ((size_t)b * geo.Hq + qh0 + h) * kD + tid;
                if (a.out_dtype == KL_FP32) static_cast<float *>(a.out)[oi] = 0.f;
                else static_cast<__nv_bfloat16 *>(a.out)[oi] = __float2bfloat16_rn(0.f);
            }
        }
        if (warp == kWideMma) ptx::tmem_dealloc(sm.tmem_base, kWideTmemCols);
        if (warp == kWideProducer) {
            for (int r = 0; r < early_route; ++r) {
                const uint64_t t0 = ptx::globaltimer();
                while (!ptx::mbar_try_wait(&sm.full[r], 0) && ptx::globaltimer() - t0 < kTimeoutNs) {
                }
            }
        }
        return;
    }

    const uint32_t tmem = sm.tmem_base;
    int issued = 0;                 // ring uses whose copies the producer issued
    const Waiter<kExact> wait{&sm.abort, a.err, a.wait_ns};

    if (warp == kWideProducer) {
        // ------------------------------------------------------------------ producer ----
        const int P = geo.P;
        const int ppt = kTile / P;                   // pages per tile (<= 8)
        const int end_page = (t_end + P - 1) / P;
        const uint32_t page_bytes = (uint32_t)P * 128u;   // one half of one page
        bool bad = false;
        int app_tile = -1;
        size_t app_off = 0;
        uint2 app_val = make_uint2(0, 0);
        if (app_owner) {
            const int page = bt[pos_raw / P];
            if (page >= 0 && page < geo.num_pages) {
                app_tile = pos_raw < t_end ? (pos_raw - t_begin) / kTile : 0;
                app_off = (((size_t)page * geo.Hkv + g) * P + pos_raw % P) * kD;
                app_val = reinterpret_cast<const uint2 *>(a.v_new + ((size_t)b * geo.Hkv + g) * kD)[lane];
            } else if (lane == 0) {
                raise_flag(a.err, KL_FLAG_BAD_PAGE);
            }
        }
        bool ok = true;
        for (int r = 0; ok && r < ro; ++r) {
            if (r >= early_route) {
                ok = wait(&sm.empty[r % NS], ((r / NS) & 1) ^ 1);
                if (!ok) break;
                issue_route(r);
            }
            issued = r + 1;
        }
        const int split_pages = end_page - first_page;
        int bt_batch = 0;
        for (int i = 0; ok && i < n_tiles; ++i) {
            const int r = i + ro, s = r % NS;
            const int p0 = i * ppt;                       // first page of the tile in the run
            if ((p0 >> 5) != bt_batch) {
                bt_batch = p0 >> 5;
                bt_cur = bt_nxt;
                const int q = (bt_batch + 1) * 32 + lane;
                bt_nxt = q < split_pages ? bt[first_page + q] : -1;
            }
            const int page = __shfl_sync(0xffffffffu, bt_cur, ((p0 & 31) + lane) & 31);
            const bool exists = lane < ppt && p0 + lane < split_pages;
            if (r >= NS && !wait(&sm.empty[s], ((r / NS) & 1) ^ 1)) break;
            const bool in_range = exists && page >= 0 && page < geo.num_pages;
            if (exists && !in_range) bad = true;
            if (i == app_tile) {
                reinterpret_cast<uint2 *>(a.cache_rw + app_off)[lane] = app_val;
                ptx::fence_proxy_async_global();
                __syncwarp();
            }
            const unsigned mask = __ballot_sync(0xffffffffu, in_range);
            ptx::for_pages(
                (page * geo.Hkv + g) * P, mask,
                [&] { ptx::mbar_arrive_expect_tx(&sm.full[s], __popc(mask) * page_bytes * 2u); },
                [&](int p, int row) {
                    uint8_t *dst = sm.tiles[s] + p * page_bytes;
                    ptx::tma_load_2d(dst, &vmap, &sm.full[s], 0, row);
                    ptx::tma_load_2d(dst + kHalfBytes, &vmap, &sm.full[s], 64, row);
                });
            issued = r + 1;
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) raise_flag(a.err, KL_FLAG_BAD_PAGE);

    } else if (warp == kWideMma) {
        // ---------------------------------------- routing, then the scores of every tile ----
        constexpr uint32_t idesc_s = ptx::idesc_bf16(128, N, false, false);
        const uint64_t q_desc = ptx::smem_desc(ptx::smem_addr(sm.qr), 16, 1024, ptx::kSwizzle128B);
        const uint64_t k_desc = ptx::smem_desc(ptx::smem_addr(sm.tiles[0]), 16, 1024, ptx::kSwizzle128B);
        const uint64_t w_desc =
            ptx::smem_desc(ptx::smem_addr(sm.tiles[0]), kHalfBytes, 1024, ptx::kSwizzle128B);
        bool ok = true;
        // q_r^T[128 j x N'] = W^R^T (MN-major, ring slot) . q^T (K-major rows of the q_r buffer):
        // one W^R for all NH rows, into the columns of O; or one per query head h, with the
        // block of 16 rows that holds h, into columns 16 h .. (column 16 h + h % 16 is q_r of h).
        for (int r = 0; ok && r < ro; ++r) {
            const int s = r % NS;
            ok = wait(&sm.full[s], (r / NS) & 1);
            if (!ok) break;
            ptx::tc_fence_after();
            if (ptx::elect_one()) {
                const uint64_t w0 = w_desc + ((s * kTileBytes) >> 4);
                const uint64_t q0 = q_desc + (route_pq ? ((r >> 4) * 2048) >> 4 : 0);
                const uint32_t dst = route_pq ? tmem + 16 * r : tmem + kColO;
                const uint32_t idesc_r = route_pq ? ptx::idesc_bf16(128, 16, true, false)
                                                  : ptx::idesc_bf16(128, NH, true, false);
#pragma unroll
                for (int kk = 0; kk < kD / 16; ++kk)
                    ptx::mma_bf16(dst, w0 + ((kk * 2048) >> 4),
                                  q0 + (((kk >> 2) * kQHalf + (kk & 3) * 32) >> 4), idesc_r, kk > 0);
                ptx::mma_commit(&sm.empty[s]);
                if (r == ro - 1) ptx::mma_commit(&sm.r_full);
            }
            __syncwarp();
        }
        ok = ok && wait(&sm.qr_full, 0);
        if (ok) ptx::tc_fence_after();
        for (int i = 0; ok && i < n_tiles; ++i) {
            const int r = i + ro, s = r % NS, sb = i % (2 * NG);
            if (!wait(&sm.full[s], (r / NS) & 1)) break;
            if (i >= 2 * NG && !wait(&sm.s_empty[sb], (i / (2 * NG) - 1) & 1)) break;
            ptx::tc_fence_after();
            if (ptx::elect_one()) {
                const uint64_t a0 = k_desc + ((s * kTileBytes) >> 4);
#pragma unroll
                for (int kk = 0; kk < kD / 16; ++kk)
                    ptx::mma_bf16(tmem + kColS + sb * N,
                                  a0 + (((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4),
                                  q_desc + (((kk >> 2) * kQHalf + (kk & 3) * 32) >> 4), idesc_s, kk > 0);
                ptx::mma_commit(&sm.s_full[sb]);
            }
            __syncwarp();
        }
        // every MMA this warp issued completes before TMEM is freed
        if (ptx::elect_one()) ptx::mma_commit(&sm.drain);
        __syncwarp();
        const uint64_t t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(&sm.drain, 0) && ptx::globaltimer() - t0 < kTimeoutNs) {
        }
    } else if (warp == kWidePv) {
        // ------------------------------------------------------ output MMA issuer -------
        // A = V^T: MN-major SW128, 64-dim halves kHalfBytes apart (LBO), 8-token row groups
        // 1 KiB apart (SBO). B = P^T: MN-major, no swizzle; blocks of 8 columns 128 B apart
        // (SBO), 8-token groups kGroupBytes apart (LBO).
        constexpr uint32_t idesc_o = ptx::idesc_bf16(128, N, true, true);
        const uint64_t v_desc =
            ptx::smem_desc(ptx::smem_addr(sm.tiles[0]), kHalfBytes, 1024, ptx::kSwizzle128B);
        const uint64_t p_desc = ptx::smem_desc(ptx::smem_addr(sm.p[0]), kGroupBytes, 128, ptx::kSwizzleNone);
        for (int j = 0; j < n_tiles; ++j) {
            const int s = (j + ro) % NS, pb = j % NG, k = j / NG;
            if (!wait(&sm.p_full[pb], k & 1)) break;
            ptx::tc_fence_after();
            const int nvalid = min(kTile, t_end - (t_begin + j * kTile));
            const int ksteps = (nvalid + 15) >> 4;
            if (ptx::elect_one()) {
                const uint64_t a0 = v_desc + ((s * kTileBytes) >> 4);
                const uint64_t b0 = p_desc + ((pb * sizeof(sm.p[0])) >> 4);
                for (int kk = 0; kk < ksteps; ++kk)
                    ptx::mma_bf16(tmem + kColO + pb * N, a0 + ((kk * 2048) >> 4),
                                  b0 + ((kk * 2 * kGroupBytes) >> 4), idesc_o, kk > 0);
                ptx::mma_commit(&sm.o_full[pb]);
                ptx::mma_commit(&sm.empty[s]);
            }
            __syncwarp();
        }
        if (ptx::elect_one()) ptx::mma_commit(&sm.drain2);
        __syncwarp();
        const uint64_t t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(&sm.drain2, 0) && ptx::globaltimer() - t0 < kTimeoutNs) {
        }
    } else {
        // ------------------------------------------------------------------ compute -----
        const int grp = NG == 2 ? warp >> 3 : 0, qd = warp & 3, hs = (warp >> 2) & 1;
        const int t = qd * 32 + lane;                   // token, and output dim
        const int h0 = KH * hs;
        const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
        bool ok = true;

        // Routed query, thread = dim t: the groups share the warp pair's KH heads between them
        // (heads h1 .. h1 + KR - 1 each), split into hi and lo bf16 rows of the operand.
        constexpr int KR = KH / NG;
        const int h1 = h0 + KR * grp;
        if (route) {
            ok = wait(&sm.r_full, 0);
            ptx::tc_fence_after();
        }
        if (ok) {
            float acc[KR];
#pragma unroll
            for (int e = 0; e < KR; ++e) {
                const int h = h1 + e;
                acc[e] = 0.f;
                if (h < G) {
                    if (route)
                        acc[e] = ptx::tmem_ld1(tmem + lane_base +
                                               (route_pq ? 16 * h + (h & 15) : kColO + h));
                    else
                        acc[e] = __uint_as_float((uint32_t)a.q[((size_t)b * geo.Hq + qh0 + h) * kD + t] << 16);
                }
            }
            ptx::tc_fence_before();
            // (the query rows at the front of the buffer were read by the routing MMA)
            const float sl2 = geo.scale * kLog2e;
#pragma unroll
            for (int e = 0; e < KR; ++e) {
                const float v = acc[e] * sl2;
                const __nv_bfloat16 hi = __float2bfloat16_rn(v);
                const __nv_bfloat16 lo = __float2bfloat16_rn(v - __bfloat162float(hi));
                const int n = h1 + e, k = t;
                uint8_t *row = sm.qr + (k >> 6) * kQHalf + (n & 7) * 128 +
                               ((((k & 63) >> 3) ^ (n & 7)) << 4) + ((k & 7) << 1);
                *reinterpret_cast<__nv_bfloat16 *>(row + (n >> 3) * 1024) = hi;
                *reinterpret_cast<__nv_bfloat16 *>(row + ((NH + n) >> 3) * 1024) = lo;
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm.qr_full);
        }

        // The group's softmax state: the references in shared memory, this thread's share of the
        // row sums. Padded heads have zero query rows: scores 0, finite, never written out.
        float *const mref = &sm.mref[grp][h0];
        float lsum[KH];
#pragma unroll
        for (int e = 0; e < KH; ++e) lsum[e] = 0.f;
        // One barrier per tile for the group: it counts the threads with a weight past the slack
        // or a failed wait. Only then a second one exchanges the tile maxima (or lets the whole
        // group leave together).
        // summed O of heads h .. h + 7 += the tile's O, hi and lo (thread = output dim t)
        auto fold = [&](int h, bool add) {
            float oh[8], ol[8];
            const uint32_t oc = tmem + kColO + grp * N + h + lane_base;
            const uint32_t fc = tmem + kColF + grp * NH + h + lane_base;
            tmem_ld_cols8(oc, oc + NH, oh, ol);
#pragma unroll
            for (int e = 0; e < 8; ++e) oh[e] += ol[e];
            if (add) {
                tmem_ld_col8(fc, ol);
#pragma unroll
                for (int e = 0; e < 8; ++e) oh[e] += ol[e];
            }
            tmem_st_cols8(fc, oh);
        };
        bool carried = ok;
        ok = true;
        for (int i = grp; i < n_tiles; i += NG) {
            const int k = i / NG, sb = i % (2 * NG);     // the group's tile count, S buffer
            const uint32_t sc = tmem + kColS + sb * N + h0 + lane_base;
            const int nvalid = min(kTile, t_end - (t_begin + i * kTile));
            const bool past = t >= nvalid;               // a token past the end: weight 0
            bool ready = carried && wait(&sm.s_full[sb], (k >> 1) & 1);
            // the weights against the current references, 8 heads at a time
            float p[KH];
            float pmax = 0.f;
            if (ready) {
                ptx::tc_fence_after();
#pragma unroll
                for (int c = 0; c < KH; c += 8) {
                    float hi[8], lo[8], m[8];
                    tmem_ld_cols8(sc + c, sc + NH + c, hi, lo);
                    *reinterpret_cast<float4 *>(m) = *reinterpret_cast<const float4 *>(mref + c);
                    *reinterpret_cast<float4 *>(m + 4) = *reinterpret_cast<const float4 *>(mref + c + 4);
#pragma unroll
                    for (int e = 0; e < 8; e += 2) {
                        const F2 d = sub2(add2(f2(hi[e], hi[e + 1]), f2(lo[e], lo[e + 1])),
                                          f2(m[e], m[e + 1]));
                        p[c + e] = past ? 0.f : ptx::ex2(d.x);
                        p[c + e + 1] = past ? 0.f : ptx::ex2(d.y);
                        pmax = max3(pmax, p[c + e], p[c + e + 1]);
                    }
                }
            }
            const bool first = i == grp;
            // the output MMAs of the group's previous tile are done: its weight buffer is free
            bool freed = first;
            if (first || ptx::bar_popc(kBarGroup + grp, kWideGroupThreads, pmax > kWideLazy || !ready) != 0) {
                // the per-head maximum over the tile's 128 tokens becomes the reference
                if (ready) {
#pragma unroll
                    for (int c = 0; c < KH; c += 8) {
                        float hi[8], lo[8];
                        tmem_ld_cols8(sc + c, sc + NH + c, hi, lo);
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            p[c + e] = past ? -INFINITY : hi[e] + lo[e];
                            const float wm = warp_max_redux(p[c + e]);
                            if (lane == e) sm.red[grp][qd][h0 + c + e] = wm;
                        }
                    }
                    if (!first) ready = freed = wait(&sm.o_full[grp], (k - 1) & 1);
                }
                if (!ptx::bar_and(kBarGroup + grp, kWideGroupThreads, ready)) {
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
#pragma unroll
                for (int c = 0; c < KH; c += 8) {
                    float alpha[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int h = h0 + c + e;
                        const float tmax = fmaxf(fmaxf(sm.red[grp][0][h], sm.red[grp][1][h]),
                                                 fmaxf(sm.red[grp][2][h], sm.red[grp][3][h]));
                        // (scores all -inf so far, as a row of a group's own first tile may be: weights
                        // 0 against any reference, and the reference stays -inf)
                        const float mx = fmaxf(mref[c + e], tmax), mn = mx == -INFINITY ? 0.f : mx;
                        alpha[e] = ptx::ex2(mref[c + e] - mn);    // 0 for the first tile
                        lsum[c + e] *= alpha[e];
                        p[c + e] = ptx::ex2(p[c + e] - mn);
                    }
                    if (!first) {
                        // O holds the group's previous tile, the sum the ones before it: rescale both
                        float oh[8], ol[8];
                        const uint32_t oc = tmem + kColO + grp * N + h0 + c + lane_base;
                        tmem_ld_cols8(oc, oc + NH, oh, ol);
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            oh[e] *= alpha[e];
                            ol[e] *= alpha[e];
                        }
                        tmem_st_cols8(oc, oh);
                        tmem_st_cols8(oc + NH, ol);
                        if (k > 1) {
                            const uint32_t fc = tmem + kColF + grp * NH + h0 + c + lane_base;
                            tmem_ld_col8(fc, oh);
#pragma unroll
                            for (int e = 0; e < 8; ++e) oh[e] *= alpha[e];
                            tmem_st_cols8(fc, oh);
                        }
                    }
                }
                ptx::tmem_wait_st();
                // every warp has read the old references: the new ones take their place (the
                // group's next barrier separates the maxima of two slow tiles the same way)
                ptx::bar_sync(kBarGroup + grp, kWideGroupThreads);
                if (qd == 0 && lane < KH) {
                    const int h = h0 + lane;
                    mref[lane] = fmaxf(mref[lane], fmaxf(fmaxf(sm.red[grp][0][h], sm.red[grp][1][h]),
                                                         fmaxf(sm.red[grp][2][h], sm.red[grp][3][h])));
                }
                ptx::bar_sync(kBarGroup + grp, kWideGroupThreads);
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm.s_empty[sb]);
            // P^T row of token t, this warp's heads, hi and lo (formed before the wait: the MMAs that
            // read the weight buffer are still running)
            uint32_t ph[KH / 2], pl[KH / 2];
#pragma unroll
            for (int e = 0; e < KH / 2; ++e) {
                const F2 pe = f2(p[2 * e], p[2 * e + 1]);
                const F2 l = add2(f2(lsum[2 * e], lsum[2 * e + 1]), pe);
                lsum[2 * e] = l.x;
                lsum[2 * e + 1] = l.y;
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(pe.x, pe.y);
                ph[e] = *reinterpret_cast<const uint32_t *>(&h2);
                const F2 r = sub2(pe, f2(__uint_as_float(ph[e] << 16), __uint_as_float(ph[e] & 0xffff0000u)));
                const __nv_bfloat162 l2 = __floats2bfloat162_rn(r.x, r.y);
                pl[e] = *reinterpret_cast<const uint32_t *>(&l2);
            }
            if (!freed) carried = wait(&sm.o_full[grp], (k - 1) & 1);
            if (carried) {
                if (k > 0) {
                    // fold the group's previous tile; this tile's MMAs start over
                    ptx::tc_fence_after();
#pragma unroll
                    for (int c = 0; c < KH; c += 8) fold(h0 + c, k > 1);
                    ptx::tmem_wait_st();
                    ptx::tc_fence_before();
                }
                uint8_t *row = sm.p[grp] + (t >> 3) * kGroupBytes + (t & 7) * 16 + (h0 >> 3) * 128;
#pragma unroll
                for (int c = 0; c < KH / 8; ++c) {
                    *reinterpret_cast<uint4 *>(row + c * 128) =
                        make_uint4(ph[4 * c], ph[4 * c + 1], ph[4 * c + 2], ph[4 * c + 3]);
                    *reinterpret_cast<uint4 *>(row + (NH / 8 + c) * 128) =
                        make_uint4(pl[4 * c], pl[4 * c + 1], pl[4 * c + 2], pl[4 * c + 3]);
                }
                // rows past the end inside the last 16-token MMA step must be finite: zero them
                // (each of the lane quarter's two warps one 64-dim half)
                if (nvalid < kTile) {
                    const int st = (i + ro) % NS;
                    carried = wait(&sm.full[st], ((i + ro) / NS) & 1);
                    if (carried && past && t < ((nvalid + 15) & ~15)) {
                        uint4 *z = reinterpret_cast<uint4 *>(sm.tiles[st] + hs * kHalfBytes + t * 128);
#pragma unroll
                        for (int c = 0; c < 8; ++c) z[c] = make_uint4(0, 0, 0, 0);
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && carried) ptx::mbar_arrive(&sm.p_full[grp]);
            }
        }
        // the group's last output MMAs (a group without a tile has an empty state)
        const int mine = (n_tiles + NG - 1 - grp) / NG;
        ok = ok && carried;
        if (ok && mine > 0) ok = wait(&sm.o_full[grp], (mine - 1) & 1);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int e = 0; e < KH; ++e) lsum[e] += __shfl_xor_sync(0xffffffffu, lsum[e], off);
        if (lane == 0) {
#pragma unroll
            for (int e = 0; e < KH; ++e) {
                sm.lred[grp][qd][h0 + e] = lsum[e];
            }
        }
        if (ptx::bar_and(kBarComputeAnd, kWideComputeThreads, ok)) {
            ptx::tc_fence_after();
            // merge of the two groups' states, thread = output dim t, heads h1 .. h1 + KR - 1:
            // one run of the whole sequence writes the output, else the run's state
            const int n_cta_u = (L + geo.chunk * geo.spc - 1) / (geo.chunk * geo.spc);
            const bool write_out = a.direct_out || n_cta_u == 1;
            const bool two = NG == 2 && n_tiles > 1;
            const int mine0 = (n_tiles + NG - 1) / NG;
            // O of heads h1 .. h1 + KR - 1 of a group that ran n tiles: the sum and the last tile's
            auto group_o = [&](int gi, int n, float (&o)[KR]) {
                const uint32_t oc = tmem + kColO + gi * N + h1 + lane_base;
                const uint32_t fc = tmem + kColF + gi * NH + h1 + lane_base;
                if constexpr (KR == 8) {
                    float lo[8];
                    tmem_ld_cols8(oc, oc + NH, o, lo);
#pragma unroll
                    for (int e = 0; e < 8; ++e) o[e] += lo[e];
                    if (n > 1) {
                        tmem_ld_col8(fc, lo);
#pragma unroll
                        for (int e = 0; e < 8; ++e) o[e] += lo[e];
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < KR; ++e) {
                        o[e] = ptx::tmem_ld1(oc + e) + ptx::tmem_ld1(oc + NH + e);
                        if (n > 1) o[e] += ptx::tmem_ld1(fc + e);
                    }
                }
            };
            float o0[KR], o1[KR];
            group_o(0, mine0, o0);
            if (two) group_o(NG - 1, n_tiles >> 1, o1);
#pragma unroll
            for (int e = 0; e < KR; ++e) {
                const int h = h1 + e;
                if (h >= G) continue;
                const float m0 = sm.mref[0][h], m1 = two ? sm.mref[NG - 1][h] : -INFINITY;
                const float M = fmaxf(m0, m1);
                const float w0 = ptx::ex2(m0 - M), w1 = two ? ptx::ex2(m1 - M) : 0.f;
                float lt = w0 * ((sm.lred[0][0][h] + sm.lred[0][1][h]) + (sm.lred[0][2][h] + sm.lred[0][3][h]));
                float o = w0 * o0[e];
                if (two) {
                    const auto &l1 = sm.lred[NG - 1];
                    lt += w1 * ((l1[0][h] + l1[1][h]) + (l1[2][h] + l1[3][h]));
                    o += w1 * o1[e];
                }
                const float val = o / lt;
                const size_t bh = (size_t)b * geo.Hq + qh0 + h;
                if (write_out) {
                    if (a.out_dtype == KL_FP32) static_cast<float *>(a.out)[bh * kD + t] = val;
                    else static_cast<__nv_bfloat16 *>(a.out)[bh * kD + t] = __float2bfloat16_rn(val);
                } else {
                    const size_t slot = bh * geo.S + cta;
                    a.part_o[slot * kD + t] = val;
                    if (t == 0) {
                        a.part_ml[slot * 2] = M * kLn2;
                        a.part_ml[slot * 2 + 1] = lt;
                    }
                }
            }
            if (!write_out) {
                // the last CTA of the unit to finish merges its n_cta_u states (as kl_combine)
                ptx::bar_sync(kBarCompute, kWideComputeThreads);
                if (tid == 0)
                    sm.is_last = arrive_last(a.counters + ((size_t)b * geo.Hkv + g) * geo.nhb + hb,
                                             n_cta_u) ? 1 : 0;
                ptx::bar_sync(kBarCompute, kWideComputeThreads);
                if (sm.is_last)
                    merge_states<kWideWarps, kD>(sm, a, b, qh0, G, n_cta_u, tid, warp, lane, wait);
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kWideMma) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, kWideTmemCols);
    }
    // A CTA that gave up: the cache copies still in flight land before its shared memory goes away.
    if (warp == kWideProducer && sm.abort) {
        for (int i = max(0, issued - NS); i < issued; ++i) {
            const uint64_t t0 = ptx::globaltimer();
            while (!ptx::mbar_try_wait(&sm.full[i % NS], (i / NS) & 1) &&
                   ptx::globaltimer() - t0 < kTimeoutNs) {
            }
        }
    }
}

template <int NH, int NG, bool kExact>
cudaError_t launch_kernel_wide(const DecodeArgs &la, const CUtensorMap &vmap, const CUtensorMap &wmap,
                               const CUtensorMap &qmap) {
    const Geometry &g = la.geo;
    const size_t smem = sizeof(WideSmem<NH, NG>);
    static PerDeviceOnce once;
    const cudaError_t e = once.run([&] {
        return cudaFuncSetAttribute(decode_wide_kernel<NH, NG, kExact>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((g.S + g.spc - 1) / g.spc * g.nhb, g.Hkv, g.B);
    cfg.blockDim = dim3(Wide<NH, NG>::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = la.stream;
    const OverlapAttr overlap(cfg);
    return cudaLaunchKernelEx(&cfg, decode_wide_kernel<NH, NG, kExact>, vmap, wmap, qmap, la);
}

template <int NH, int NG>
cudaError_t launch_wide(const DecodeArgs &la, const CUtensorMap &vmap, const CUtensorMap &wmap,
                        const CUtensorMap &qmap) {
    return la.wait_ns < kExactWaitNs ? launch_kernel_wide<NH, NG, true>(la, vmap, wmap, qmap)
                                     : launch_kernel_wide<NH, NG, false>(la, vmap, wmap, qmap);
}

}  // namespace

cudaError_t launch_tc_wide(const DecodeArgs &a) {
    DecodeArgs la = a;
    Geometry &g = la.geo;
    const int64_t sms = device_sm_count();
    // consecutive splits per CTA: the fewest that fit one wave (when the units alone do not fill
    // it), and at most kWideMaxRuns states to merge
    const auto splits_per_cta = [&](int64_t units, int64_t slots) {
        int spc = (g.S + kWideMaxRuns - 1) / kWideMaxRuns;
        if (g.S > 1 && units < slots)
            while ((int64_t)((g.S + spc - 1) / spc) * units > slots) ++spc;
        return spc;
    };
    // Groups of 17 or more heads: CTAs of 32 heads (about 1200 cycles per tile where HBM does not set
    // the pace), unless CTAs of 16 (about 1000) have an SM each and not 6/5 as many splits to run.
    // (Group of 32, measured with CTAs of 16 and of 32: 104 sequences of 8192 tokens 67.7 and 51.4 us,
    // 77 68.1 and 49.8, 30 of 32768 in 4 splits 72.6 and 55.5, 20 of 40000 in 5 71.1 and 53.0, 150 of
    // 1000 in a group of 24 14.9 and 13.9; 52 sequences of 8192, one CTA of 16 on each of 104 SMs,
    // 39.1 and about 45.)
    const int64_t seq_heads = (int64_t)g.B * g.Hkv;
    const int64_t units32 = seq_heads * ((g.G + 31) / 32), units16 = seq_heads * ((g.G + 15) / 16);
    const bool w32 = g.G > 16 && (units16 > sms || 6 * splits_per_cta(units32, sms) <=
                                                       5 * splits_per_cta(units16, sms));
    const int NH = w32 ? 32 : 16;
    g.nhb = (g.G + NH - 1) / NH;
    g.qbox = g.G < NH ? g.G : NH;
    // Blocks of 16 heads that overflow one CTA per SM go two to an SM with one softmax group each:
    // their waves overlap, and the last one shares HBM evenly. (Within one wave, the
    // deeper ring and the two groups of a CTA that has its SM alone are faster.)
    const int64_t units = w32 ? units32 : units16;
    const bool two_per_sm = !w32 && units > sms;
    const int64_t slots = two_per_sm ? 2 * sms : sms;
    g.spc = splits_per_cta(units, slots);
    CUtensorMap vmap, wmap, qmap;
    if (!make_map(&vmap, a.v_cache, kD, (uint64_t)g.num_pages * g.Hkv * g.P, (uint32_t)g.P))
        return cudaErrorInvalidValue;
    wmap = qmap = vmap;
    if (a.w_r) {
        const uint64_t hw = g.wr_per_qh ? (uint64_t)g.Hq : (uint64_t)g.Hkv;
        if (!make_map(&wmap, a.w_r, kD, hw * kD, (uint32_t)kD)) return cudaErrorInvalidValue;
        if (!make_map(&qmap, a.q, kD, (uint64_t)g.B * g.Hq, (uint32_t)g.qbox))
            return cudaErrorInvalidValue;
    }
    if (w32) return launch_wide<32, 2>(la, vmap, wmap, qmap);
    return two_per_sm ? launch_wide<16, 1>(la, vmap, wmap, qmap) : launch_wide<16, 2>(la, vmap, wmap, qmap);
}

}  // namespace kl
