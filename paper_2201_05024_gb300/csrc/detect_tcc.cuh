// detect_tcc.cuh -- reduced-precision detection with both contractions on the tensor cores
// (Sec. III-B detection; the BF16/FP16 form of detect_tc.cuh).
//
// The dist-Gram is the BF16 or FP16 GEMM of detect_tc.cuh (query operand 2 k2 [Re r_s; Im r_s],
// two rows per entry, accumulators in TMEM).  The coefficient sums
//   acc1_k = sum_t g1_tk E_A + g2_tk E_C,   acc2_k = sum_t g1_tk E_B + g2_tk E_A
// (E_A, E_B, E_C the three exponentials of a pair, g1, g2 the entry's two real-split
// coefficients) are a second GEMM Y[s][n] = sum_j X[s][j] G[n][j] over j = (exponential kind c,
// entry t): X = the exponentials in BF16, written by the epilogue threads into shared memory a
// chunk of 16 entries at a time, and G the coefficients arranged per output column (n = k:
// g1 against E_A, g2 against E_C; n = KB + k: g2 against E_A, g1 against E_B) as a BF16 hi + lo
// pair (rows n and NY + n of one operand), so that their rounding does not count.  Y (128 rows x 2 NY
// columns, FP32) accumulates in TMEM over the whole dictionary, its halves added at the end; the FP32
// pipe then only forms the exponent arguments.  Pairs flagged by the cancellation guard (theta = 2^-4,
// see detect_tc.cuh) enter X as zero and are recomputed by direct differences into FP32 sums, one set
// per epilogue group, added in group order.
//
// Both operands that depend on the dictionary alone -- the Gram's entry operand and G -- are
// packed once per call by tcc_pack_kernel into the caller's workspace, one contiguous block per
// 64-entry tile [Gram entry operand | G | -k2 n_t] in exactly the shared-memory layout the MMAs read;
// the detection CTAs fetch a tile with two bulk copies, each into its own ring: the Gram operand's
// stage is free as soon as the Gram has read it, a tile's coefficients only after its last GEMM.
//
// Roles: epilogue groups of four warps (query row = thread mod 128; group g takes the chunks g,
// g + groups, .. of every tile, into its own exponential buffer), which also build the query operand and,
// each for a share of the users, the linear part; one thread that copies and issues the Gram; one that
// copies the coefficients and issues the coefficient GEMMs (each as soon as a chunk is written).  All
// waits are bounded.
//
// What bounds it: the thread that issues the coefficient GEMMs, 12 small MMAs and 4 waits per tile, some
// 390 cycles per chunk of which 270 the three MMAs (stamps: a tile every 1900 cycles; an epilogue chunk
// takes 1200, four at a time).  Measured (BF16, 64 antennas, 16 users, 4096 entries, 262144 vectors):
// 2717 us with one group of four warps, two stages of whole tiles and hi and lo as MMAs of their own;
// 2034 with four groups; 1859 with the rings apart and descriptors made once; 1380 with hi and lo as one
// operand; 1186 with the linear part's rows read once per group (it took 44000 of a CTA's 190000
// cycles) and the coefficient refill two chunks later.
#pragma once

#include <type_traits>

#include "detect_tc.cuh"

namespace apsm {

constexpr int kTccChunk = 16;     // entries per exponential chunk
// The two shapes of a CTA: the wide one (one per SM), and a half one for small dictionaries,
// two of which share an SM, so that one's set-up and output run beside the other's tiles.
template <bool kHalfCta>
struct TccCfg {
    static constexpr int kGroups = kHalfCta ? 2 : 4;   // epilogue groups of 128 threads, a chunk of a tile each in turn
    static constexpr int kXBuf = kGroups;              // exponential buffers, one per group
    static constexpr int kEpi = 128 * kGroups;
    static constexpr int kThreads = kEpi + 64;
    static constexpr int kAcc = kHalfCta ? 1 : 3;      // Gram accumulators
    static constexpr int kGStages = kHalfCta ? 2 : 3;  // coefficient stages: a tile's are free only after its last GEMM
    static constexpr int kCols = kHalfCta ? 256 : 512; // TMEM columns
    static constexpr int kCtas = kHalfCta ? 2 : 1;     // per SM
    static_assert(kTcEntries / kTccChunk % kGroups == 0, "every group the same chunks of each tile");
};
// The half CTA where there are more query tiles than SMs and the set-up counts: dictionaries of up to 8
// tiles, and up to 24 where its waves of two per SM round up to no more than the wide one's.  us of
// device time, wide and half (16 antennas, 6 users, BF16): 128 entries 38900 vectors 24.1 and 18.5,
// 262144: 122.7 and 79.0; 512 entries 50000 vectors 49.4 and 46.7; 1024 entries 50000 vectors (three waves
// or two double ones) 72.5 and 76.0, 65536: 93.8 and 85.8; 4096 entries 262144: 951 and 957.  32 antennas,
// 11 users, 1500 entries: 38900 vectors 80.1 and 76.3, 50000: 113 and 122.
constexpr int kTccSms = 152, kTccHalfTiles = 8, kTccHalfTilesEven = 24;

// Shared-memory matrix descriptor, K-major, no swizzle, with an explicit leading byte offset
// (bytes between k-adjacent core matrices) and stride byte offset (between 8-row groups).
__device__ __forceinline__ uint64_t umma_sdesc_lbo(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// 32 accumulator columns of this warp's 32 lanes.
__device__ __forceinline__ void tcc_tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

template <int M, int KB, bool kHalfCta = false>
struct TccSmem {
    using C = TccCfg<kHalfCta>;
    using Sh = TcShape<M, kHalf>;
    static constexpr int E = kTcEntries;
    static constexpr int NY = round_up(2 * KB, 16);               // coefficient GEMM N
    static constexpr int KX = 3 * kTccChunk;                      // its K per chunk (48)
    static constexpr int kXBytes = kTcRows * KX * 2;              // one exponential buffer
    static constexpr int kGBytes = NY * 3 * E * 2;                // one copy of G for a tile
    // a packed tile (the same layout in the workspace and in a shared-memory stage)
    static constexpr int kOG = Sh::kBytesB;                       // G, 2 NY rows: hi, then lo
    static constexpr int kOH = kOG + 2 * kGBytes;                 // -k2 n_t [E]
    static constexpr int kTile = round_up(kOH + E * 4, 1024);
    static constexpr int kA = 0;
    static constexpr int kS = round_up(Sh::kBytesA, 1024);        // kBS stages of the Gram operand
    static constexpr int kGBytesAll = 2 * kGBytes + E * 4;        // G and norms of a tile
    static constexpr int kGPart = round_up(kGBytesAll, 128);      // C::kGStages stages of them
    static constexpr int kBS = kHalfCta && M == 32 && NY == 32 ? 1 : 2;  // (one where two would take the SM's second CTA)
    static constexpr int kG = kS + kBS * kOG;
    static constexpr int kX = kG + C::kGStages * kGPart;          // exponential buffers
    static constexpr int kBar = kX + C::kXBuf * kXBytes;          // mbarriers
    static constexpr int kTmem = kBar + 24 * 8;
    static constexpr int kBytes = kTmem + 16;
    static_assert(kBytes <= 227 * 1024, "one CTA per SM");
    static_assert(Sh::kBytesB % 16 == 0 && kGBytes % 16 == 0, "bulk-copy granules");
};

// Workspace of the packed form: one kTile block per 64-entry tile of the dictionary capacity.
template <int M, int KB>
constexpr size_t tcc_workspace_bytes(int D) {
    return (size_t)((D + kTcEntries - 1) / kTcEntries) * TccSmem<M, KB>::kTile;
}

// One block per tile: the Gram entry operand (rows 2e: [Re r_t; Im r_t], 2e+1: [-Im r_t; Re r_t],
// in BF16 or FP16), G in BF16 hi + lo, and -k2 n_t; zeros past the held entries.
template <int M, int KB>
__global__ void __launch_bounds__(128) tcc_pack_kernel(const TcArgs a, unsigned char *packed) {
    using Sh = TcShape<M, kHalf>;
    using L = TccSmem<M, KB>;
    constexpr int E = kTcEntries, NY = L::NY, CE = kTccChunk;
    __shared__ float s_coef[E * 2 * KB];
    const int tile = blockIdx.x, ct = threadIdx.x, e0 = tile * E;
    int n_ent = a.n_entries;
    if (a.meta) n_ent = min(n_ent, max(__ldg(a.meta), 0));
    unsigned char *blk = packed + (size_t)tile * L::kTile;
    if constexpr (tc_core_rows<M, kHalf>()) {
        using Rows = EntryRows<M, kHalf>;
        for (int i = 0; i < Rows::P; ++i) {
            int e, h, p;
            Rows::task(ct, i, e, h, p);
            float4 v[Rows::V];
            Rows::load(a.dict, e0 + e, n_ent, p, v);
            Rows::put(blk, e, h, p, v, a.half_fmt);
        }
    } else {
        const int t = e0 + (ct >> 1), h = ct & 1;
        const float2 *rt = a.dict + (size_t)t * M;
        for (int m = 0; m < M; ++m) {
            const float2 v = t < n_ent ? __ldg(rt + m) : make_float2(0.f, 0.f);
            put_elem<kHalf>(blk, Sh::kBytesB, Sh::off(ct, m), h ? -v.y : v.x, a.half_fmt);
            put_elem<kHalf>(blk, Sh::kBytesB, Sh::off(ct, M + m), h ? v.x : v.y, a.half_fmt);
        }
        for (int k = 2 * M; k < Sh::KD; ++k) put_elem<kHalf>(blk, Sh::kBytesB, Sh::off(ct, k), 0.f, a.half_fmt);
    }
    for (int i = ct; i < E * 2 * KB; i += 128) {
        const int e = i / (2 * KB), j = i % (2 * KB), l = j / KB, k = j % KB, t = e0 + e;
        s_coef[i] = (t < n_ent && k < a.K) ? __ldg(a.gamma + ((size_t)t * 2 + l) * a.K + k) : 0.f;
    }
    if (ct < E) {
        const int t = e0 + ct;
        reinterpret_cast<float *>(blk + L::kOH)[ct] = t < n_ent ? -a.k2 * __ldg(a.dict_norm + t) : 0.f;
    }
    __syncthreads();
    // G: row n, k = (chunk c, kind, entry within chunk); one task = one 16-byte core row (8
    // entries of one kind) of one output column
    constexpr int kTasks = NY * 3 * E / 8;
    for (int task = ct; task < kTasks; task += 128) {
        const int n = task % NY, kc = task / NY;  // k-chunk: 6 per chunk
        const int c = kc / 6, kind = (kc % 6) / 2, half8 = kc % 2;
        const int t0 = c * CE + half8 * 8;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float *gr = s_coef + (t0 + i) * 2 * KB;  // [g1 (KB) | g2 (KB)]
            float x = 0.f;
            if (n < KB) {  // acc1: g1 E_A + g2 E_C
                x = kind == 0 ? gr[n] : (kind == 2 ? gr[KB + n] : 0.f);
            } else if (n < 2 * KB) {  // acc2: g2 E_A + g1 E_B
                const int k = n - KB;
                x = kind == 0 ? gr[KB + k] : (kind == 1 ? gr[k] : 0.f);
            }
            v[i] = x;
        }
        uint4 hi, lo;
        uint32_t *hp = &hi.x, *lp = &lo.x;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            const float2 hf = __bfloat1622float2(h2);
            const __nv_bfloat162 l2 = __floats2bfloat162_rn(v[2 * i] - hf.x, v[2 * i + 1] - hf.y);
            hp[i] = *reinterpret_cast<const uint32_t *>(&h2);
            lp[i] = *reinterpret_cast<const uint32_t *>(&l2);
        }
        const int off = L::kOG + (kc * 2 * NY + n) * 16;  // rows n (hi) and NY + n (lo)
        *reinterpret_cast<uint4 *>(blk + off) = hi;
        *reinterpret_cast<uint4 *>(blk + off + NY * 16) = lo;
    }
}

template <int M, int KB, bool kHalfCta>
__global__ void __launch_bounds__(TccCfg<kHalfCta>::kThreads, TccCfg<kHalfCta>::kCtas) detect_tcc_kernel(const TcArgs a, const unsigned char *packed) {
    using Sh = TcShape<M, kHalf>;
    using L = TccSmem<M, KB, kHalfCta>;
    using Cfg = TccCfg<kHalfCta>;
    constexpr int kGroups = Cfg::kGroups, kXBuf = Cfg::kXBuf, kEpi = Cfg::kEpi, kAcc = Cfg::kAcc, kGStages = Cfg::kGStages;
    constexpr int E = kTcEntries, NB = 2 * kTcEntries, CE = kTccChunk, NY = L::NY;
    constexpr int kChunks = E / CE;
    static_assert(KB % 2 == 0 && 2 * KB <= NY, "users in pairs");
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sA = smem + L::kA;
    unsigned char *sS = smem + L::kS;
    unsigned char *sG = smem + L::kG;
    unsigned char *sX = smem + L::kX;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::kBar);
    uint64_t *b_full = bars, *mma_done = bars + 2, *epi_done = mma_done + kAcc, *x_full = epi_done + kAcc,
             *x_free = x_full + kXBuf, *g_full = x_free + kXBuf, *y_done = g_full + kGStages;
    static_assert(2 + 2 * kAcc + 2 * kXBuf + kGStages + 1 <= 24, "barriers");
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L::kTmem);
    __shared__ float s_nq[kEpi];
    __shared__ int s_some;  // some pair of the CTA went to the direct differences
    constexpr uint32_t kYCol = kAcc * NB;  // Gram accumulators below it, Y at it: 2 NY columns, hi and lo
    constexpr uint32_t kCols = Cfg::kCols;
    static_assert(kYCol + 2 * NY <= kCols, "TMEM columns");

    const int tid = threadIdx.x, warp = tid >> 5;
    const int q0 = blockIdx.x * kTcRows;
    int n_ent = a.n_entries;
    if (a.meta) n_ent = min(n_ent, max(__ldg(a.meta), 0));
    const int n_tiles = (n_ent + E - 1) / E;
    const int n_chunks = n_tiles * kChunks;
    const float g2 = 2.f * a.k2;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        s_some = 0;
        for (int i = 0; i < 2; ++i) mbar_init(&b_full[i], 1);
        for (int i = 0; i < kAcc; ++i) {
            mbar_init(&mma_done[i], 1);
            mbar_init(&epi_done[i], kEpi);
        }
        for (int i = 0; i < kGStages; ++i) mbar_init(&g_full[i], 1);
        mbar_init(y_done, 1);
        for (int i = 0; i < kXBuf; ++i) {
            mbar_init(&x_full[i], kTcRows);
            mbar_init(&x_free[i], 1);
        }
        fence_mbar_init();
    }
    // the first two tiles' copies go out before the query operand is built
    __syncthreads();
    auto copy_b = [&](int t) {  // tile t's Gram operand; its coefficients and norms
        mbar_arrive_expect_tx(&b_full[t % L::kBS], (uint32_t)L::kOG);
        bulk_g2s(sS + t % L::kBS * L::kOG, packed + (size_t)t * L::kTile, (uint32_t)L::kOG, &b_full[t % L::kBS]);
    };
    auto copy_g = [&](int t) {
        const int sg = t % kGStages;
        mbar_arrive_expect_tx(&g_full[sg], (uint32_t)L::kGBytesAll);
        bulk_g2s(sG + sg * L::kGPart, packed + (size_t)t * L::kTile + L::kOG, (uint32_t)L::kGBytesAll, &g_full[sg]);
    };
    if (tid == kEpi) {
        for (int t = 0; t < kGStages && t < n_tiles; ++t) {
            if (t < L::kBS) copy_b(t);
            copy_g(t);
        }
    }
    // ---- the query operand (as detect_tc.cuh) -------------------------------------------------
    // (a group takes every kGroups-th piece of eight antennas of its rows)
    static_assert(tc_core_rows<M, kHalf>(), "whole core rows");
    if (warp < 4 * kGroups) {
        constexpr int C = Sh::kCoreK;
        const int row = tid & (kTcRows - 1), s = q0 + row;
        const float2 *rq = a.rx + (size_t)s * M;
        float np = 0.f;
#pragma unroll
        for (int p = tid / kTcRows; p < M / C; p += kGroups) {
            float re[C], im[C];
            if (s < a.N) {
                const float4 *src = reinterpret_cast<const float4 *>(rq + p * C);
#pragma unroll
                for (int q = 0; q < C / 2; ++q) {
                    const float4 v = __ldg(src + q);
                    re[2 * q] = v.x; im[2 * q] = v.y; re[2 * q + 1] = v.z; im[2 * q + 1] = v.w;
                }
            } else {
#pragma unroll
                for (int c = 0; c < C; ++c) re[c] = im[c] = 0.f;
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {
                np = fmaf(re[c], re[c], fmaf(im[c], im[c], np));
                re[c] *= g2;
                im[c] *= g2;
            }
            put_core<kHalf, C>(sA, Sh::kBytesA, Sh::off(row, p * C), re, a.half_fmt);
            put_core<kHalf, C>(sA, Sh::kBytesA, Sh::off(row, M + p * C), im, a.half_fmt);
        }
        s_nq[tid] = np;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    float nq = 0.f;  // this row's squared norm
    if (warp < 4 * kGroups) {
#pragma unroll
        for (int i = 0; i < kGroups; ++i) nq += s_nq[i * kTcRows + (tid & (kTcRows - 1))];
    }
    const bool cta_in_range = __syncthreads_and(a.k2 * nq <= kFactorLimit);
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    bool ok = true;

    if (warp == 4 * kGroups) {
        // ================= tile copies and Gram MMAs (one thread) =================
        if (tid == kEpi) {
            const uint32_t idesc = (1u << 4) | ((a.half_fmt ? 1u : 0u) << 7) | ((a.half_fmt ? 1u : 0u) << 10) |
                                   ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(kTcRows >> 4) << 24);
            const uint64_t ad = umma_sdesc(smem_u32(sA), Sh::SBO);
            int issued = min(L::kBS, n_tiles), committed = -1;
            for (int t = 0; t < n_tiles; ++t) {
                const int sb = t % L::kBS, st = t % kAcc;
                // tile t's operand has landed; the epilogue of tile t - kAcc freed TMEM stage st
                if (!mbar_wait_bounded(&b_full[sb], (t / L::kBS) & 1) ||
                    (t >= kAcc && !mbar_wait_bounded(&epi_done[st], (t / kAcc - 1) & 1))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(st * NB);
                const uint64_t bd = umma_sdesc(smem_u32(sS + sb * L::kOG), Sh::SBO);
#pragma unroll
                for (int s = 0; s < Sh::kSteps; ++s) umma_f16(d, ad + s * 16, bd + s * 16, idesc, s > 0);
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&mma_done[st]))
                             : "memory");
                committed = t;
                if (t + L::kBS < n_tiles) {  // its stage is free once the Gram has read it
                    if (!mbar_wait_bounded(&mma_done[st], (t / kAcc) & 1)) {
                        ok = false;
                        break;
                    }
                    copy_b(t + L::kBS);
                    issued = t + L::kBS + 1;
                }
            }
            // every copy and MMA issued here has landed before the CTA may exit
            for (int t = max(0, issued - L::kBS); t < issued; ++t) mbar_wait_sleepy(&b_full[t % L::kBS], (t / L::kBS) & 1);
            if (committed >= 0) mbar_wait_sleepy(&mma_done[committed % kAcc], (committed / kAcc) & 1);
        }
    } else if (warp == 4 * kGroups + 1) {
        // ================= coefficient copies and GEMM issue (one thread) =================
        if (tid == kEpi + 32) {
            const uint32_t coef_idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * NY >> 3) << 17) |
                                        ((uint32_t)(kTcRows >> 4) << 24);
            const uint32_t y = tmem + kYCol;
            const uint64_t xd0 = umma_sdesc_lbo(smem_u32(sX), kTcRows * 16, 128);
            const uint64_t gd0 = umma_sdesc_lbo(smem_u32(sG), 2 * NY * 16, 128);
            int issued = min(kGStages, n_tiles);
            for (int t = 0; t < n_tiles && ok; ++t) {
                const int sg = t % kGStages;
                if (!mbar_wait_bounded(&g_full[sg], (t / kGStages) & 1)) {
                    ok = false;
                    break;
                }
#pragma unroll
                for (int c = 0; c < kChunks; ++c) {
                    const int g = t * kChunks + c, xb = g % kXBuf;
                    if (!mbar_wait_bounded(&x_full[xb], (g / kXBuf) & 1)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    // X chunk: [k-chunk of 8][128 rows][16 B]; G: [k-chunk of 8][2 NY rows][16 B], this
                    // chunk's k-chunks are 6c .. 6c + 5
                    const uint64_t xd = xd0 + xb * (L::kXBytes >> 4);
                    const uint64_t gd = gd0 + (sg * L::kGPart >> 4) + c * 6 * 2 * NY;
#pragma unroll
                    for (int ks = 0; ks < L::KX / 16; ++ks)
                        umma_f16(y, xd + ks * 2 * kTcRows, gd + ks * 2 * 2 * NY, coef_idesc, (c > 0 || ks > 0 || t > 0) ? 1u : 0u);
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     smem_u32(&x_free[xb]))
                                 : "memory");
                    // the coefficient stage of tile t-1 is free once its last chunk's GEMM is done (whose
                    // x_full also says that every epilogue thread has read the norms); by now it is
                    // (with fewer buffers than chunks a later chunk's x_full has said so already)
                    if (c == kChunks - 2 && t >= 1 && t - 1 + kGStages < n_tiles) {
                        const int gp = t * kChunks - 1;
                        if (kXBuf == kChunks && !mbar_wait_bounded(&x_free[gp % kXBuf], (gp / kXBuf) & 1)) {
                            ok = false;
                            break;
                        }
                        copy_g(t - 1 + kGStages);
                        issued = t + kGStages;
                    }
                }
            }
            // Y's own barrier (its one phase cannot be taken for another, as a group's wait for a chunk that
            // is not its own could); reached on errors too, when the MMAs issued so far are done
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(y_done))
                         : "memory");
            for (int t = max(0, issued - kGStages); t < issued; ++t)
                mbar_wait_sleepy(&g_full[t % kGStages], (t / kGStages) & 1);
            mbar_wait_sleepy(y_done, 0);
        }
    } else {
        // ================= epilogue: exponentials into X, exact pairs in FP32 =================
        const int grp = warp >> 2, row = tid & (kTcRows - 1);
        const float hq = cta_in_range ? 0.f : -a.k2 * nq;
        const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
        const int s_row = q0 + row;
        const float one_m_theta = 1.f - kGuardHalf;
        const float thr_q = one_m_theta * a.k2 * nq;
        const float base_q = a.k2 * nq + hq;
        // direct-difference pairs only: indexed by a variable, so that the sums live in local memory and leave
        // the registers to the exponentials; set at the thread's first such pair (shared memory leaves next to
        // no L1, so every access to them is a trip to L2)
        float acc[2 * KB];
        bool exact = false;
        // A pair's loads go out in few rounds (the first eight users' coefficients, then eight antennas at a
        // time): where such pairs are rare each is a chain of trips to L2 that the other warps of the CTA end
        // up waiting for.  32 antennas, 11 users, 159 entries, 18688 vectors, 9 such pairs among them: 33.4 us with
        // serial loads and sums set and read back one by one, 27.3 so, 25.1 without any such pair (one epilogue
        // group and the sums in registers: 28.6 and 27.2).  16 antennas, 2 users, 1500 entries, 60000 vectors, such
        // pairs in every warp: 2065 and 1356 (2602).
        auto exact_pair = [&](int t) {
            if (t >= n_ent || s_row >= a.N) return;
            const float4 *rq = reinterpret_cast<const float4 *>(a.rx + (size_t)s_row * M);
            const float4 *rt = reinterpret_cast<const float4 *>(a.dict + (size_t)t * M);
            const float *gt = a.gamma + (size_t)t * 2 * a.K;
            constexpr int kU = KB < 8 ? KB : 8;
            float g1[kU], gg[kU];
            auto load_users = [&](int k0) {
#pragma unroll
                for (int i = 0; i < kU; ++i) {
                    g1[i] = k0 + i < a.K ? __ldg(gt + k0 + i) : 0.f;
                    gg[i] = k0 + i < a.K ? __ldg(gt + a.K + k0 + i) : 0.f;
                }
            };
            load_users(0);
            float dA = 0.f, dB = 0.f, dC = 0.f;
#pragma unroll 1
            for (int m = 0; m < M / 2; m += 4) {
                float4 q[4], d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    q[i] = __ldg(rq + m + i);
                    d[i] = __ldg(rt + m + i);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float qx = i & 1 ? q[i / 2].z : q[i / 2].x, qy = i & 1 ? q[i / 2].w : q[i / 2].y;
                    const float dx = i & 1 ? d[i / 2].z : d[i / 2].x, dy = i & 1 ? d[i / 2].w : d[i / 2].y;
                    const float ax = dx - qx, ay = dy - qy;
                    const float bx = dx - qy, by = dy + qx;
                    const float cx = dx + qy, cy = dy - qx;
                    dA = fmaf(ax, ax, fmaf(ay, ay, dA));
                    dB = fmaf(bx, bx, fmaf(by, by, dB));
                    dC = fmaf(cx, cx, fmaf(cy, cy, dC));
                }
            }
            const float eA = ex2(base_q - a.k2 * dA), eB = ex2(base_q - a.k2 * dB), eC = ex2(base_q - a.k2 * dC);
            if (!exact) {
#pragma unroll
                for (int k = 0; k < 2 * KB; ++k) acc[k] = 0.f;
                exact = true;
            }
#pragma unroll 1
            for (int k0 = 0; k0 < a.K; k0 += kU) {
                if (k0 > 0) load_users(k0);
#pragma unroll
                for (int i = 0; i < kU; ++i) {
                    if (k0 + i < a.K) {
                        acc[k0 + i] = fmaf(g1[i], eA, fmaf(gg[i], eC, acc[k0 + i]));
                        acc[KB + k0 + i] = fmaf(g1[i], eB, fmaf(gg[i], eA, acc[KB + k0 + i]));
                    }
                }
            }
        };
        for (int tile = 0; tile < n_tiles && ok; ++tile) {
            const int st = tile % kAcc, sg = tile % kGStages;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&g_full[sg], (tile / kGStages) & 1) &&
                                             mbar_wait_bounded(&mma_done[st], (tile / kAcc) & 1))) {
                ok = false;
                break;
            }
            tc_fence_after();
            const float *hh = reinterpret_cast<const float *>(sG + sg * L::kGPart + 2 * L::kGBytes);
#pragma unroll 1
            for (int c = grp; c < kChunks; c += kGroups) {
                const int g = tile * kChunks + c, xb = g % kXBuf;
                float vr[32];  // (Re z, Im z) of the chunk's 16 entries
                tcc_tmem_ld32(tmem + lane_base + (uint32_t)(st * NB + 32 * c), vr);
                // the coefficient GEMM of chunk g - kXBuf has read buffer xb
                if (g >= kXBuf &&
                    !__all_sync(0xffffffffu, mbar_wait_bounded(&x_free[xb], ((g - kXBuf) / kXBuf) & 1))) {
                    ok = false;
                    break;
                }
                // X row: k-chunk 2 kind + (j / 8) holds entries 8 (j / 8) .. of one kind
                unsigned char *xrow = sX + xb * L::kXBytes + row * 16;
                bool any = false;
#pragma unroll
                for (int h8 = 0; h8 < 2; ++h8) {
                    float hv[8], xA[8], xB[8], xC[8];
                    *reinterpret_cast<float4 *>(hv) = *reinterpret_cast<const float4 *>(hh + CE * c + 8 * h8);
                    *reinterpret_cast<float4 *>(hv + 4) = *reinterpret_cast<const float4 *>(hh + CE * c + 8 * h8 + 4);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float re = vr[16 * h8 + 2 * j], im = vr[16 * h8 + 2 * j + 1], h = hv[j] + hq;
                        any |= fmaxf(re, fabsf(im)) > fmaf(-one_m_theta, hv[j], thr_q);
                        float a2 = re, b2 = im;
                        add2_bcast(a2, b2, h);
                        xA[j] = ex2(a2);
                        xB[j] = ex2(b2);
                        xC[j] = ex2(h - im);
                    }
                    const float *src[3] = {xA, xB, xC};
#pragma unroll
                    for (int kind = 0; kind < 3; ++kind) {
                        uint4 v;
                        uint32_t *vp = &v.x;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const __nv_bfloat162 b2 = __floats2bfloat162_rn(src[kind][2 * i], src[kind][2 * i + 1]);
                            vp[i] = *reinterpret_cast<const uint32_t *>(&b2);
                        }
                        *reinterpret_cast<uint4 *>(xrow + (2 * kind + h8) * kTcRows * 16) = v;
                    }
                }
                // flagged: max(v_re, |v_im|) > (1 - theta) k2 (n_s + n_t); such a pair's exponentials leave X
                uint32_t fbits = 0;
                const bool slow = __any_sync(0xffffffffu, any);
                if (slow) {
#pragma unroll
                    for (int j = 0; j < CE; ++j) {
                        const bool f = fmaxf(vr[2 * j], fabsf(vr[2 * j + 1])) > fmaf(-one_m_theta, hh[CE * c + j], thr_q);
                        if (f) {
                            fbits |= 1u << j;
#pragma unroll
                            for (int kind = 0; kind < 3; ++kind)
                                *reinterpret_cast<uint16_t *>(xrow + (2 * kind + j / 8) * kTcRows * 16 + (j & 7) * 2) = 0;
                        }
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive(&x_full[xb]);
                if (slow) {
#pragma unroll 1
                    while (fbits) {
                        const int j = __ffs(fbits) - 1;
                        fbits &= fbits - 1;
                        exact_pair(tile * E + CE * c + j);
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();
            mbar_arrive(&epi_done[st]);
        }
        // ---- Y (complete once the last chunk's GEMM has committed) plus the exact pairs -----------
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(y_done, 0))) ok = false;
        tc_fence_after();
        // the groups' exact sums meet in the tile stages, which nothing reads any more; each group then
        // writes its share of the users
        float *s_acc = reinterpret_cast<float *>(sS);  // [group][2KB][128 rows]
        static_assert(kGroups * 2 * KB * kTcRows * 4 <= L::kX - L::kS, "exact sums fit the tile stages");
        // the filter as [antenna][KB] behind them, for the linear part
        float2 *s_clin = reinterpret_cast<float2 *>(sX);
        static_assert(M * KB * 8 <= kXBuf * L::kXBytes, "filter fits the exponential buffers");
        for (int i = tid; i < M * KB; i += kEpi)
            s_clin[i] = i % KB < a.K ? __ldg(a.clin + (size_t)(i / KB) * a.K + i % KB) : make_float2(0.f, 0.f);
        const bool warp_exact = __any_sync(0xffffffffu, exact);
        if (warp_exact) s_some = 1;
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"n"(kEpi) : "memory");
        const bool some = *reinterpret_cast<volatile int *>(&s_some) != 0;
        if (some) {
#pragma unroll
            for (int n = 0; n < 2 * KB; ++n) s_acc[(grp * 2 * KB + n) * kTcRows + row] = exact ? acc[n] : 0.f;
            asm volatile("bar.sync 1, %0;" ::"n"(kEpi) : "memory");
        }
        constexpr int KG = (KB + kGroups - 1) / kGroups;  // users per group
        float y[NY];
#pragma unroll
        for (int n = 0; n < NY; ++n) y[n] = 0.f;
        if (ok && n_chunks > 0) {
#pragma unroll
            for (int n0 = 0; n0 < NY; n0 += 16) {
                float lo[16];
                tmem_ld16(tmem + lane_base + (uint32_t)(kYCol + n0), *reinterpret_cast<float(*)[16]>(y + n0));
                tmem_ld16(tmem + lane_base + (uint32_t)(kYCol + NY + n0), lo);
#pragma unroll
                for (int n = 0; n < 16; ++n) y[n0 + n] += lo[n];
            }
        }
        const int s = s_row, k0 = grp * KG;
        if (ok && s < a.N) {
            const float fq = cta_in_range ? ex2(-a.k2 * nq) : 1.f;
            const float2 *rq = a.rx + (size_t)s * M;
            float l1[KG], l2[KG], y1[KG], y2[KG];
#pragma unroll
            for (int u = 0; u < KG; ++u) {
                l1[u] = l2[u] = y1[u] = y2[u] = 0.f;
#pragma unroll
                for (int gi = 0; gi < kGroups; ++gi)
                    if (gi == grp && gi * KG + u < KB) {
                        y1[u] = y[gi * KG + u];
                        y2[u] = y[KB + gi * KG + u];
                    }
            }
#pragma unroll 2
            for (int m = 0; m < M; m += 8) {
                float4 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = __ldg(reinterpret_cast<const float4 *>(rq + m) + q);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float x = c & 1 ? v[c / 2].z : v[c / 2].x, z = c & 1 ? v[c / 2].w : v[c / 2].y;
#pragma unroll
                    for (int u = 0; u < KG; ++u) {
                        const float2 cl = s_clin[(m + c) * KB + min(k0 + u, KB - 1)];
                        l1[u] = fmaf(cl.x, x, fmaf(cl.y, z, l1[u]));
                        l2[u] = fmaf(cl.x, z, fmaf(-cl.y, x, l2[u]));
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < KG; ++u) {
                const int k = k0 + u;
                if (k >= a.K || k >= KB) continue;
                float e1 = 0.f, e2 = 0.f;
                if (some)
                    for (int gi = 0; gi < kGroups; ++gi) {
                        e1 += s_acc[(gi * 2 * KB + k) * kTcRows + row];
                        e2 += s_acc[(gi * 2 * KB + KB + k) * kTcRows + row];
                    }
                const float v1 = fmaf(a.wL, l1[u], a.wG * fq * (y1[u] + e1));
                const float v2 = fmaf(a.wL, l2[u], a.wG * fq * (y2[u] + e2));
                a.soft[(size_t)s * a.K + k] = make_float2(v1, v2);
                if (a.hard) a.hard[(size_t)s * a.K + k] = (uint8_t)((v1 < 0.f ? 1 : 0) | (v2 < 0.f ? 2 : 0));
            }
        }
    }
    if (!ok && (tid & 31) == 0) report(a.status, APSM_ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// Packs the dictionary's operands into `workspace` (tcc_workspace_bytes(D) bytes, 16-byte
// aligned) and runs the detection; with a smaller or missing workspace the form of
// detect_tc.cuh (coefficient sums on the FP32 pipe) runs instead.
template <int M, int KB>
cudaError_t launch_detect_tcc(const TcArgs &a, void *workspace, size_t ws_bytes, cudaStream_t stream) {
    const int grid = (a.N + kTcRows - 1) / kTcRows;
    if (grid == 0) return cudaSuccess;
    const int n_tiles = (a.n_entries + kTcEntries - 1) / kTcEntries;
    if (!workspace || ws_bytes < tcc_workspace_bytes<M, KB>(a.n_entries) ||
        (reinterpret_cast<uintptr_t>(workspace) & 15))
        return launch_detect_tc<M, KB, kHalf>(a, stream);
    unsigned char *packed = static_cast<unsigned char *>(workspace);
    tcc_pack_kernel<M, KB><<<n_tiles, 128, 0, stream>>>(a, packed);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    auto run = [&](auto half) {
        constexpr bool kHalfCta = decltype(half)::value;
        using S = TccSmem<M, KB, kHalfCta>;
        auto fn = detect_tcc_kernel<M, KB, kHalfCta>;
        const cudaError_t r = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kBytes);
        if (r != cudaSuccess) return r;
        fn<<<grid, TccCfg<kHalfCta>::kThreads, S::kBytes, stream>>>(a, packed);  // ordinary launches (see launch_detect_tc)
        return cudaGetLastError();
    };
    if constexpr (2 * (TccSmem<M, KB, true>::kBytes + 4096) <= 228 * 1024) {
        const bool even = (grid + kTccSms - 1) / kTccSms == 2 * ((grid + 2 * kTccSms - 1) / (2 * kTccSms));
        if (grid > kTccSms && n_tiles <= (even ? kTccHalfTilesEven : kTccHalfTiles)) return run(std::true_type{});
    }
    return run(std::false_type{});
}

using TccLauncher = cudaError_t (*)(const TcArgs &, void *, size_t, cudaStream_t);

}  // namespace apsm
