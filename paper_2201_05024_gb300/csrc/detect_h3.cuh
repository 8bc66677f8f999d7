// detect_h3.cuh -- FP32-accuracy detection for 16, 32 and 64 antennas with the complex dist-Gram on the
// tensor cores as three FP16 products (Sec. III-B detection; the same result as detect_tc.cuh).
//
// FP16 and TF32 hold the same 11 significant bits, so hi*hi + hi*lo + lo*hi with hi = fp16(x),
// lo = fp16(x - hi) is as exact as the TF32 x3 form while an operand copy takes half the shared
// memory and the MMAs run at twice the rate: at 64 antennas the TF32 copies of 128 queries and two
// entry tiles do not fit an SM at all.  FP16's narrow exponent is taken care of by one power of two
// per row, from the row's squared norm: a row scaled to components below 2^12 keeps its hi
// components exact to 11 bits and its lo ones to 2^-36 of the row; the factors return to the
// exponent in FP32 (m = 2 k2 / (query scale x entry scale), one multiply per pair).
//
// A CTA takes 256 queries (two MMA tiles of 128 rows) against a run of 32-entry tiles.  Entry rows
// 2e = [Re r_t; Im r_t] and 2e+1 = [-Im r_t; Re r_t] give Re z and Im z in adjacent accumulator
// columns.  Each epilogue thread owns one row of BOTH query tiles, so that a coefficient read from
// shared memory serves two pairs.  The linear part stays in FP32 (each CTA of a cluster a share of
// the antennas): as one more tile of the Gram, a filter in place of an entry, it cost nothing, but the
// MMA's sums left 4.6e-7 of error in the outputs where FP32 leaves 1.6e-7.
//
// Inside the factor range (k2 n_s <= kFactorLimit for every query of the CTA) the Gram's error is
// below 2^-21 of k2 (n_s + n_t) in the exponent wherever a term matters; a CTA with a query
// outside it takes the unfactored exponent and, for the rows that need it, FP32 direct differences
// (H3Guard).
//
// Work split: CTAs of a cluster share one query tile and take contiguous parts of the dictionary;
// at the end each CTA sums the parts of its share of the rows through distributed shared memory,
// in CTA order (results do not depend on timing).  The cluster size fills the SMs when there are
// few query tiles; many go one CTA each in whole waves, the last, partial wave split (h3_plan).
//
// Roles (384 threads): warps 0-7 prepare the query operand, then are the epilogue (TMEM lanes
// 32 (w mod 4) .., entries 16 (w / 4) .. of a tile), warps 8-10 convert entry tiles (hi and lo copies,
// coefficients, norms; a tile's global loads are issued before the wait for its stage), warp 11
// issues the MMAs.  Entry operand two stages, coefficients four, accumulators four over the sums
// (h3_sums).  All waits on an mbarrier are bounded; a timed-out CTA still meets its cluster at both barriers.  Those and the TMEM
// allocation are the hardware's own waits, without a limit, and end because a CTA has its SM to itself as
// far as this kernel goes (kH3OneCta) and no other kernel waits for another CTA while it holds TMEM.
//
// What bounds it: the FP32 pipe, 4K + 4 FMA per pair (cycle stamps at 64 antennas and 16 users: the
// epilogue of a tile takes 6700 cycles, 5700 while the converters rest, against 4400 of packed FMAs;
// the MMAs 3000, beside it; ncu: FMA pipe 66 % active).
// Measured (FP32, 64 antennas, 16 users, 4096 entries, 100003 vectors): 8025 us on the FMA engine
// (323 FMA per pair), 1290 us here.  32 antennas, 11 users, 1500 entries, 10001 vectors: 110 us in the
// TF32 x3 converter form (79 CTAs of 128 queries for 152 SMs), 62 us here.  16 antennas, 6 users, 1024
// entries: an entry tile takes 3340 cycles (1800 of FMAs) against 3950 per 32 entries and 256 queries in
// the TMA-staged TF32 x3 form; resting the converters, dropping the exponentials or the coefficient reads
// saves 5, 5 and 10 %, four epilogue groups instead of two nothing: warps wait for the FMA pipe.
#pragma once

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "detect_tc.cuh"

namespace apsm {

constexpr int kH3Rows = 256;      // queries per CTA
constexpr int kH3Entries = 32;    // entries per tile
constexpr int kH3Epi = 256;       // epilogue threads
constexpr int kH3Conv = 96;       // converter threads
constexpr int kH3Threads = kH3Epi + kH3Conv + 32;
constexpr int kH3MaxSplit = 8;    // CTAs per cluster
// 16 antennas: dictionaries up to here keep the TMA-staged form.  This is not where the forms cross (us of
// device time, TMA-staged form and this; 6 users, 260 entries: 64 vectors 16.2 and 10.6, 16384: 34.8 and 17.1,
// 100000: 84.6 and 70.9; 1024 entries: 64 vectors 25.7 and 13.8, 4000: 33.1 and 19.0, 65536: 138.6 and 128.0;
// 2 users, 1024, 65536: 93.1 and 84.5; 16 users: 258.8 and 236.9), which lies lower.  It is the largest
// dictionary whose results are kept to the last bit: gradient calls train on up to 256 pilots and return
// their sums over these outputs in FP64, in which any other rounding of the Gram shows.
constexpr int kH3MinEntries16 = 256;
// Whether this form takes a call of N vectors.  Its CTA is set up for 256 queries and its first tile of entries
// takes as long as a full one, so small dictionaries over few vectors keep the former form (us of device
// time, former and this):
//   64 antennas (FMA engine)  6 users, 300 vectors: 1 entry 5.6 and 22.0, 64: 13.2 and 18.9, 96: 17.6 and 18.1, 97:
//                             18.7 and 17.7; 16 users: 96: 20.0 and 25.2, 128: 24.2 and 25.1, 160: 28.5 and 26.6;
//                             12000 vectors, 6 users: 32: 15.4 and 22.3, 64: 23.0 and 19.0; 11 users: 16: 22.9 and
//                             26.2, 32: 31.0 and 26.3
//   32 antennas (TF32 x3)     300 vectors, 2 users: 32: 10.0 and 12.1, 64: 10.7 and 10.9, 65: 13.0 and 10.5; 6 users: 32:
//                             12.3 and 14.5, 33: 12.6 and 12.8; 24000 vectors, 2 users, 1 entry: 18.4 and 12.7
inline bool h3_pays(int M, int K, int dict_cap, int N) {
    if (M == 16) return dict_cap > kH3MinEntries16;
    if (M == 32) return dict_cap > (K <= 4 ? 64 : 32) || N > 16384;
    return dict_cap > (K > 12 ? 128 : 96) || (long long)N * dict_cap > (K <= 8 ? 400000 : 300000);
}
constexpr int kH3Devices = 16;    // devices whose cluster counts are kept
// One CTA per SM is a condition of this kernel, not a matter of occupancy: a CTA holds all 512 TMEM
// columns while it waits for its cluster, so of two on one SM the second would wait in its allocation,
// and two clusters that meet on two SMs in opposite order would wait for each other for ever.  (Registers do
// not see to it: at 16 antennas and 2 users two fitted with 77 a thread and 53 KB of shared memory.)  So every launch asks for
// more than half of an SM's 228 KB, of which each CTA has 1 KB reserved.
constexpr int kH3OneCta = 116 * 1024;
static_assert(2 * (kH3OneCta + 1024) > 228 * 1024, "two CTAs of any instantiations do not fit an SM");

// Outside the factor range the exponent X - S (X = 2 k2 max(Re z, |Im z|), S = k2 (n_s + n_t)) is off by up to
// 2^-21 S and its term by as much of itself.  Where 2^(X - S) S <= 4 that is less than 2e-6 of a coefficient;
// a row with a nearer entry (inputs that share a large offset, which the norm expansion cancels) takes direct
// differences for all of this CTA's entries.  The test is X <= S - (A + B S) with A + B S >= log2(S) - 2, its
// tangent at S0 = 2 k2 n_s, plus 2^-12 S for the error itself at any S.
// Measured (us; the former TF32 x3 or FMA form, the whole CTA by direct differences, and this; 16 antennas, 6
// users, 1024 entries, 65536 vectors / 32, 11, 1500, 10001 / 64, 16, 4096, 20000): one row in 97 outside 161, 754,
// 151 / 120, 389, 72 / 2493, 3508, 368; every row, far from the entries, 160, 755, 150 / 119, 388, 72 / 4155, 3509,
// 368; a common offset that cancels in every pair 160, 755, 705 / 119, 388, 361 / 4149, 3509, 3087, the former
// forms with errors of up to 6e-5 and 2.5e-4 of the output scale at 16 and 32 antennas, this one 1e-6.
struct H3Guard {
    float a, b1;  // -A, B - 1: nearer if X > fmaf(b1, -S, a); never for a row inside the range
};
__device__ __forceinline__ H3Guard h3_guard(float k2_ns) {
    const float s0 = 2.f * k2_ns, e = 1.442695f;
    if (!(k2_ns > kFactorLimit)) return H3Guard{INFINITY, 0.f};
    return H3Guard{2.f + e - __log2f(s0), e / s0 + kGuardF32 - 1.f};
}

// Sums that hi times hi of a pair is formed in, each over a share of the antennas, added in FP32: every MMA
// truncates the sum it adds to, so shorter and smaller sums lose less.  Few users' outputs average the
// errors of the Gram the least.  With four sums a stage takes all of TMEM, so its halves (16 entries each,
// one half of the epilogue) are issued, waited for and released one by one, which keeps the MMAs running.
// Error of the outputs against 64 bits at 64 antennas, FMA engine and this (rms over the output's):
//   2 users, 300 / 700 / 1500 entries   1.64, 2.43, 3.88e-7   four sums 1.29, 1.78, 2.43e-7 (two 1.89, 2.78, 3.51e-7)
//   3 users, 300 / 700                  1.23, 1.66e-7         two sums 1.15, 1.62e-7
//   6 users, 300 / 4096                 1.08, 2.71e-7         two sums 0.64, 1.49e-7
//   8, 12, 16 users, 300                1.06, 1.12, 1.17e-7   one sum 0.64, 0.65, 0.67e-7
// Four sums cost time: 2 users, 1024 entries, 40000 vectors 152 us against 97 with two (FMA engine 666).
constexpr int h3_sums(int M, int KB) { return M < 64 || KB > 6 ? 1 : KB > 2 ? 2 : 4; }

template <int M, int KB>
struct H3Smem {
    static constexpr int kCols = 2 * M / 8;                 // 16-byte k-columns of an operand row
    static constexpr int SBO = kCols * 128;                 // bytes per 8-row group
    static constexpr int kACopy = 128 / 8 * SBO;            // one query tile, one copy
    static constexpr int kBCopy = 2 * kH3Entries / 8 * SBO;
    static constexpr int kCStage = kH3Entries * 2 * KB * 4;
    static constexpr int kPart = kH3Rows + 1;               // row stride of a partial sum's column (odd)
    static constexpr int kA = 0;                            // [query tile][hi, lo]
    static constexpr int kB = kA + 4 * kACopy;              // 2 stages x [hi, lo]
    static constexpr int kC = kB + 4 * kBCopy;              // 4 stages of coefficients [E][2KB]
    static constexpr int kH = kC + 4 * kCStage;             // 4 stages of (1 / scale, -k2 n_t) [E]
    static constexpr int kN = kH + 4 * kH3Entries * 8;      // query norms [256]
    static constexpr int kBar = kN + kH3Rows * 4;
    static constexpr int kMask = kBar + 19 * 8;             // rows that take direct differences [8]
    static constexpr int kTmem = round_up(kMask + 8 * 4, 16);
    static constexpr int kBytes = kTmem + 16;
    // rows that take direct differences (h3_direct_rows): their queries, then a tile of entries, after
    // the partial sums in the operands' space and the first coefficient stages (the last holds theirs), at 16
    // antennas behind everything, in what the launch asks for anyway
    static constexpr int kDStride = M + 2;                  // float2 per entry row (groups of a warp: other banks)
    static constexpr int kDirectQ = M > 16 ? 2 * KB * kPart * 4 : kBytes;
    static constexpr int kDirectD = kDirectQ + kH3Rows * M * 8;
    static constexpr int kDirectEnd = kDirectD + kH3Entries * kDStride * 8;
    static_assert(kDirectEnd <= (M > 16 ? kC + 3 * kCStage : kH3OneCta), "within them");
    static_assert(kDirectQ % 16 == 0 && 2 * KB * kH3Rows * 4 <= kDirectEnd - kDirectQ, "aligned; the groups' sums fit");
    // what a launch asks for: more than half an SM, whatever the registers allow (kH3OneCta)
    static constexpr int kLaunch = std::max(kBytes, kH3OneCta);
    // the sums [2KB][kPart] reuse the operands when every MMA is done
    static_assert(2 * KB * kPart * 4 <= kC, "partial sums fit the operand space");
    static_assert(kLaunch <= 227 * 1024, "fits an SM");
};

// Power of two that brings a vector of squared norm n to components below 2^12 (1 for n = 0), and its
// inverse; 0 for a norm that is not finite, whose row then enters the MMAs as zeros.
__device__ __forceinline__ float h3_scale(float n, float &inv) {
    const int ex = (int)((__float_as_uint(n) >> 23) & 0xff);  // biased exponent
    if (ex == 0xff) {
        inv = 1.f;
        return 0.f;
    }
    const int c = n > 0.f ? (ex - 127 + 2) >> 1 : 12;         // |component| <= sqrt(n) < 2^c
    inv = __uint_as_float((uint32_t)(c - 12 + 127) << 23);
    return __uint_as_float((uint32_t)(12 - c + 127) << 23);
}

// Eight FP32 values as FP16 hi and lo, 16 bytes each.
__device__ __forceinline__ void h3_split8(const float (&x)[8], uint4 &hi, uint4 &lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h[i]) : "f"(x[2 * i + 1]), "f"(x[2 * i]));
        float a, b;
        asm("{\n\t.reg .b16 p, q;\n\tmov.b32 {p, q}, %2;\n\tcvt.f32.f16 %0, p;\n\tcvt.f32.f16 %1, q;\n\t}"
            : "=f"(a), "=f"(b)
            : "r"(h[i]));
        a = x[2 * i] - a;
        b = x[2 * i + 1] - b;
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(l[i]) : "f"(b), "f"(a));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Eight antennas of a row (four float4 of interleaved Re, Im) times s.
__device__ __forceinline__ void h3_unpack(const float4 (&v)[4], float s, float (&re)[8], float (&im)[8]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        re[2 * i] = v[i].x * s;
        im[2 * i] = v[i].y * s;
        re[2 * i + 1] = v[i].z * s;
        im[2 * i + 1] = v[i].w * s;
    }
}

__device__ __forceinline__ void h3_tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ float ld_cluster(uint32_t smem_addr, uint32_t rank) {
    uint32_t a;
    float v;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}

// Adds the kernel sums of the rows in `mask` (one bit per query row of the CTA) to their partial sums, by FP32
// direct differences against this CTA's entries.  Called by the whole CTA when its operands are free.  The
// rows are gathered into a power of two of 8 to 256 slots; 256 threads take a slot each and, with few rows, one
// of 256 / slots groups of the entries, so that one such row in a tile costs a fraction of it.
template <int M, int KB>
__device__ __noinline__ void h3_direct_rows(const TcArgs &a, unsigned char *smem, const uint32_t *mask, int *count, int q0,
                                            int t_lo, int J, int n_ent) {
    using L = H3Smem<M, KB>;
    constexpr int E = kH3Entries, S = L::kDStride;
    float *s_part = reinterpret_cast<float *>(smem), *s_grp = reinterpret_cast<float *>(smem + L::kDirectQ);
    float2 *sq = reinterpret_cast<float2 *>(smem + L::kDirectQ);  // [M][slots]
    float2 *sd = reinterpret_cast<float2 *>(smem + L::kDirectD);  // [E][S]
    float *sC = reinterpret_cast<float *>(smem + L::kC + 3 * L::kCStage);
    int *rows = reinterpret_cast<int *>(smem + L::kH);
    static_assert(kH3Rows * 4 <= 4 * E * 8, "row list in the norms' stages");
    const int tid = threadIdx.x, lane = tid & 31;
    __syncthreads();  // the mask and the partial sums are complete, the operands and the norms' stages free
    if (tid < 32) {
        int n = 0;
        for (int w = 0; w < kH3Rows / 32; ++w) {
            const uint32_t m = mask[w];
            if (m >> lane & 1) rows[n + __popc(m & ((1u << lane) - 1u))] = 32 * w + lane;
            n += __popc(m);
        }
        if (lane == 0) *count = n;
    }
    __syncthreads();
    const int n_rows = *count;
    if (n_rows == 0) return;
    int slots = 8;
    while (slots < n_rows) slots *= 2;
    for (int i = tid; i < slots * (M / 2); i += kH3Threads) {
        const int r = i & (slots - 1), c = i / slots;
        const float4 v = r < n_rows ? __ldg(reinterpret_cast<const float4 *>(a.rx + (size_t)(q0 + rows[r]) * M) + c)
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
        sq[2 * c * slots + r] = make_float2(v.x, v.y);
        sq[(2 * c + 1) * slots + r] = make_float2(v.z, v.w);
    }
    const int slot = tid & (slots - 1), grp = tid / slots, groups = kH3Rows / slots;
    float acc1[KB], acc2[KB];
#pragma unroll
    for (int k = 0; k < KB; ++k) acc1[k] = acc2[k] = 0.f;
    // this group's entries of a tile, kT at a time (a query component serves kT pairs), x and y parts of
    // the differences as packed pairs
    auto tile = [&](auto t_c, int cnt) {
        constexpr int kT = decltype(t_c)::value;
        const uint64_t neg = pack2(-1.f, -1.f), turn_b = pack2(-1.f, 1.f), turn_c = pack2(1.f, -1.f);
#pragma unroll 1
        for (int e = grp; e < cnt; e += kT * groups) {
            uint64_t dA[kT], dB[kT], dC[kT];
            const float2 *row[kT];
#pragma unroll
            for (int i = 0; i < kT; ++i) {
                dA[i] = dB[i] = dC[i] = 0;
                row[i] = sd + min(e + i * groups, cnt - 1) * S;
            }
#pragma unroll 2
            for (int m = 0; m < M; m += 2) {
                const float2 q[2] = {sq[m * slots + slot], sq[(m + 1) * slots + slot]};
                const uint64_t qs[2] = {pack2(q[0].x, q[0].y), pack2(q[1].x, q[1].y)};
                const uint64_t qt[2] = {pack2(q[0].y, q[0].x), pack2(q[1].y, q[1].x)};
#pragma unroll
                for (int i = 0; i < kT; ++i) {
                    const float4 d = *reinterpret_cast<const float4 *>(row[i] + m);
                    const uint64_t t[2] = {pack2(d.x, d.y), pack2(d.z, d.w)};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint64_t x = ffma2(qs[h], neg, t[h]), y = ffma2(qt[h], turn_b, t[h]), z = ffma2(qt[h], turn_c, t[h]);
                        dA[i] = ffma2(x, x, dA[i]);  // r_t - r_s
                        dB[i] = ffma2(y, y, dB[i]);  // r_t + i r_s
                        dC[i] = ffma2(z, z, dC[i]);  // r_t - i r_s
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < kT; ++i) {
                if (e + i * groups >= cnt) break;
                const float eA = ex2(-a.k2 * sum2(dA[i])), eB = ex2(-a.k2 * sum2(dB[i])), eC = ex2(-a.k2 * sum2(dC[i]));
                float g1[KB], gg[KB];
                load_coef<KB>(sC + (e + i * groups) * 2 * KB, g1, gg);
#pragma unroll
                for (int k = 0; k < KB; k += 2) {
                    fma2_pair(acc1[k], acc1[k + 1], gg[k], gg[k + 1], eC);
                    fma2_pair(acc1[k], acc1[k + 1], g1[k], g1[k + 1], eA);
                    fma2_pair(acc2[k], acc2[k + 1], gg[k], gg[k + 1], eA);
                    fma2_pair(acc2[k], acc2[k + 1], g1[k], g1[k + 1], eB);
                }
            }
        }
    };
    for (int j = 0; j < J; ++j) {
        const int e0 = (t_lo + j) * E, cnt = min(E, n_ent - e0);
        __syncthreads();
        for (int i = tid; i < cnt * (M / 2); i += kH3Threads)
            *reinterpret_cast<float4 *>(sd + i / (M / 2) * S + i % (M / 2) * 2) =
                __ldg(reinterpret_cast<const float4 *>(a.dict + (size_t)e0 * M) + i);
        for (int i = tid; i < cnt * 2 * KB; i += kH3Threads) {
            const int t = e0 + i / (2 * KB), l = i / KB % 2, k = i % KB;
            sC[i] = k < a.K ? __ldg(a.gamma + ((size_t)t * 2 + l) * a.K + k) : 0.f;
        }
        __syncthreads();
        if (tid < kH3Rows) {
            if (groups <= E / 4) tile(std::integral_constant<int, 4>{}, cnt);
            else tile(std::integral_constant<int, 1>{}, cnt);
        }
    }
    // the groups' sums [group][2KB][slots], added in group order
    __syncthreads();
    if (tid < kH3Rows) {
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            s_grp[(grp * 2 * KB + k) * slots + slot] = acc1[k];
            s_grp[(grp * 2 * KB + KB + k) * slots + slot] = acc2[k];
        }
    }
    __syncthreads();
    for (int i = tid; i < 2 * KB * slots; i += kH3Threads) {
        const int r = i & (slots - 1), k = i / slots;
        if (r >= n_rows) continue;
        float y = 0.f;
        for (int g = 0; g < groups; ++g) y += s_grp[(g * 2 * KB + k) * slots + r];
        s_part[k * L::kPart + rows[r]] = fmaf(a.wG, y, s_part[k * L::kPart + rows[r]]);
    }
}

template <int M, int KB>
__global__ void __launch_bounds__(kH3Threads, 1) detect_h3_kernel(const __grid_constant__ TcArgs a) {
    using L = H3Smem<M, KB>;
    constexpr int kSums = h3_sums(M, KB), kHalves = kSums == 4 ? 2 : 1;
    constexpr int kAcc = 4 / kSums;                // accumulator stages
    constexpr int kStageCols = 512 / kAcc, kNB = 2 * kH3Entries / kHalves;  // TMEM columns of one; MMA N
    constexpr int E = kH3Entries, P8 = M / 8;  // pieces of eight antennas per row
    static_assert(M % 16 == 0 && KB % 2 == 0, "whole MMA k-steps, users in pairs");
    extern __shared__ __align__(1024) unsigned char smem[];
    float *sC = reinterpret_cast<float *>(smem + L::kC);
    float2 *sH = reinterpret_cast<float2 *>(smem + L::kH);
    float *s_nq = reinterpret_cast<float *>(smem + L::kN);
    float *s_part = reinterpret_cast<float *>(smem);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::kBar);
    uint64_t *full = bars, *a_ready = bars + 2, *mma_done = bars + 3, *epi_done = mma_done + 4 * kHalves;  // [2], [1], [4][halves] x 2
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L::kTmem);
    uint32_t *s_mask = reinterpret_cast<uint32_t *>(smem + L::kMask);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int split = (int)cluster_size(), rank = (int)cluster_rank();
    const int q0 = (int)(blockIdx.x / split) * kH3Rows;
    int n_ent = a.n_entries;
    if (a.meta) n_ent = min(n_ent, max(__ldg(a.meta), 0));
    const int NT = (n_ent + E - 1) / E;
    const int t_lo = (int)((long long)rank * NT / split), J = (int)((long long)(rank + 1) * NT / split) - t_lo;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) mbar_init(&full[i], kH3Conv);
        for (int i = 0; i < 4 * kHalves; ++i) {
            mbar_init(&mma_done[i], 1 + kH3Conv);
            mbar_init(&epi_done[i], kH3Epi / kHalves);
        }
        mbar_init(a_ready, kH3Epi);
        fence_mbar_init();
        for (int i = 0; i < 8; ++i) s_mask[i] = 0;
    }
    // ---- squared norms of the queries, eight loads in flight per lane (warp w: rows 32 w ..)
    bool in_rng = true;
    if (warp < 8) {
        constexpr int LR = M / 2, RL = 32 / LR;  // lanes per row, rows per load
#pragma unroll 1
        for (int r0 = 0; r0 < 32; r0 += 8 * RL) {
            float4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = 32 * warp + r0 + RL * i + lane / LR;
                v[i] = q0 + r < a.N ? __ldg(reinterpret_cast<const float4 *>(a.rx + (size_t)(q0 + r) * M) + lane % LR)
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float n = fmaf(v[i].x, v[i].x, fmaf(v[i].y, v[i].y, fmaf(v[i].z, v[i].z, v[i].w * v[i].w)));
#pragma unroll
                for (int o = LR / 2; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
                if (lane % LR == 0) s_nq[32 * warp + r0 + RL * i + lane / LR] = n;
                in_rng = in_rng && a.k2 * n <= kFactorLimit;
            }
        }
    }
    tc_fence_before();
    const bool in_range = __syncthreads_and(in_rng);  // (also: norms, barriers and the TMEM address are visible)
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    bool ok = true;

    if (warp >= 8 && warp < 11) {
        // ================= converters =================
        // one task = eight antennas of one entry: both operand rows.  Of eight consecutive lanes four
        // take one piece and four the next; each stores row 2e + f first, f its piece's parity, so that
        // the eight 16-byte stores of a quarter-warp hit eight different rows of a k-column group.
        const int ct = tid - kH3Epi;
        constexpr int kTaskN = E * P8, kTasks = (kTaskN + kH3Conv - 1) / kH3Conv;
        auto task = [](int i, int &e, int &p, int &f) {
            f = i & 1;
            e = (i >> 1 & 3) | (i / (8 * (P8 / 2))) << 2;
            p = (i >> 3) % (P8 / 2) * 2 + f;
        };
        auto put = [&](int sb, int e, int p, int f, const float (&re)[8], const float (&im)[8]) {
            uint4 rh, rl, ih, il;
            h3_split8(re, rh, rl);
            h3_split8(im, ih, il);
            const uint32_t sg = 0x80008000u;
            const uint4 nh = make_uint4(ih.x ^ sg, ih.y ^ sg, ih.z ^ sg, ih.w ^ sg);
            const uint4 nl = make_uint4(il.x ^ sg, il.y ^ sg, il.z ^ sg, il.w ^ sg);
            unsigned char *base = smem + L::kB + sb * 2 * L::kBCopy;
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const int form = f ^ o, r = 2 * e + form;  // form 0: [Re; Im], 1: [-Im; Re]
                unsigned char *dst = base + (r >> 3) * L::SBO + (r & 7) * 16;
                *reinterpret_cast<uint4 *>(dst + p * 128) = form ? nh : rh;
                *reinterpret_cast<uint4 *>(dst + (P8 + p) * 128) = form ? rh : ih;
                *reinterpret_cast<uint4 *>(dst + L::kBCopy + p * 128) = form ? nl : rl;
                *reinterpret_cast<uint4 *>(dst + L::kBCopy + (P8 + p) * 128) = form ? rl : il;
            }
        };
        for (int j = 0; j < J; ++j) {
            const int e0 = (t_lo + j) * E, sb = j & 1, sc = j & 3;
            float4 v[kTasks][4];
            float n_row[kTasks];
            constexpr int kCoef = (E * 2 * KB + kH3Conv - 1) / kH3Conv;
            float cf[kCoef];
#pragma unroll
            for (int q = 0; q < kTasks; ++q) {
                int e, p, f;
                task(min(ct + kH3Conv * q, kTaskN - 1), e, p, f);
                const int t = e0 + e;
                n_row[q] = t < n_ent ? __ldg(a.dict_norm + t) : 0.f;
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    v[q][c] = t < n_ent ? __ldg(reinterpret_cast<const float4 *>(a.dict + (size_t)t * M + p * 8) + c)
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int q = 0; q < kCoef; ++q) {
                const int i = ct + kH3Conv * q, t = e0 + i / (2 * KB), l = i / KB % 2, k = i % KB;
                cf[q] = i < E * 2 * KB && t < n_ent && k < a.K ? __ldg(a.gamma + ((size_t)t * 2 + l) * a.K + k) : 0.f;
            }
            const float n_t = ct < E && e0 + ct < n_ent ? __ldg(a.dict_norm + e0 + ct) : 0.f;
            // the entry stage is free when the MMAs of tile j-2 are done, the coefficient stage when the
            // epilogue of tile j-4 is
#pragma unroll
            for (int h = 0; h < kHalves; ++h)
                if ((j >= 2 && !mbar_wait_sleepy(&mma_done[((j - 2) & 3) * kHalves + h], ((j - 2) >> 2) & 1)) ||
                    (j >= 4 && !mbar_wait_sleepy(&epi_done[sc * kHalves + h], ((j - 4) >> 2) & 1)))
                    ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
#pragma unroll
            for (int q = 0; q < kTasks; ++q) {
                int e, p, f;
                task(min(ct + kH3Conv * q, kTaskN - 1), e, p, f);
                float inv, re[8], im[8];
                const float s = h3_scale(n_row[q], inv);
                if (s == 0.f) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[q][c] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                h3_unpack(v[q], s, re, im);
                if (ct + kH3Conv * q < kTaskN) put(sb, e, p, f, re, im);
            }
#pragma unroll
            for (int q = 0; q < kCoef; ++q) {
                const int i = ct + kH3Conv * q;
                if (i < E * 2 * KB) sC[sc * E * 2 * KB + i] = cf[q];
            }
            if (ct < E) {
                float inv;
                h3_scale(n_t, inv);
                sH[sc * E + ct] = make_float2(inv, e0 + ct < n_ent ? -a.k2 * n_t : -INFINITY);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&full[sb]);
#pragma unroll
            for (int h = 0; h < kHalves; ++h)  // releases this thread's coefficients and norms to the epilogue
                mbar_arrive(&mma_done[sc * kHalves + h]);
        }
    } else if (warp == 11) {
        // ================= MMA issue =================
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(kNB >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);  // FP16, FP32 sums
            const uint32_t a0 = smem_u32(smem + L::kA);
            int committed = -1;
            if (J > 0 && !mbar_wait_bounded(a_ready, 0)) ok = false;
            for (int j = 0; j < J && ok; ++j) {
                if (!mbar_wait_bounded(&full[j & 1], (j >> 1) & 1)) {
                    ok = false;
                    break;
                }
#pragma unroll
                for (int h = 0; h < kHalves; ++h) {
                    if (j >= kAcc && !mbar_wait_bounded(&epi_done[((j - kAcc) & 3) * kHalves + h], ((j - kAcc) >> 2) & 1)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t b0 = smem_u32(smem + L::kB + (j & 1) * 2 * L::kBCopy) + h * (kNB / 8) * L::SBO;
                    const uint32_t d0 = tmem + (uint32_t)(j % kAcc * kStageCols + h * (kStageCols / kHalves));
                    // the small products first, into the first sum: only hi times hi adds at the size of the result
#pragma unroll
                    for (int part = 0; part < 3; ++part) {
#pragma unroll
                        for (int ks = 0; ks < 2 * M / 16; ++ks) {
                            const uint64_t bd = umma_sdesc(b0 + (part == 1 ? L::kBCopy : 0) + ks * 256, L::SBO);
                            constexpr int kPer = 2 * M / 16 / kSums;  // k-steps of hi times hi per sum
                            const int sum = part == 2 ? ks / kPer : 0;
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const uint64_t ad = umma_sdesc(a0 + (q * 2 + (part == 0 ? 1 : 0)) * L::kACopy + ks * 256, L::SBO);
                                umma_f16(d0 + (2 * sum + q) * kNB, ad, bd, idesc, sum > 0 ? ks % kPer > 0 : part > 0 || ks > 0);
                            }
                        }
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     smem_u32(&mma_done[(j & 3) * kHalves + h]))
                                 : "memory");
                    committed = j * kHalves + h;
                }
            }
            if (committed >= 0) {  // (of the last tile's halves the one committed last)
                const int j = committed / kHalves;
                mbar_wait_bounded(&mma_done[(j & 3) * kHalves + committed % kHalves], (j >> 2) & 1);
            }
        }
        __syncwarp();
    } else {
        // ================= epilogue =================
        // ---- this warp's 32 query rows as scaled hi and lo copies, by pieces of eight antennas (eight
        // consecutive lanes write eight consecutive rows of one k-column)
        constexpr int kBatch = P8 < 4 ? P8 : 4;
#pragma unroll 1
        for (int i0 = 0; i0 < 32 * P8; i0 += 32 * kBatch) {  // up to sixteen loads in flight per lane
            float4 va[kBatch][4];
#pragma unroll
            for (int n = 0; n < kBatch; ++n) {
                const int i = i0 + 32 * n + lane, r = 32 * warp + ((i & 7) | (i / (8 * P8) << 3)), p = (i >> 3) % P8;
                const bool ok = q0 + r < a.N && fabsf(s_nq[r]) < INFINITY;  // (zeros where the norm is not finite)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    va[n][q] = ok ? __ldg(reinterpret_cast<const float4 *>(a.rx + (size_t)(q0 + r) * M + p * 8) + q)
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int n = 0; n < kBatch; ++n) {
                const int i = i0 + 32 * n + lane, r = 32 * warp + ((i & 7) | (i / (8 * P8) << 3)), p = (i >> 3) % P8;
                float inv;
                const float s = h3_scale(s_nq[r], inv);
                float re[8], im[8];
                h3_unpack(va[n], s, re, im);
                unsigned char *dst = smem + L::kA + (r >> 7) * 2 * L::kACopy + ((r & 127) >> 3) * L::SBO + (r & 7) * 16;
                uint4 hi, lo;
                h3_split8(re, hi, lo);
                *reinterpret_cast<uint4 *>(dst + p * 128) = hi;
                *reinterpret_cast<uint4 *>(dst + L::kACopy + p * 128) = lo;
                h3_split8(im, hi, lo);
                *reinterpret_cast<uint4 *>(dst + (P8 + p) * 128) = hi;
                *reinterpret_cast<uint4 *>(dst + L::kACopy + (P8 + p) * 128) = lo;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(a_ready);

        const int row = tid & 127, hf = tid >> 7;  // query rows row and 128 + row, entry half
        const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
        float gq[2];  // 2 k2 / query scale
        float acc1[2][KB], acc2[2][KB];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            h3_scale(s_nq[row + 128 * i], gq[i]);
            gq[i] *= 2.f * a.k2;
#pragma unroll
            for (int k = 0; k < KB; ++k) acc1[i][k] = acc2[i][k] = 0.f;
        }
        // kGuard: a CTA with a query outside the factor range: -k2 n_s goes inside the exponent, and a row
        // outside it whose terms the Gram's error reaches (H3Guard) is marked
        auto run_tiles = [&](auto guard_c) {
            constexpr bool kGuard = decltype(guard_c)::value;
            float hq[2];  // -k2 n_s
            H3Guard guard[2];
            bool mark[2] = {false, false};
            if constexpr (kGuard) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    hq[i] = -a.k2 * s_nq[row + 128 * i];
                    guard[i] = h3_guard(-hq[i]);
                }
            }
            for (int j = 0; j < J; ++j) {
                const int s = j & 3;
                const int bar = s * kHalves + (kHalves > 1 ? hf : 0);
                if (!__all_sync(0xffffffffu, mbar_wait_bounded(&mma_done[bar], (j >> 2) & 1))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const float *g = sC + (s * E + 16 * hf) * 2 * KB;
                const float2 *hh = sH + s * E + 16 * hf;
                const uint32_t col =
                    tmem + lane_base + (uint32_t)(j % kAcc * kStageCols + (kHalves > 1 ? hf * (kStageCols / 2) : 32 * hf));
                uint32_t v[kSums][2][8];  // [sum][query tile]
                auto load = [&](int c) {
#pragma unroll
                    for (int w = 0; w < kSums; ++w)
#pragma unroll
                        for (int q = 0; q < 2; ++q) h3_tmem_ld8(col + (2 * w + q) * kNB + 8 * c, v[w][q]);
                };
                load(0);
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {  // four entries of both rows; the next four's accumulators follow
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    float x[2][8];
#pragma unroll
                    for (int q = 0; q < 2; ++q)
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            auto val = [&](int w) { return __uint_as_float(v[w < kSums ? w : 0][q][i]); };
                            x[q][i] = kSums == 4 ? (val(0) + val(1)) + (val(2) + val(3)) : kSums == 2 ? val(0) + val(1) : val(0);
                        }
                    if (c < 3) load(c + 1);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 mh = hh[4 * c + e];
                        float g1[KB], gg[KB];
                        load_coef<KB>(g + (4 * c + e) * 2 * KB, g1, gg);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const float re = x[i][2 * e], im = x[i][2 * e + 1];
                            const float m = gq[i] * mh.x;
                            const float h = kGuard ? mh.y + hq[i] : mh.y;
                            const float eA = ex2(fmaf(m, re, h)), eB = ex2(fmaf(m, im, h)), eC = ex2(fmaf(-m, im, h));
                            if constexpr (kGuard) mark[i] |= m * fmaxf(re, fabsf(im)) > fmaf(guard[i].b1, h, guard[i].a);
#pragma unroll
                            for (int k = 0; k < KB; k += 2) {
                                fma2_pair(acc1[i][k], acc1[i][k + 1], gg[k], gg[k + 1], eC);
                                fma2_pair(acc1[i][k], acc1[i][k + 1], g1[k], g1[k + 1], eA);
                                fma2_pair(acc2[i][k], acc2[i][k + 1], gg[k], gg[k + 1], eA);
                                fma2_pair(acc2[i][k], acc2[i][k + 1], g1[k], g1[k + 1], eB);
                            }
                        }
                    }
                }
                tc_fence_before();
                mbar_arrive(&epi_done[bar]);
            }
            if constexpr (kGuard) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (mark[i]) atomicOr(s_mask + (row + 128 * i) / 32, 1u << (row & 31));
            }
        };
        if (in_range) run_tiles(std::false_type{});
        else run_tiles(std::true_type{});
        // every MMA of this CTA is done (the last tile's wait above): the coefficient stages take the
        // filter as [antenna][Re, Im][user], the operands' space the sums
        // this CTA's share of the antennas, in pieces of kLin: eight, whose short sums lose the least, but all at
        // once with as many users as antennas, where the filter's terms are large and cancel, and a part of
        // their sum added to the kernel sums costs bits (16 antennas and users, error of the outputs: 300 entries
        // 2.59e-7 in two pieces, 2.36e-7 in one, 2.31e-7 in the TMA-staged form; 1500: 2.68e-7, 2.37e-7, 2.43e-7)
        constexpr int kLin = M == 16 && KB == 16 ? 16 : 8, kPieces = M / kLin;
        const int p_lo = rank * kPieces / split, p_hi = (rank + 1) * kPieces / split;
        // query factor (inside the exponent already in the guarded form) and weight; a marked row keeps
        // nothing of the Gram
        if (in_range) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float f = a.wG * ex2(-a.k2 * s_nq[row + 128 * i]);
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    acc1[i][k] *= f;
                    acc2[i][k] *= f;
                }
            }
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");  // (the halves' marks are complete)
        if (!in_range) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const bool keep = !(s_mask[(row + 128 * i) / 32] >> (row & 31) & 1);
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    acc1[i][k] = keep ? acc1[i][k] * a.wG : 0.f;
                    acc2[i][k] = keep ? acc2[i][k] * a.wG : 0.f;
                }
            }
        }
        for (int i = tid; i < kLin * (p_hi - p_lo) * KB; i += kH3Epi) {
            const int m = i / KB, k = i % KB;
            const float2 c = k < a.K ? __ldg(a.clin + (size_t)(kLin * p_lo + m) * a.K + k) : make_float2(0.f, 0.f);
            sC[2 * m * KB + k] = c.x;
            sC[(2 * m + 1) * KB + k] = c.y;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        // linear part w_L c_k^H r of query row tid (= this thread's row of query tile hf), in FP32: the
        // MMA's sums are not exact enough for it
        const float2 *rq = a.rx + (size_t)min(q0 + tid, a.N - 1) * M;
#pragma unroll 1
        for (int p = p_lo; p < p_hi; ++p) {
            float4 v[kLin / 2];
#pragma unroll
            for (int c = 0; c < kLin / 2; ++c) v[c] = __ldg(reinterpret_cast<const float4 *>(rq + kLin * p) + c);
            float l1[KB], l2[KB];  // a piece's sums, then added
#pragma unroll
            for (int k = 0; k < KB; ++k) l1[k] = l2[k] = 0.f;
#pragma unroll
            for (int m = 0; m < kLin; ++m) {
                const float x = m & 1 ? v[m >> 1].z : v[m >> 1].x, y = m & 1 ? v[m >> 1].w : v[m >> 1].y;
                const float *cx = sC + 2 * (kLin * (p - p_lo) + m) * KB, *cy = cx + KB;
#pragma unroll
                for (int k = 0; k < KB; k += 2) {
                    const float2 u = *reinterpret_cast<const float2 *>(cx + k), w = *reinterpret_cast<const float2 *>(cy + k);
                    fma2_pair(l1[k], l1[k + 1], u.x, u.y, x);
                    fma2_pair(l1[k], l1[k + 1], w.x, w.y, y);
                    fma2_pair(l2[k], l2[k + 1], u.x, u.y, y);
                    fma2_pair(l2[k], l2[k + 1], w.x, w.y, -x);
                }
            }
#pragma unroll
            for (int k = 0; k < KB; ++k) {
                acc1[0][k] = hf == 0 ? fmaf(a.wL, l1[k], acc1[0][k]) : acc1[0][k];
                acc2[0][k] = hf == 0 ? fmaf(a.wL, l2[k], acc2[0][k]) : acc2[0][k];
                acc1[1][k] = hf == 1 ? fmaf(a.wL, l1[k], acc1[1][k]) : acc1[1][k];
                acc2[1][k] = hf == 1 ? fmaf(a.wL, l2[k], acc2[1][k]) : acc2[1][k];
            }
        }
        // the halves meet: each leaves one row's sums to the other and adds the other's to its own row
        // (first half's terms first)
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            s_part[k * L::kPart + row + 128 * (1 - hf)] = hf == 0 ? acc1[1][k] : acc1[0][k];
            s_part[(KB + k) * L::kPart + row + 128 * (1 - hf)] = hf == 0 ? acc2[1][k] : acc2[0][k];
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            const float o1 = s_part[k * L::kPart + tid], o2 = s_part[(KB + k) * L::kPart + tid];
            s_part[k * L::kPart + tid] = hf == 0 ? acc1[0][k] + o1 : o1 + acc1[1][k];
            s_part[(KB + k) * L::kPart + tid] = hf == 0 ? acc2[0][k] + o2 : o2 + acc2[1][k];
        }
    }
    if (!in_range) h3_direct_rows<M, KB>(a, smem, s_mask, reinterpret_cast<int *>(s_tmem + 1), q0, t_lo, J, n_ent);
    if (!ok && lane == 0) report(a.status, APSM_ERR_TIMEOUT);
    __syncwarp();
    cluster_sync_all();  // every part of the cluster's query tile is in shared memory
    // ---- outputs: this CTA's share of the rows, parts in CTA order
    const int r_lo = rank * kH3Rows / split, r_hi = (rank + 1) * kH3Rows / split;
    const uint32_t part0 = smem_u32(s_part);
    for (int i = tid; i < (r_hi - r_lo) * a.K; i += kH3Threads) {
        const int r = r_lo + i / a.K, k = i % a.K, s = q0 + r;
        if (s >= a.N) break;
        float v1[kH3MaxSplit], v2[kH3MaxSplit], y1 = 0.f, y2 = 0.f;
#pragma unroll
        for (int c = 0; c < kH3MaxSplit; ++c) {
            v1[c] = c < split ? ld_cluster(part0 + (k * L::kPart + r) * 4, c) : 0.f;
            v2[c] = c < split ? ld_cluster(part0 + ((KB + k) * L::kPart + r) * 4, c) : 0.f;
        }
#pragma unroll
        for (int c = 0; c < kH3MaxSplit; ++c) {
            y1 += v1[c];
            y2 += v2[c];
        }
        a.soft[(size_t)s * a.K + k] = make_float2(y1, y2);
        if (a.hard) a.hard[(size_t)s * a.K + k] = (uint8_t)((y1 < 0.f ? 1 : 0) | (y2 < 0.f ? 2 : 0));
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();  // nobody reads this CTA's sums any more
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// How `nq` query tiles of `nt` entry tiles each are launched: `full` of them first, one CTA each in
// whole waves, then the rest with `split` CTAs per tile, whichever costs the least in entry tiles per
// SM (a CTA's set-up and merge count as kSetup of them; `resident` [s] clusters of s CTAs fit the GPU
// at a time).  The time of a full wave puts the set-up at 6 to 10 tiles at 16 antennas and 6 users, more
// than kSetup; but of 99 sizes timed with 3 and with 8 (16, 32 and 64 antennas, 2 to 16 users, 300 to 4096
// entries, 300 to 100003 vectors) 90 take the same time, and of the other nine five are faster with 3 (by
// up to 4 %: 16 antennas, 6 users, 4096 entries, 20000 vectors 155 and 161 us) and four with 8 (64, 4, 2048,
// 20000: 117 and 112).
struct H3Plan {
    int full, split;
};
inline H3Plan h3_plan(int nq, int nt, const int *resident) {
    constexpr int kSetup = 3;
    H3Plan best{0, 1};
    long long cost = -1;
    const int whole = resident[1] > 0 ? nq / resident[1] * resident[1] : 0;
    for (int full : {0, whole}) {
        const long long first = full > 0 ? (long long)(full / resident[1]) * (nt + kSetup) : 0;
        for (int s = 1; s <= kH3MaxSplit && s <= std::max(nt, 1); ++s) {
            if (resident[s] < 1) continue;
            const long long waves = (nq - full + resident[s] - 1) / resident[s];
            const long long c = first + waves * ((nt + s - 1) / s + kSetup) + (full > 0 && nq > full ? 1 : 0);
            if (cost < 0 || c < cost) {
                cost = c;
                best = H3Plan{full, s};
            }
        }
    }
    return best;
}

template <int M, int KB>
cudaError_t launch_detect_h3(const TcArgs &a, int *launches, cudaStream_t stream) {
    using L = H3Smem<M, KB>;
    auto fn = detect_h3_kernel<M, KB>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kLaunch);
    if (e != cudaSuccess) return e;
    const int nq = (a.N + kH3Rows - 1) / kH3Rows, nt = (a.n_entries + kH3Entries - 1) / kH3Entries;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kH3Threads);
    cfg.dynamicSmemBytes = L::kLaunch;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // clusters of each size that fit the device at a time (one query per device and kernel)
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    static std::atomic<int> cached[kH3Devices][kH3MaxSplit + 1];
    int resident[kH3MaxSplit + 1] = {};
    for (int s = 1; s <= kH3MaxSplit; ++s) {
        int n = dev < kH3Devices ? cached[dev][s].load(std::memory_order_relaxed) : 0;
        if (n == 0) {
            attr[0].val.clusterDim.x = s;
            cfg.gridDim = dim3(s);
            if ((e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg)) != cudaSuccess) return e;
            n = n > 0 ? n : -1;
            if (dev < kH3Devices) cached[dev][s].store(n, std::memory_order_relaxed);
        }
        resident[s] = n;
    }
    // ordinary launches otherwise: every read may take the L1 path (see launch_detect_tc)
    const H3Plan plan = h3_plan(nq, nt, resident);
    auto run = [&](int tile0, int tiles, int split) {
        TcArgs b = a;
        const size_t s0 = (size_t)tile0 * kH3Rows;
        b.rx += s0 * M;
        b.soft += s0 * a.K;
        if (b.hard) b.hard += s0 * a.K;
        b.N = (int)std::min<size_t>((size_t)a.N - s0, (size_t)tiles * kH3Rows);
        attr[0].val.clusterDim.x = split;
        cfg.gridDim = dim3((unsigned)tiles * split);
        return cudaLaunchKernelEx(&cfg, fn, b);
    };
    if (plan.full > 0 && (e = run(0, plan.full, 1)) != cudaSuccess) return e;
    if (nq > plan.full && (e = run(plan.full, nq - plan.full, plan.split)) != cudaSuccess) return e;
    *launches = (plan.full > 0) + (nq > plan.full);
    return cudaGetLastError();
}

using H3Launcher = cudaError_t (*)(const TcArgs &, int *, cudaStream_t);

}  // namespace apsm
