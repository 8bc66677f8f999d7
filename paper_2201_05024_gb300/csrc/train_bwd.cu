// train_bwd.cu -- adjoint of the APSM training recurrence (apsm_train_backward).
//
// Forward (Eq. apsm with Eq. beta over the window J_n, Sec. II-D), per user, state
// S_n = (w, gamma_i for every centre):
//   y_j = w_L <w, x_j> + w_G sum_{i alive at n} gamma_i kappa_G(x_i, x_j),  e_j = y_j - b_j,
//   kappa_jj = w_L ||x_j||^2 + w_G,  beta_j = (-e_j - s_j eps) / kappa_jj for s_j = +1 (e < -eps)
//   or -1 (e > eps), beta_j = 0 inside the slab;
//   S_{n+1} = S_n + sum_{j in J_n} a_j (unit vector of centre j, x_j),  a_j = mu q beta_j.
// Reverse mode, with (gbar, wbar) the adjoint of S_{n+1}:
//   abar_j = gbar_j + <wbar, x_j>;  mubar += q beta_j abar_j;  betabar_j = mu q abar_j;
//   outside the slab: ybar_j = -betabar_j / kappa_jj, epsbar += -s_j betabar_j / kappa_jj,
//   w_Lbar += (-betabar_j beta_j / kappa_jj) (||x_j||^2 - 1);
//   then wbar += ybar_j w_L x_j, w_Lbar += ybar_j (<w, x_j> - gauss_j),
//   sigmabar += ybar_j w_G sum_i gamma_i kappa_G(x_i, x_j) d_ij^2 / sigma^3,
//   gbar_i += ybar_j w_G kappa_G(x_i, x_j) for every alive centre i.
// Inside the slab the derivative is taken as 0 (also at |e| = eps exactly).
//
// Cost per step O(W^2 + S) instead of O(W S):
//  * forward: the predictions of the window samples are carried from step to step (the W
//    projections of a step change them by sum_o a_o kappa(x_{j_o}, x_j); an evicted centre's
//    contribution is subtracted), and a sample's prediction is formed once, on arrival, from the
//    live centres; every step's tape (beta, branch, kappa, <w, x_j>, gauss_j, its sigma weight)
//    goes to the workspace, so nothing is re-run;
//  * reverse: gbar_i is read only while centre i is in the window.  R_j, the sum of the cg terms
//    of sample j over the steps swept so far, gives centre i's adjoint when it enters the window
//    from below: gbar_i = final_i + sum_j R_j kappa_G(x_i, x_j) over the steps in which i is
//    alive (for a centre evicted during the call, R at the eviction step is kept and subtracted);
//    from then on it is pushed the W terms of each step like the forward predictions.
// Kernel values between samples come from tables built once per call.  One CTA of 4 warps per
// user: the threads split the O(S) sums of an arrival, a thread per window slot for the scalar
// terms (summed in slot order at the end), a thread per component or window sample for the
// O(W) updates.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "apsm_common.cuh"
#include "train_f32.cuh"

namespace apsm {

extern std::atomic<long long> g_launches;  // apsm_api.cu

struct Tape {  // one window slot of one step
    float beta, s, kappa, dotw, gauss, gd2;
};

struct TrainBwdArgs {
    int M, K, W, D, P;
    int Sp;                 // row stride of the tables: 2P rounded up to a multiple of 4
    float sigma, mu, eps, wL, wG, k2;
    const float2 *rx;       // [P][M]
    const float2 *sym;      // [P][K]
    const float2 *clin0;    // [M][K] or null
    const float *dgamma;    // [A][2][K] adjoint of the final coefficients (ring layout)
    const float2 *dclin;    // [M][K] adjoint of the final linear filter
    float *ltab;            // [2P][Sp] x_i . x_j
    float *gtab;            // [2P][Sp] kappa_G(x_i, x_j)
    float *gdtab;           // [2P][Sp] kappa_G(x_i, x_j) ||x_i - x_j||^2
    Tape *tape;             // [K][2P][W]
    float *snap;            // [K][P - D][W] R at the eviction steps (P > D only)
    float *scal;            // [K][4] per-user sigma, mu, eps, w_L adjoints
    float2 *dclin0;         // [M][K] out
    float *dscalars;        // [4] out
    // instance i of a batch: the pointers above advanced by i times these (elements; ws_stride in
    // bytes for the workspace regions ltab, gtab, gdtab, tape, snap, scal)
    size_t st_rx, st_sym, st_clin0, st_dgamma, st_mk, ws_stride;
    int mode;  // 1: tables' forward pass (tape), 2: reverse sweep, 3: both
};

// The arguments of instance i (blockIdx.y of every launch below).
__device__ __forceinline__ TrainBwdArgs for_instance(const TrainBwdArgs &a0, int i) {
    TrainBwdArgs a = a0;
    auto adv = [&](auto *ptr) {
        return reinterpret_cast<decltype(ptr)>(reinterpret_cast<unsigned char *>(ptr) + i * a0.ws_stride);
    };
    a.rx += i * a.st_rx;
    a.sym += i * a.st_sym;
    if (a.clin0) a.clin0 += i * a.st_clin0;
    a.dgamma += i * a.st_dgamma;
    a.dclin += i * a.st_mk;
    a.dclin0 += i * a.st_mk;
    a.dscalars += 4 * (size_t)i;
    a.ltab = adv(a.ltab);
    a.gtab = adv(a.gtab);
    a.gdtab = adv(a.gdtab);
    a.tape = adv(a.tape);
    a.snap = adv(a.snap);
    a.scal = adv(a.scal);
    return a;
}

__global__ void train_bwd_tables_kernel(const TrainBwdArgs a0) {
    const TrainBwdArgs a = for_instance(a0, blockIdx.y);
    const int S = 2 * a.P, Sp = a.Sp;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)S * Sp;
         idx += (long long)gridDim.x * blockDim.x) {
        const int i0 = (int)(idx / Sp), j0 = (int)(idx % Sp);
        if (j0 >= S) {  // row padding
            a.ltab[idx] = 0.f;
            a.gtab[idx] = 0.f;
            a.gdtab[idx] = 0.f;
            continue;
        }
        const int i = min(i0, j0), j = max(i0, j0);  // both halves from one ordering: exactly symmetric
        float dot, d2;
        sample_pair(a.rx + (size_t)(i >> 1) * a.M, a.rx + (size_t)(j >> 1) * a.M, a.M, i & 1, j & 1, dot, d2);
        const float g = ex2(-a.k2 * d2);
        a.ltab[idx] = dot;
        a.gtab[idx] = g;
        a.gdtab[idx] = g * d2;
    }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// component m of the real-split sample j (Sec. II-D): x_{2t} = [Re r; Im r], x_{2t+1} = [Im r; -Re r]
__device__ __forceinline__ float xcomp(const float2 *rx, int M, int j, int m) {
    const float2 *r = rx + (size_t)(j >> 1) * M;
    if (m < M) {
        const float2 v = __ldg(r + m);
        return (j & 1) ? v.y : v.x;
    }
    const float2 v = __ldg(r + (m - M));
    return (j & 1) ? -v.x : v.y;
}

// Slot of a sample in a ring of R slots from the slot b of a reference sample below it and the
// offset off in [0, 3R] between the two (no integer division on the per-step path).
__device__ __forceinline__ int ring_slot(int b, int off, int R) {
    int x = b + off;
    x -= x >= R ? R : 0;
    x -= x >= R ? R : 0;
    x -= x >= R ? R : 0;
    return x;
}

// Loads issued a step ahead of their use: predicated rather than followed by a select, so that no
// instruction waits on the data before it is used; volatile, so that they stay ahead of the barriers.
// (the predicate is set inside the asm, so no branch surrounds the load)
__device__ __forceinline__ float ldg_if(bool c, const float *p) {  // read-only data of earlier kernels
    float v = 0.f;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q ld.global.nc.f32 %0, [%1];\n\t}"
                 : "+f"(v)
                 : "l"(p), "r"((int)c));
    return v;
}
__device__ __forceinline__ float2 ld2_if(bool c, const float *p) {  // data this kernel wrote; 8-byte aligned
    float2 v = make_float2(0.f, 0.f);
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\t@q ld.global.v2.f32 {%0, %1}, [%2];\n\t}"
                 : "+f"(v.x), "+f"(v.y)
                 : "l"(p), "r"((int)c)
                 : "memory");
    return v;
}

constexpr int kBwdThreads = 128;  // 4 warps per user
constexpr int kPf = 4;            // entries of the next O(S) row a thread fetches a step ahead, per table

// Entries lo + tid + q * kBwdThreads (q < kPf, below hi) of one or two table rows, a step early.
struct RowPf {
    float g[kPf], d[kPf];
};

__device__ __forceinline__ void row_fetch(RowPf &f, const float *grow, const float *drow, int lo, int hi) {
#pragma unroll
    for (int q = 0; q < kPf; ++q) {
        const int i = lo + (int)threadIdx.x + q * kBwdThreads;
        f.g[q] = ldg_if(i < hi, grow + i);
        f.d[q] = ldg_if(drow != nullptr && i < hi, drow + i);
    }
}

// The band of row r that the window needs: entries s0 + t, t = 0..W (thread t holds one, thread 0
// also t = W when W = kBwdThreads), inside [0, S).  Stored into the window rings kg, kd, kl
// [(W+1)^2] (sample j in slot j mod (W+1)) at both (r, j) and (j, r): the tables are exactly
// symmetric.
struct BandPf {
    float g[2], d[2], l[2];
};

__device__ __forceinline__ void band_fetch(BandPf &b, const TrainBwdArgs &a, int S, int W, int r, int s0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int t = (int)threadIdx.x + q * kBwdThreads, j = s0 + t;
        const bool ok = r >= 0 && r < S && t <= W && j >= 0 && j < S;
        const size_t x = ok ? (size_t)r * a.Sp + j : 0;
        b.g[q] = ldg_if(ok, a.gtab + x);
        b.d[q] = ldg_if(ok, a.gdtab + x);
        b.l[q] = ldg_if(ok, a.ltab + x);
    }
}

// (sr, s0r: the ring slots of r and s0)
__device__ __forceinline__ void band_store(const BandPf &b, float *kg, float *kd, float *kl, int S, int W, int r,
                                           int s0, int sr, int s0r) {
    const int WR = W + 1;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int t = (int)threadIdx.x + q * kBwdThreads, j = s0 + t;
        if (r >= 0 && r < S && t <= W && j >= 0 && j < S) {
            const int sj = ring_slot(s0r, t, WR);
            const int u = sr * WR + sj, v = sj * WR + sr;
            kg[u] = b.g[q];
            kg[v] = b.g[q];
            kd[u] = b.d[q];
            kd[v] = b.d[q];
            kl[u] = b.l[q];
            kl[v] = b.l[q];
        }
    }
}

// smem (floats): gamma (forward) / R (reverse) [2P], norms [2P], w / wbar [2M], window rings
// py, pd, pw [W] (forward: gauss_j, its sigma weight, <w, x_j>; reverse: py = abar_j), ca, cb [W],
// targets pb [W], warp partials [3 * 4], kg, kd, kl [(W+1)^2] (kappa_G, kappa_G d^2 and x_i . x_j
// among the samples of the window and the one entering or leaving it), xw [(W+1)][2M] (their
// components)
__global__ void __launch_bounds__(kBwdThreads, 6) train_bwd_kernel(const TrainBwdArgs a0) {
    extern __shared__ __align__(16) float sm[];
    const TrainBwdArgs a = for_instance(a0, blockIdx.y);
    constexpr int T = kBwdThreads, NW = T / 32;
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int M = a.M, K = a.K, W = a.W, D = a.D, P = a.P, S = 2 * P, L2 = 2 * M, WR = W + 1;
    float *gam = sm, *nrm = gam + S, *w = nrm + S, *py = w + L2, *pd = py + W, *pw = pd + W;
    float *ca = pw + W, *cb = ca + W, *pb = cb + W, *part = pb + W, *kg = part + 3 * NW, *kd = kg + WR * WR;
    float *kl = kd + WR * WR, *xw = kl + WR * WR;
    Tape *tape = a.tape + (size_t)k * S * W;
    float *snap = a.snap + (size_t)k * (P > D ? P - D : 0) * W;
    const float inv_s3 = 1.f / (a.sigma * a.sigma * a.sigma);
    const float mqW = a.mu / (float)W, qW = 1.f / (float)W;  // mu q and q of a full window
    // ring slots relative to the reference sample n - W - 1 of the current step: sW, sR are its
    // slots (mod W, mod W + 1), kept up to date as n moves (the samples used lie in [n - W - 1, n + 1])
    auto pmod = [](int x, int R) { return ((x % R) + R) % R; };
    int sW = 0, sR = 0;
    auto slotW = [&](int n, int j) { return ring_slot(sW, j - (n - W - 1), W); };
    auto slotR = [&](int n, int j) { return ring_slot(sR, j - (n - W - 1), WR); };

    auto first_centre = [&](int n) { return 2 * max(0, (n >> 1) - D + 1); };
    // centre i takes part in the steps n < evict_step(i) (its entry leaves at that step)
    auto evict_step = [&](int i) { return 2 * ((i >> 1) + D); };
    auto reduce3 = [&](float x, float y, float z) {  // per-warp partials, combined in warp order
        x = warp_sum(x);
        y = warp_sum(y);
        z = warp_sum(z);
        if (lane == 0) {
            part[3 * warp] = x;
            part[3 * warp + 1] = y;
            part[3 * warp + 2] = z;
        }
    };
    auto total = [&](int c) {
        float s = 0.f;
        for (int v = 0; v < NW; ++v) s += part[3 * v + c];
        return s;
    };
    // component tid of sample j as stored (x_{2t+1}'s upper half is the negated real part: xsign)
    auto xc = [&](int j) {
        const bool ok = tid < L2 && j >= 0 && j < S;
        const bool up = tid >= M, odd = j & 1;
        const int mm = up ? tid - M : tid, comp = up ? (odd ? 0 : 1) : (odd ? 1 : 0);
        return ldg_if(ok, reinterpret_cast<const float *>(a.rx + (ok ? (size_t)(j >> 1) * M + mm : 0)) + comp);
    };
    auto xsign = [&](int j, float v) { return (tid >= M && (j & 1)) ? -v : v; };
    // target b_j of user k (real part for even j, imaginary for odd)
    auto target_at = [&](bool ok, int j) {
        return ldg_if(ok, reinterpret_cast<const float *>(a.sym + (ok ? (size_t)(j >> 1) * K + k : 0)) + (j & 1));
    };

    for (int i = tid; i < S; i += T) {
        gam[i] = 0.f;
        nrm[i] = a.ltab[(size_t)i * a.Sp + i];  // ||x_i||^2
    }
    for (int m = tid; m < M; m += T) {
        const float2 c = a.clin0 ? a.clin0[m * K + k] : make_float2(0.f, 0.f);
        w[m] = c.x;  // w = [Re c; Im c]
        w[M + m] = c.y;
    }
    RowPf pf;
    BandPf bp;
    float xn = 0.f;
    if (a.mode & 1) {
        sW = pmod(-W - 1, W);
        sR = pmod(-W - 1, WR);
        band_fetch(bp, a, S, W, 0, -W);
        band_store(bp, kg, kd, kl, S, W, 0, -W, slotR(0, 0), slotR(0, -W));
        band_fetch(bp, a, S, W, 1, 1 - W);
        if (S > 1) row_fetch(pf, a.gtab + a.Sp, a.gdtab + a.Sp, first_centre(1), 1);
        if (tid < L2) xw[slotR(0, 0) * L2 + tid] = xcomp(a.rx, M, 0, tid);
        xn = xc(1);
        float bn = target_at(tid == T - 1 && S > 1, 1);  // the target of the next arrival, a step early
        if (tid == 0) pb[0] = target_at(true, 0);
        __syncthreads();

        // ---- forward: sample 0 arrives with no live centre --------------------------------------------
        reduce3(0.f, 0.f, tid < L2 ? w[tid] * xw[slotR(0, 0) * L2 + tid] : 0.f);
        __syncthreads();
        if (tid == 0) {
            py[0] = 0.f;
            pd[0] = 0.f;
            pw[0] = total(2);
        }
        __syncthreads();
        for (int n = 0; n < S; ++n, sW = ring_slot(sW, 1, W), sR = ring_slot(sR, 1, WR)) {
            const int jlo = max(0, n - W + 1), nJ = n - jlo + 1, jn = n + 1;
            const float mq = nJ == W ? mqW : a.mu / (float)nJ;
            const float b_jn = bn;
            if (warp == NW - 1) bn = target_at(tid == T - 1 && jn + 1 < S, jn + 1);
            // the next sample's prediction from the live centres, before this step's update
            if (jn < S) {
                if (tid <= W) {
                    band_store(bp, kg, kd, kl, S, W, jn, jn - W, slotR(n, jn), slotR(n, jn - W));
                    band_fetch(bp, a, S, W, jn + 1, jn + 1 - W);
                }
                float ws = 0.f;
                if (tid < L2) {
                    const float x = xsign(jn, xn);
                    xw[slotR(n, jn) * L2 + tid] = x;
                    ws = w[tid] * x;
                    xn = xc(jn + 1);
                }
                const int lo = first_centre(jn);
                const float *grow = a.gtab + (size_t)jn * a.Sp, *drow = a.gdtab + (size_t)jn * a.Sp;
                float ys = 0.f, ds = 0.f;
#pragma unroll
                for (int q = 0; q < kPf; ++q) {
                    const int i = lo + tid + q * T;
                    if (i < jn) {
                        ys = fmaf(gam[i], pf.g[q], ys);
                        ds = fmaf(gam[i], pf.d[q], ds);
                    }
                }
                for (int i = lo + tid + kPf * T; i < jn; i += T) {
                    ys = fmaf(gam[i], __ldg(grow + i), ys);
                    ds = fmaf(gam[i], __ldg(drow + i), ds);
                }
                reduce3(ys, ds, ws);
                if (jn + 1 < S)
                    row_fetch(pf, a.gtab + (size_t)(jn + 1) * a.Sp, a.gdtab + (size_t)(jn + 1) * a.Sp,
                              first_centre(jn + 1), jn + 1);
            }
            // the window's projections (Eq. beta), all from f_n
            if (tid < nJ) {
                const int j = jlo + tid, r = slotW(n, j);
                const float dw = pw[r], yg = py[r], gd = pd[r];
                const float y = fmaf(a.wL, dw, a.wG * yg);
                const float e = y - pb[r];
                const float kap = fmaf(a.wL, nrm[j], a.wG);
                float beta = 0.f, s = 0.f;
                if (kap != 0.f) {
                    if (e < -a.eps) { s = 1.f; beta = (-e - a.eps) / kap; }
                    else if (e > a.eps) { s = -1.f; beta = (-e + a.eps) / kap; }
                }
                tape[(size_t)n * W + tid] = Tape{beta, s, kap, dw, yg, gd};
                ca[tid] = mq * beta;
                cb[tid] = gam[j] + mq * beta;  // the coefficient after the step
            }
            __syncthreads();
            // Eq. apsm: coefficients, linear part, and the carried predictions of J_{n+1}.  With
            // 2D = W + 1 the oldest centre of J_n leaves before step n+1: the arrival jn takes no term
            // of it, and the other samples drop its coefficient after this step's update.
            if (tid < nJ) gam[jlo + tid] = cb[tid];
            if (tid == T - 1 && jn < S) pb[slotW(n, jn)] = b_jn;
            const int t_lo = max(0, n - W + 2), n_t = jn < S ? jn - t_lo + 1 : 0;
            const int e_lo = first_centre(n), e_hi = jn < S ? first_centre(jn) : e_lo;  // leave before step n+1
            const int s_lo = slotR(n, jlo);
            for (int u = tid; u < L2 + n_t; u += T) {
                if (u < L2) {
                    float acc = w[u];
                    int si = s_lo;
#pragma unroll 4
                    for (int o = 0; o < nJ; ++o, si = ring_slot(si, 1, WR)) acc = fmaf(ca[o], xw[si * L2 + u], acc);
                    w[u] = acc;
                } else {
                    const int j = t_lo + (u - L2), r = slotW(n, j), sj = slotR(n, j) * WR;
                    float ay, ad, aw;
                    if (j == jn) {
                        ay = total(0);
                        ad = total(1);
                        aw = total(2);
                    } else {
                        ay = py[r];
                        ad = pd[r];
                        aw = pw[r];
                    }
                    const int o_lo = j == jn ? max(0, e_hi - jlo) : 0;  // sources still live at jn
                    int si = s_lo;
#pragma unroll 4
                    for (int o = 0; o < nJ; ++o, si = ring_slot(si, 1, WR)) {
                        const float c = ca[o];
                        aw = fmaf(c, kl[sj + si], aw);
                        if (o >= o_lo) {
                            ay = fmaf(c, kg[sj + si], ay);
                            ad = fmaf(c, kd[sj + si], ad);
                        }
                    }
                    if (j != jn) {
                        const float *grow = a.gtab + (size_t)j * a.Sp, *drow = a.gdtab + (size_t)j * a.Sp;
                        for (int i = e_lo; i < e_hi; ++i) {  // centres leaving before step n+1
                            const float gi = i >= jlo ? cb[i - jlo] : gam[i];
                            ay = fmaf(-gi, __ldg(grow + i), ay);
                            ad = fmaf(-gi, __ldg(drow + i), ad);
                        }
                    }
                    py[r] = ay;
                    pd[r] = ad;
                    pw[r] = aw;
                }
            }
            __syncthreads();
        }

    }  // forward
    if (!(a.mode & 2)) return;

    // ---- reverse sweep: R = 0, wbar = dL/dw of the final state ------------------------------------
    __syncthreads();
    {  // kernel values and components of the last W + 1 samples (as the forward left them)
        const int j0 = max(0, S - W - 1), nr = S - j0;
        for (int t = tid; t < nr * nr; t += T) {
            const int i = j0 + t / nr, j = j0 + t % nr;
            const size_t x = (size_t)i * a.Sp + j;
            const int u = (i % WR) * WR + j % WR;
            kg[u] = a.gtab[x];
            kl[u] = a.ltab[x];
        }
        for (int t = tid; t < nr * L2; t += T) {
            const int j = j0 + t / L2, m = t % L2;
            xw[(j % WR) * L2 + m] = xcomp(a.rx, M, j, m);
        }
    }
    for (int i = tid; i < S; i += T) gam[i] = 0.f;
    for (int m = tid; m < M; m += T) {
        const float2 d = a.dclin[m * K + k];
        w[m] = d.x;
        w[M + m] = d.y;
    }
    const int alive0 = max(0, P - D);  // first pilot whose entry is held at the end
    auto final_at = [&](int j) {       // adjoint of the final coefficient of sample j (0 if evicted)
        const bool ok = j >= 0 && (j >> 1) >= alive0;
        return ldg_if(ok, a.dgamma + (ok ? ((size_t)((j >> 1) % D) * 2 + (j & 1)) * K + k : 0));
    };
    // centres with a nonzero R when the entrant n - W is pulled at step n (none when it is not alive
    // in any step after n)
    auto pull_hi = [&](int n) {
        const int e = evict_step(n - W);
        return e > n + 1 ? min(e, S) : n - W + 2;
    };
    __syncthreads();
    for (int j = max(0, S - W) + tid; j < S; j += T) {  // abar of the last window
        float d = 0.f;
        for (int m = 0; m < L2; ++m) d = fmaf(w[m], xcomp(a.rx, M, j, m), d);
        py[j % W] = d + final_at(j);
    }
    const int je0 = S - 1 - W;  // the first entrant
    if (je0 >= 0) row_fetch(pf, a.gtab + (size_t)je0 * a.Sp, nullptr, je0 + 2, pull_hi(S - 1));
    band_fetch(bp, a, S, W, je0, je0);
    xn = xc(je0);
    const int t_fa = L2 % T;  // the thread that updates the entrant's abar
    float fa = tid == t_fa ? final_at(je0) : 0.f;  // the entrant's final adjoint, a step early
    Tape tnext;
    auto tape_at = [&](Tape &t, bool ok, int n) {
        const float *f = reinterpret_cast<const float *>(tape + (ok ? (size_t)n * W + tid : 0));
        const float2 u0 = ld2_if(ok, f), u1 = ld2_if(ok, f + 2), u2 = ld2_if(ok, f + 4);
        t = Tape{u0.x, u0.y, u1.x, u1.y, u2.x, u2.y};
    };
    if (tid < W) tape_at(tnext, tid < S - max(0, S - W), S - 1);
    sW = pmod(S - 1 - W - 1, W);
    sR = pmod(S - 1 - W - 1, WR);
    __syncthreads();
    // scalar adjoints: thread o sums the terms of window slot o over all steps (fixed order)
    float sig_bar = 0.f, mu_bar = 0.f, eps_bar = 0.f, wl_bar = 0.f;
    for (int n = S - 1; n >= 0; --n, sW = ring_slot(sW, W - 1, W), sR = ring_slot(sR, WR - 1, WR)) {
        const int jlo = max(0, n - W + 1), nJ = n - jlo + 1, je = n - W;
        const float q = nJ == W ? qW : 1.f / (float)nJ;
        float fa_je = 0.f;
        if (tid == t_fa) {
            fa_je = fa;
            fa = final_at(je - 1);
        }
        // R after the steps >= e, kept for the centres whose entry leaves at step e = n + 1
        if (((n + 1) & 1) == 0 && n + 1 <= S - 1 && ((n + 1) >> 1) >= D && tid < W - 1) {
            const int e = n + 1;
            snap[(size_t)((e >> 1) - D) * W + tid] = gam[e - W + 1 + tid];
        }
        // the entrant's pull: sum_j R_j kappa_G(x_je, x_j) over the steps after n in which it is alive,
        // and <wbar, x_je>, both before this step's terms
        if (je >= 0) {
            if (tid <= W) {
                band_store(bp, kg, kd, kl, S, W, je, je, slotR(n, je), slotR(n, je));
                band_fetch(bp, a, S, W, je - 1, je - 1);
            }
            float ls = 0.f;
            if (tid < L2) {
                const float x = xsign(je, xn);
                xw[slotR(n, je) * L2 + tid] = x;
                ls = w[tid] * x;
                xn = xc(je - 1);
            }
            const int lo = je + 2, hi = pull_hi(n), e = evict_step(je);
            const int s_lo = e <= S - 1 ? e - W + 1 : S;  // centres whose R holds steps >= e
            const float *sv = snap + (size_t)((e >> 1) - D) * W;
            const float *grow = a.gtab + (size_t)je * a.Sp;
            float gs = 0.f;
#pragma unroll
            for (int qq = 0; qq < kPf; ++qq) {
                const int i = lo + tid + qq * T;
                if (i < hi) gs = fmaf(i >= s_lo ? gam[i] - sv[i - s_lo] : gam[i], pf.g[qq], gs);
            }
            for (int i = lo + tid + kPf * T; i < hi; i += T)
                gs = fmaf(i >= s_lo ? gam[i] - sv[i - s_lo] : gam[i], __ldg(grow + i), gs);
            reduce3(gs, ls, 0.f);
            if (je - 1 >= 0) row_fetch(pf, a.gtab + (size_t)(je - 1) * a.Sp, nullptr, je + 1, pull_hi(n - 1));
        }
        if (tid < nJ) {  // slot tid: its scalar terms and its coefficients for the state adjoint
            const Tape tp = tnext;
            tape_at(tnext, n > 0 && tid < n - max(0, n - W), n - 1);
            const int o = tid, j = jlo + o;
            const float ab = py[slotW(n, j)];
            mu_bar += q * tp.beta * ab;
            const float bbar = a.mu * q * ab;
            float cwo = 0.f, cgo = 0.f;
            if (tp.s != 0.f) {  // inside the slab beta does not depend on the state
                const float ybar = -bbar / tp.kappa;
                eps_bar += tp.s * ybar;
                wl_bar += (ybar * tp.beta) * (nrm[j] - 1.f);
                wl_bar += ybar * (tp.dotw - tp.gauss);
                sig_bar += ybar * a.wG * tp.gd2 * inv_s3;
                cwo = ybar * a.wL;
                cgo = ybar * a.wG;
            }
            ca[o] = cwo;
            cb[o] = cgo;
        } else if (tid < W) {
            tape_at(tnext, n > 0 && tid < n - max(0, n - W), n - 1);
        }
        __syncthreads();
        // adjoint of S_n: R, wbar, and abar of the samples of J_{n-1}
        if (tid < nJ) gam[jlo + tid] += cb[tid];
        const int t_lo = max(0, n - W), n_t = n - t_lo;
        const int s_lo = slotR(n, jlo);
        for (int u = tid; u < L2 + n_t; u += T) {
            if (u < L2) {
                float acc = w[u];
                int si = s_lo;
#pragma unroll 4
                for (int o = 0; o < nJ; ++o, si = ring_slot(si, 1, WR)) acc = fmaf(ca[o], xw[si * L2 + u], acc);
                w[u] = acc;
            } else {
                const int j = t_lo + (u - L2), r = slotW(n, j), sj = slotR(n, j) * WR;
                float acc;
                bool alive = true;  // centres of J_{n-1} other than the entrant are alive at step n
                if (j == je) {
                    acc = fa_je + total(0) + total(1);
                    alive = n < evict_step(j);
                } else {
                    acc = py[r];
                }
                int si = s_lo;
#pragma unroll 4
                for (int o = 0; o < nJ; ++o, si = ring_slot(si, 1, WR)) {
                    acc = fmaf(ca[o], kl[sj + si], acc);
                    if (alive) acc = fmaf(cb[o], kg[sj + si], acc);
                }
                py[r] = acc;
            }
        }
        __syncthreads();
    }

    // ---- results -------------------------------------------------------------------------------------
    for (int m = tid; m < M; m += T) a.dclin0[m * K + k] = make_float2(w[m], w[M + m]);
    float *red = py;  // py, pd, pw, ca: 4 W floats, free now
    if (tid < W) {
        red[4 * tid + 0] = sig_bar;
        red[4 * tid + 1] = mu_bar;
        red[4 * tid + 2] = eps_bar;
        red[4 * tid + 3] = wl_bar;
    }
    __syncthreads();
    if (tid < 4) {
        float s = 0.f;
        for (int o = 0; o < W; ++o) s += red[4 * o + tid];
        a.scal[k * 4 + tid] = s;
    }
}

// ---- four warps per user -----------------------------------------------------------------------
// The same recurrence and adjoint as train_bwd_kernel, for windows of at most 30 slots.  A step has
// two phases, each a set of independent pieces that one warp ran one after the other (740 warp
// instructions and 1700 cycles a step, a third of them issuing); four warps of a user now take
// them side by side and meet at a barrier of their own after each phase:
//   window warp   phase 1: the window's projections (reverse: the slots' terms), lane o = window slot o;
//                 phase 2: the carried predictions (reverse: adjoints) of the window's samples
//   row warp      phase 1: the O(S) sum over the coefficients at the sample that arrives (reverse: the
//                 pull of the one that enters), 4 kPfV entries per lane (float4) staged ahead, the rest
//                 directly; phase 2: the coefficients
//   filter warp   phase 1: the arriving sample's product with the filter; phase 2: the filter
//   staging warp  phase 1: the next arrival's kernel values and components into the window rings;
//                 phase 2: the copies of the one kAhead steps later
// Every sum keeps the order it had in one warp.  A step is bound by the instructions and latencies
// of its longest warp in each phase.  kTeamUsers users of an instance per CTA.
// 16 antennas, 6 users, 256 pilots, W = 8: one call 1.71 ms as one warp per user, about 0.75 ms here
// (cycle stamps per real-split step: forward 600 + 950, reverse 580 + 780).
constexpr int kTeamUsers = 3;
constexpr int kTeamThreads = 128;
constexpr int kPfV = 4;    // float4 of a row per lane and table that are staged ahead (512 entries)
// The team form's launches: all of its CTAs on the GPU at once, or in two goes where rows are short and no
// entry leaves, and not where the users leave a quarter of the teams empty with wide windows, nor for up to
// 6 users over the shortest sequences; more run one warp per user, all resident at once.  16 antennas, window
// 8 unless said, us as teams and as single warps:
//   one go     6 users, 256 pilots, 64 instances 1360 and 2320; 1000 pilots 17370 and 22700
//   two goes   6 users, 256 pilots, 100 instances 2400 and 2636, 150: 2820 and 3036; window 16: 2500 and 3159;
//              7 users, 300 pilots, 64: 2588 and 2880;
//              12 users, 64: 2120 and 2552; but 400 pilots, 6 users, 150: 6340 and 6130; 700 pilots over 200
//              entries, 150: 15700 and 14900; window 24, 4 users, 150: 4570 and 4190; 40 pilots, 4 users,
//              150: 326 and 308
//   more       6 users, 256 pilots, 200 instances 4083 and 3603, 512: 9763 and 8021
// (two team CTAs on an SM at 80 registers a thread: 256 instances 5597, 5356 without).
constexpr int kTeamTwoRow = 128, kTeamTwoUsers = 6, kTeamTwoMax = 640, kTeamTwoMaxWide = 512;
// Rows from which on the entries past the staged ones are loaded sixteen (then four) to a lane together, instead
// of one after the other, each a wait for L2 in the row warp (one call, 6 users, ms, one by one and together):
// window 8: 600 entries 1.03 and 1.07, 800: 1.83 and 1.68, 1024: 3.29 and 2.37, 2000: 17.0 and 8.1, 4000: 140 and 35;
// window 20: 1024 entries 3.64 and 3.83; window 24, 4 users, 64 instances: 1400 entries 8.58 and 7.74.
constexpr int kLongRow = 768, kLongRowWide = 1280;  // windows up to 16, and wider ones
constexpr int kAhead = 3;  // steps ahead that global reads are issued; a ring of kAhead + 1 slots

// Reads of a later step, copied to the lane's own slots of a shared-memory ring (cp.async: no register
// waits for them, and a lane reads only what it copied, so its own wait orders them).  A step takes
// less than the L2 latency, so one step ahead is not enough.
__device__ __forceinline__ void cp16(float *dst, const float *src) {  // both 16-byte aligned
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(float *dst, const float *src, bool ok) {  // 0 where !ok (nothing is read)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// the copies committed kAhead - 1 or more commits ago have landed
__device__ __forceinline__ void cp_wait_oldest() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
}

// Entries lo4 + 4 (lane + 32 q) + 0..3 (q < kPfV, lo4 = lo rounded down to a multiple of 4, the
// first of the four below hi) of one or two table rows (rows are padded to a multiple of 4 floats).
__device__ __forceinline__ void row_copy(float *slot, const float *grow, const float *drow, int lo, int hi, int lane) {
    const int lo4 = lo & ~3;
#pragma unroll
    for (int q = 0; q < kPfV; ++q) {
        const int o = 4 * (lane + 32 * q), i0 = lo4 + o;
        if (i0 < hi) {
            cp16(slot + o, grow + i0);
            if (drow) cp16(slot + 128 * kPfV + o, drow + i0);
        }
    }
}

__device__ __forceinline__ float f4(const float4 &v, int e) { return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w; }

// band of row r, entries s0 + lane up to s0 + W, inside [0, S), to a slot [table][32]
__device__ __forceinline__ void band_copy(float *slot, const TrainBwdArgs &a, int S, int W, int r, int s0, int lane) {
    const int j = s0 + lane;
    const bool ok = r >= 0 && r < S && lane <= W && j >= 0 && j < S;
    const size_t x = ok ? (size_t)r * a.Sp + j : 0;
    cp4(slot + lane, a.gtab + x, ok);
    cp4(slot + 32 + lane, a.gdtab + x, ok);
    cp4(slot + 64 + lane, a.ltab + x, ok);
}

// floats of one user's region: gamma / R [S rounded up to 4, zero padded], ca, cb [32], kg, kd, kl
// [RB][RB], xw [RB][2M], py, pd, pw, pb [RB], w / wbar [2M], the step's sums [4], four zeros, RB = bwd_ring(W);
// then the rings of kAhead + 1 slots: rows [2][128 kPfV], bands and components [3][32] + [128] + a target
// [4], tape [32][6] + a final adjoint [32]
constexpr int kRowSlot = 2 * 128 * kPfV, kBandSlot = 3 * 32 + 128 + 4, kTapeSlot = 32 * 6 + 32;
// samples of the window, the one entering or leaving it and the one staged for the next step, by
// their low bits
__host__ __device__ constexpr int bwd_ring(int W) { return W + 2 <= 16 ? 16 : 32; }
__host__ __device__ inline int bwd_team_rings(int S, int W, int L2) {
    const int RB = bwd_ring(W);
    return (((S + 3) & ~3) + 64 + 3 * RB * RB + RB * L2 + 4 * RB + ((L2 + 3) & ~3) + 4 + 4 + 3) & ~3;
}
__host__ __device__ inline int bwd_team_floats(int S, int W, int L2) {
    return bwd_team_rings(S, W, L2) + (kAhead + 1) * (kRowSlot + kBandSlot + kTapeSlot);
}

// WM: a bound on the window (8, 16 or 30) over which the O(W) loops are unrolled: their operands are
// loaded first, all in flight, and slots at or past |J_n| take a zero coefficient (the rings start at
// zero, so every product is finite).
// kLong: rows of more than kLongRow entries (a form of its own: short rows are up to 8 % slower with it).
template <int WM, bool kLong>
__global__ void __launch_bounds__(kTeamThreads * kTeamUsers) train_bwd_team_kernel(const TrainBwdArgs a0) {
    extern __shared__ __align__(16) float sm[];
    const TrainBwdArgs a = for_instance(a0, blockIdx.y);
    const int lane = threadIdx.x & 31, team = threadIdx.x / kTeamThreads, tl = threadIdx.x % kTeamThreads;
    const int role = tl >> 5;  // 0: window warp, 1: row warp, 2: filter warp, 3: staging warp
    const int k = blockIdx.x * kTeamUsers + team;
    const int M = a.M, K = a.K, W = a.W, D = a.D, P = a.P, S = 2 * P, L2 = 2 * M;
    const int RB = bwd_ring(W), RM = RB - 1;  // sample j sits in ring slot j & RM
    const int S4 = (S + 3) & ~3;
    float *nrm = sm, *rk = nrm + S4;  // ||x_j||^2 and 1 / kappa_jj, shared by the users
    float *gam = rk + S4 + team * bwd_team_floats(S, W, L2);
    float *ca = gam + S4, *cb = ca + 32, *kg = cb + 32, *kd = kg + RB * RB, *kl = kd + RB * RB, *xw = kl + RB * RB;
    float *py = xw + RB * L2, *pd = py + RB, *pw = pd + RB, *pb = pw + RB, *w = pb + RB, *sums = w + L2, *zero4 = sums + 4;
    constexpr int kRing = kAhead + 1;
    static_assert((kRing & (kRing - 1)) == 0, "ring slots by mask");
    float *rows = gam + bwd_team_rings(S, W, L2), *bands = rows + kRing * kRowSlot, *tapes = bands + kRing * kBandSlot;
    auto row_slot = [&](int j) { return rows + (j & (kRing - 1)) * kRowSlot; };
    auto band_slot = [&](int j) { return bands + (j & (kRing - 1)) * kBandSlot; };
    auto tape_slot = [&](int n) { return tapes + (n & (kRing - 1)) * kTapeSlot; };
    Tape *tape = a.tape + (size_t)k * S * W;
    float *snap = a.snap + (size_t)k * (P > D ? P - D : 0) * W;
    const float inv_s3 = 1.f / (a.sigma * a.sigma * a.sigma);
    const float mqW = a.mu / (float)W, qW = 1.f / (float)W;
    auto first_centre = [&](int n) { return 2 * max(0, (n >> 1) - D + 1); };
    auto evict_step = [&](int i) { return 2 * ((i >> 1) + D); };
    // component m of sample j as stored, to its place in a band slot, and its sign (x_{2t+1}'s upper
    // half is -Re r)
    auto x_copy = [&](float *slot, int j, int m) {
        const bool ok = m < L2 && j >= 0 && j < S;
        const bool up = m >= M, odd = j & 1;
        const int mm = up ? m - M : m, comp = up ? (odd ? 0 : 1) : (odd ? 1 : 0);
        cp4(slot + 96 + m, reinterpret_cast<const float *>(a.rx + (ok ? (size_t)(j >> 1) * M + mm : 0)) + comp, ok);
    };
    auto xsign = [&](int j, int m, float v) { return (m >= M && (j & 1)) ? -v : v; };
    // the band a slot holds, into the window rings at (r, s0 + t) and (s0 + t, r): the tables are
    // exactly symmetric
    auto band_store = [&](const float *slot, int r, int s0) {
        const int j = s0 + lane;
        if (r >= 0 && r < S && lane <= W && j >= 0 && j < S) {
            const int u = (r & RM) * RB + (j & RM), v = (j & RM) * RB + (r & RM);
            const float g = slot[lane], d = slot[32 + lane], l = slot[64 + lane];
            kg[u] = g;
            kg[v] = g;
            kd[u] = d;
            kd[v] = d;
            kl[u] = l;
            kl[v] = l;
        }
    };
    // w += sum_o ca_o x_{jlo+o}, component by component in slot order (ca is zero past the window)
    auto filter_update = [&](int jlo) {
        float c[WM];
#pragma unroll
        for (int o = 0; o < WM; ++o) c[o] = ca[o];
        for (int m = lane; m < L2; m += 32) {
            float x[WM], acc = w[m];
#pragma unroll
            for (int o = 0; o < WM; ++o) x[o] = xw[((jlo + o) & RM) * L2 + m];
#pragma unroll
            for (int o = 0; o < WM; ++o) acc = fmaf(c[o], x[o], acc);
            w[m] = acc;
        }
    };

    for (int i = threadIdx.x; i < S; i += blockDim.x) {
        nrm[i] = a.ltab[(size_t)i * a.Sp + i];  // ||x_i||^2
        const float kap = fmaf(a.wL, nrm[i], a.wG);
        rk[i] = kap != 0.f ? 1.f / kap : 0.f;
    }
    __syncthreads();  // the only block barrier: nrm and rk are shared by the users
    if (k >= K) return;
    auto team_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(kTeamThreads) : "memory"); };
    for (int i = tl; i < bwd_team_floats(S, W, L2); i += kTeamThreads) gam[i] = 0.f;  // and every ring
    for (int m = tl; m < M; m += kTeamThreads) {
        const float2 c = a.clin0 ? a.clin0[m * K + k] : make_float2(0.f, 0.f);
        w[m] = c.x;
        w[M + m] = c.y;
    }
    if (a.mode & 1) {
        // what arrival j needs: its rows, its band, components and target
        auto stage_issue = [&](int j) {
            if (j < S) {
                float *slot = band_slot(j);
                row_copy(row_slot(j), a.gtab + (size_t)j * a.Sp, a.gdtab + (size_t)j * a.Sp, first_centre(j), j, lane);
                band_copy(slot, a, S, W, j, j - W, lane);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (32 * c < L2) x_copy(slot, j, lane + 32 * c);
                if (lane == 0) cp4(slot + 224, reinterpret_cast<const float *>(a.sym + (size_t)(j >> 1) * K + k) + (j & 1), true);
            }
            cp_commit();
        };
        auto stage_finish = [&](int j) {  // landed: band and components into the window rings
            cp_wait_oldest();
            if (j < S) {
                const float *slot = band_slot(j);
                band_store(slot, j, j - W);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int m = lane + 32 * c;
                    if (m < L2) xw[(j & RM) * L2 + m] = xsign(j, m, slot[96 + m]);
                }
                if (lane == 0) pb[j & RM] = slot[224];
            }
        };
        team_sync();
        if (role == 3) {
            for (int j = 0; j < kAhead; ++j) stage_issue(j);
            for (int j = 0; j < 2; ++j) {
                stage_finish(j);
                stage_issue(j + kAhead);
            }
        }
        team_sync();
        if (role == 2) {  // sample 0 arrives with no live centre
            float ws = 0.f;
            for (int m = lane; m < L2; m += 32) ws = fmaf(w[m], xw[m], ws);
            ws = warp_sum(ws);
            if (lane == 0) {
                py[0] = 0.f;
                pd[0] = 0.f;
                pw[0] = ws;
            }
        }
        team_sync();

        // ---- forward ---------------------------------------------------------------------------------------
        for (int n = 0; n < S; ++n) {
            const int jlo = max(0, n - W + 1), nJ = n - jlo + 1, jn = n + 1;
            // phase 1, from the state before this step
            if (role == 0) {
                if (lane < nJ) {  // the window's projections (Eq. beta), all from f_n
                    const float mq = nJ == W ? mqW : a.mu / (float)nJ;
                    const int j = jlo + lane, r = j & RM;
                    const float dw = pw[r], yg = py[r], gd = pd[r], r_k = rk[j], gj = gam[j], bj = pb[r];
                    const float kap = fmaf(a.wL, nrm[j], a.wG);
                    const float y = fmaf(a.wL, dw, a.wG * yg);
                    const float e = y - bj;
                    float beta = 0.f, s = 0.f;
                    if (kap != 0.f) {
                        if (e < -a.eps) { s = 1.f; beta = (-e - a.eps) * r_k; }
                        else if (e > a.eps) { s = -1.f; beta = (-e + a.eps) * r_k; }
                    }
                    ca[lane] = mq * beta;
                    cb[lane] = gj + mq * beta;  // the coefficient after the step
                    tape[(size_t)n * W + lane] = Tape{beta, s, kap, dw, yg, gd};
                }
            } else if (role == 1) {
                if (jn < S) {
                    const float *pg = row_slot(jn) + 4 * lane, *pdv = pg + 128 * kPfV;  // this lane's entries
                    const int lo = first_centre(jn), lo4 = lo & ~3;
                    float4 gm[kPfV], gv[kPfV], dv[kPfV];
#pragma unroll
                    for (int q = 0; q < kPfV; ++q) {
                        if (lo4 + 128 * q < jn) {  // (an entry at or past jn meets a zero coefficient)
                            const int i0 = lo4 + 4 * (lane + 32 * q);
                            gm[q] = *reinterpret_cast<const float4 *>(i0 < jn ? gam + i0 : zero4);
                            gv[q] = *reinterpret_cast<const float4 *>(pg + 128 * q);
                            dv[q] = *reinterpret_cast<const float4 *>(pdv + 128 * q);
                        }
                    }
                    float y2[2] = {0.f, 0.f}, d2[2] = {0.f, 0.f};  // two chains of sums
                    if (lo == 0) {  // nothing evicted yet: gamma is zero from jn on (padding included)
#pragma unroll
                        for (int q = 0; q < kPfV; ++q) {
                            if (128 * q < jn) {
                                y2[0] = fmaf(gm[q].x, gv[q].x, fmaf(gm[q].z, gv[q].z, y2[0]));
                                y2[1] = fmaf(gm[q].y, gv[q].y, fmaf(gm[q].w, gv[q].w, y2[1]));
                                d2[0] = fmaf(gm[q].x, dv[q].x, fmaf(gm[q].z, dv[q].z, d2[0]));
                                d2[1] = fmaf(gm[q].y, dv[q].y, fmaf(gm[q].w, dv[q].w, d2[1]));
                            }
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < kPfV; ++q) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int i = lo4 + 4 * (lane + 32 * q) + e;
                                if (i >= lo && i < jn) {
                                    y2[e & 1] = fmaf(f4(gm[q], e), f4(gv[q], e), y2[e & 1]);
                                    d2[e & 1] = fmaf(f4(gm[q], e), f4(dv[q], e), d2[e & 1]);
                                }
                            }
                        }
                    }
                    const float *grow = a.gtab + (size_t)jn * a.Sp, *drow = a.gdtab + (size_t)jn * a.Sp;
                    int i = max(lo, lo4 + 4 * 32 * kPfV) + lane;
                    auto together = [&](auto n_c) {  // n entries of a lane with their loads in flight together
                        constexpr int n = decltype(n_c)::value;
                        for (; i + 32 * (n - 1) < jn; i += 32 * n) {
                            float g[n], d[n];
#pragma unroll
                            for (int q = 0; q < n; ++q) {
                                g[q] = ldg_if(true, grow + i + 32 * q);
                                d[q] = ldg_if(true, drow + i + 32 * q);
                            }
#pragma unroll
                            for (int q = 0; q < n; ++q) {
                                y2[0] = fmaf(gam[i + 32 * q], g[q], y2[0]);
                                d2[0] = fmaf(gam[i + 32 * q], d[q], d2[0]);
                            }
                        }
                    };
                    if constexpr (kLong) {
                        together(std::integral_constant<int, 16>{});
                        together(std::integral_constant<int, 4>{});
                    }
                    for (; i < jn; i += 32) {
                        y2[0] = fmaf(gam[i], __ldg(grow + i), y2[0]);
                        d2[0] = fmaf(gam[i], __ldg(drow + i), d2[0]);
                    }
                    const float ys = warp_sum(y2[0] + y2[1]), ds = warp_sum(d2[0] + d2[1]);
                    if (lane == 0) {
                        sums[0] = ys;
                        sums[1] = ds;
                    }
                }
            } else if (role == 2) {
                if (jn < S) {
                    float ws = 0.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int m = lane + 32 * c;
                        if (m < L2) ws = fmaf(w[m], xw[(jn & RM) * L2 + m], ws);
                    }
                    ws = warp_sum(ws);
                    if (lane == 0) sums[2] = ws;
                }
            } else {
                stage_finish(jn + 1);
            }
            team_sync();
            // phase 2, Eq. apsm: coefficients, linear part, carried predictions of J_{n+1} (2D = W + 1: the
            // oldest centre of J_n leaves before step n+1)
            if (role == 1) {
                if (lane < nJ) gam[jlo + lane] = cb[lane];
            } else if (role == 2) {
                filter_update(jlo);
            } else if (role == 3) {
                stage_issue(jn + 1 + kAhead);
            } else {
                const int t_lo = max(0, n - W + 2), n_t = jn < S ? jn - t_lo + 1 : 0;
                const int e_lo = first_centre(n), e_hi = jn < S ? first_centre(jn) : e_lo;
                if (lane < n_t) {
                    const int j = t_lo + lane, r = j & RM;
                    float c[WM], vg[WM], vd[WM], vl[WM];
#pragma unroll
                    for (int o = 0; o < WM; ++o) {
                        const int x = ((jlo + o) & RM) * RB + r;
                        c[o] = ca[o];
                        vg[o] = kg[x];
                        vd[o] = kd[x];
                        vl[o] = kl[x];
                    }
                    float ay = j == jn ? sums[0] : py[r], ad = j == jn ? sums[1] : pd[r], aw = j == jn ? sums[2] : pw[r];
                    const int o_lo = j == jn ? max(0, e_hi - jlo) : 0;
#pragma unroll
                    for (int o = 0; o < WM; ++o) {  // (ca is zero past the window)
                        const float cg = o >= o_lo ? c[o] : 0.f;
                        aw = fmaf(c[o], vl[o], aw);
                        ay = fmaf(cg, vg[o], ay);
                        ad = fmaf(cg, vd[o], ad);
                    }
                    if (j != jn) {
                        const float *grow = a.gtab + (size_t)j * a.Sp, *drow = a.gdtab + (size_t)j * a.Sp;
                        for (int i = e_lo; i < e_hi; ++i) {
                            const float gi = i >= jlo ? cb[i - jlo] : gam[i];
                            ay = fmaf(-gi, __ldg(grow + i), ay);
                            ad = fmaf(-gi, __ldg(drow + i), ad);
                        }
                    }
                    py[r] = ay;
                    pd[r] = ad;
                    pw[r] = aw;
                }
            }
            team_sync();
        }

    }  // forward
    if (!(a.mode & 2)) return;

    // ---- reverse sweep ---------------------------------------------------------------------------------
    asm volatile("cp.async.wait_all;" ::: "memory");  // the rings of slots are free
    team_sync();
    {  // kernel values and components of the last W + 1 samples (as the forward left them)
        const int j0 = max(0, S - W - 1), nr = S - j0;
        for (int t = tl; t < nr * nr; t += kTeamThreads) {
            const int i = j0 + t / nr, j = j0 + t % nr;
            const size_t x = (size_t)i * a.Sp + j;
            kg[(i & RM) * RB + (j & RM)] = a.gtab[x];
            kl[(i & RM) * RB + (j & RM)] = a.ltab[x];
        }
        for (int t = tl; t < nr * L2; t += kTeamThreads) {
            const int j = j0 + t / L2, m = t % L2;
            xw[(j & RM) * L2 + m] = xcomp(a.rx, M, j, m);
        }
    }
    for (int i = tl; i < S4; i += kTeamThreads) gam[i] = 0.f;  // R
    for (int m = tl; m < M; m += kTeamThreads) {
        const float2 d = a.dclin[m * K + k];
        w[m] = d.x;
        w[M + m] = d.y;
    }
    const int alive0 = max(0, P - D);
    auto final_src = [&](int j, bool &ok) {
        ok = j >= 0 && (j >> 1) >= alive0;
        int t = j >> 1;  // its ring slot: t mod D (t < D unless entries were evicted)
        if (P > D) t %= D;
        return a.dgamma + (ok ? ((size_t)t * 2 + (j & 1)) * K + k : 0);
    };
    auto pull_hi = [&](int n) {
        const int e = evict_step(n - W);
        return e > n + 1 ? min(e, S) : n - W + 2;
    };
    // what step n of the sweep needs: its tape, and its entrant n - W's final adjoint, row, band and
    // components
    auto stage_issue = [&](int n) {
        if (n >= 0) {
            float *slot = tape_slot(n);
            const int j = n - W;
            if (lane < min(n + 1, W)) {
                const float *f = reinterpret_cast<const float *>(tape + (size_t)n * W + lane);
#pragma unroll
                for (int i = 0; i < 3; ++i) cp8(slot + 6 * lane + 2 * i, f + 2 * i);
            }
            if (j >= 0) {
                bool ok;
                const float *fs = final_src(j, ok);
                if (lane == 0) cp4(slot + 192, fs, ok);
                row_copy(row_slot(n), a.gtab + (size_t)j * a.Sp, nullptr, j + 2, pull_hi(n), lane);
                band_copy(band_slot(n), a, S, W, j, j, lane);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (32 * c < L2) x_copy(band_slot(n), j, lane + 32 * c);
            }
        }
        cp_commit();
    };
    auto stage_finish = [&](int n) {
        cp_wait_oldest();
        const int j = n - W;
        if (j >= 0) {
            const float *slot = band_slot(n);
            band_store(slot, j, j);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int m = lane + 32 * c;
                if (m < L2) xw[(j & RM) * L2 + m] = xsign(j, m, slot[96 + m]);
            }
        }
    };
    team_sync();
    if (role == 0) {
        for (int j = max(0, S - W) + lane; j < S; j += 32) {  // abar of the last window (xw holds them)
            float d = 0.f;
            for (int m = 0; m < L2; ++m) d = fmaf(w[m], xw[(j & RM) * L2 + m], d);
            bool ok;
            const float *fs = final_src(j, ok);
            py[j & RM] = d + (ok ? __ldg(fs) : 0.f);
        }
    } else if (role == 3) {
        for (int i = 0; i < kAhead; ++i) stage_issue(S - 1 - i);
        stage_finish(S - 1);
        stage_issue(S - 1 - kAhead);
    }
    if (lane >= W && role == 0) ca[lane] = cb[lane] = 0.f;  // (and past |J_n| below: zero coefficients)
    team_sync();
    float sig_bar = 0.f, mu_bar = 0.f, eps_bar = 0.f, wl_bar = 0.f;  // lane o: window slot o's terms
    for (int n = S - 1; n >= 0; --n) {
        const int jlo = max(0, n - W + 1), nJ = n - jlo + 1, je = n - W;
        float fa_je = 0.f;
        // phase 1, from the adjoint of S_{n+1}
        if (role == 0) {
            const float *slot = tape_slot(n);  // (landed before the last barrier)
            fa_je = slot[192];
            if (lane < nJ) {
                const float q = nJ == W ? qW : 1.f / (float)nJ;
                const float2 u0 = *reinterpret_cast<const float2 *>(slot + 6 * lane),
                             u1 = *reinterpret_cast<const float2 *>(slot + 6 * lane + 2),
                             u2 = *reinterpret_cast<const float2 *>(slot + 6 * lane + 4);
                const Tape tp{u0.x, u0.y, u1.x, u1.y, u2.x, u2.y};
                const int j = jlo + lane;
                const float ab = py[j & RM], r_k = rk[j], nj = nrm[j];
                mu_bar += q * tp.beta * ab;
                const float bbar = a.mu * q * ab;
                float cwo = 0.f, cgo = 0.f;
                if (tp.s != 0.f) {
                    const float ybar = -bbar * r_k;
                    cwo = ybar * a.wL;
                    cgo = ybar * a.wG;
                    eps_bar += tp.s * ybar;
                    wl_bar += (ybar * tp.beta) * (nj - 1.f);
                    wl_bar += ybar * (tp.dotw - tp.gauss);
                    sig_bar += ybar * a.wG * tp.gd2 * inv_s3;
                }
                ca[lane] = cwo;
                cb[lane] = cgo;
            } else {
                ca[lane] = cb[lane] = 0.f;
            }
        } else if (role == 1) {
            if (((n + 1) & 1) == 0 && n + 1 <= S - 1 && ((n + 1) >> 1) >= D && lane < W - 1) {
                const int e = n + 1;  // R after the steps >= e, for the centres whose entry leaves at e
                snap[(size_t)((e >> 1) - D) * W + lane] = gam[e - W + 1 + lane];
            }
            if (je >= 0) {
                const float *pg = row_slot(n) + 4 * lane;
                const int lo = je + 2, hi = pull_hi(n), e = evict_step(je);
                const int s_lo = e <= S - 1 ? e - W + 1 : S;
                const float *sv = snap + (size_t)((e >> 1) - D) * W;
                const float *grow = a.gtab + (size_t)je * a.Sp;
                const int lo4 = lo & ~3;
                float4 rm[kPfV], gv[kPfV];
#pragma unroll
                for (int q = 0; q < kPfV; ++q) {
                    if (lo4 + 128 * q < hi) {
                        const int i0 = lo4 + 4 * (lane + 32 * q);
                        rm[q] = *reinterpret_cast<const float4 *>(i0 < hi ? gam + i0 : zero4);
                        gv[q] = *reinterpret_cast<const float4 *>(pg + 128 * q);
                    }
                }
                float g2[2] = {0.f, 0.f};
                if (hi == S && s_lo >= S) {  // no eviction after the entrant: R is zero below lo and past S
#pragma unroll
                    for (int q = 0; q < kPfV; ++q) {
                        if (lo4 + 128 * q < hi) {
                            g2[0] = fmaf(rm[q].x, gv[q].x, fmaf(rm[q].z, gv[q].z, g2[0]));
                            g2[1] = fmaf(rm[q].y, gv[q].y, fmaf(rm[q].w, gv[q].w, g2[1]));
                        }
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < kPfV; ++q) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int i = lo4 + 4 * (lane + 32 * q) + c;
                            if (i >= lo && i < hi) {
                                const float r = i >= s_lo ? f4(rm[q], c) - sv[i - s_lo] : f4(rm[q], c);
                                g2[c & 1] = fmaf(r, f4(gv[q], c), g2[c & 1]);
                            }
                        }
                    }
                }
                int i = max(lo, lo4 + 4 * 32 * kPfV) + lane;
                const int below = min(hi, s_lo);  // (no snapshot below s_lo)
                auto together = [&](auto n_c) {
                    constexpr int n = decltype(n_c)::value;
                    for (; i + 32 * (n - 1) < below; i += 32 * n) {
                        float g[n];
#pragma unroll
                        for (int q = 0; q < n; ++q) g[q] = ldg_if(true, grow + i + 32 * q);
#pragma unroll
                        for (int q = 0; q < n; ++q) g2[0] = fmaf(gam[i + 32 * q], g[q], g2[0]);
                    }
                };
                if constexpr (kLong) {
                    together(std::integral_constant<int, 16>{});
                    together(std::integral_constant<int, 4>{});
                }
                for (; i < hi; i += 32)
                    g2[0] = fmaf(i >= s_lo ? gam[i] - sv[i - s_lo] : gam[i], __ldg(grow + i), g2[0]);
                const float gs = warp_sum(g2[0] + g2[1]);
                if (lane == 0) sums[0] = gs;
            }
        } else if (role == 2) {
            if (je >= 0) {
                float ls = 0.f;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int m = lane + 32 * c;
                    if (m < L2) ls = fmaf(w[m], xw[(je & RM) * L2 + m], ls);
                }
                ls = warp_sum(ls);
                if (lane == 0) sums[1] = ls;
            }
        } else {
            stage_finish(n - 1);
        }
        team_sync();
        // phase 2: the adjoint of S_n
        if (role == 1) {
            if (lane < nJ) gam[jlo + lane] += cb[lane];
        } else if (role == 2) {
            filter_update(jlo);
        } else if (role == 3) {
            stage_issue(n - 1 - kAhead);
        } else {
            const int t_lo = max(0, n - W), n_t = n - t_lo;
            if (lane < n_t) {
                const int j = t_lo + lane, r = j & RM;
                float c[WM], b[WM], vg[WM], vl[WM];
#pragma unroll
                for (int o = 0; o < WM; ++o) {
                    const int x = ((jlo + o) & RM) * RB + r;
                    c[o] = ca[o];
                    b[o] = cb[o];
                    vg[o] = kg[x];
                    vl[o] = kl[x];
                }
                const bool alive = j != je || n < evict_step(j);
                float acc = j == je ? fa_je + sums[0] + sums[1] : py[r];
#pragma unroll
                for (int o = 0; o < WM; ++o) {
                    acc = fmaf(c[o], vl[o], acc);
                    acc = fmaf(alive ? b[o] : 0.f, vg[o], acc);
                }
                py[r] = acc;
            }
        }
        team_sync();
    }

    if (role == 2)
        for (int m = lane; m < M; m += 32) a.dclin0[m * K + k] = make_float2(w[m], w[M + m]);
    // slot partials combined in slot order
    float *red = kg;
    if (role == 0) {
        if (lane < W) {
            red[4 * lane + 0] = sig_bar;
            red[4 * lane + 1] = mu_bar;
            red[4 * lane + 2] = eps_bar;
            red[4 * lane + 3] = wl_bar;
        }
        __syncwarp();
        if (lane < 4) {
            float s = 0.f;
            for (int o = 0; o < W; ++o) s += red[4 * o + lane];
            a.scal[k * 4 + lane] = s;
        }
    }
}

#include "train_bwd_warp.cuh"

__global__ void train_bwd_sum_kernel(const TrainBwdArgs a0) {
    const TrainBwdArgs a = for_instance(a0, blockIdx.y);
    if (threadIdx.x < 4) {
        float s = 0.f;
        for (int k = 0; k < a.K; ++k) s += a.scal[k * 4 + threadIdx.x];  // users in order
        a.dscalars[threadIdx.x] = s;
    }
}

size_t train_bwd_smem(int M, int W, int P) {
    return sizeof(float) * (size_t)(2 * 2 * P + 2 * M + 6 * W + 3 * (kBwdThreads / 32) + 3 * (W + 1) * (W + 1) +
                                    (W + 1) * 2 * M);
}

}  // namespace apsm

using namespace apsm;

namespace {

struct BwdLayout {
    size_t ltab, gtab, gdtab, tape, snap, scal, total;
};

BwdLayout bwd_layout(const apsm_params *p, int P) {
    BwdLayout b;
    const size_t S = 2 * (size_t)P;
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    size_t off = 0;
    const size_t Sp = (S + 3) & ~size_t(3);
    b.ltab = off;
    off = al(off + sizeof(float) * S * Sp);
    b.gtab = off;
    off = al(off + sizeof(float) * S * Sp);
    b.gdtab = off;
    off = al(off + sizeof(float) * S * Sp);
    b.tape = off;
    off = al(off + sizeof(Tape) * (size_t)p->K * S * p->window);
    b.snap = off;
    off = al(off + sizeof(float) * (size_t)p->K * (size_t)std::max(0, P - p->dict_cap) * p->window);
    b.scal = off;
    off = al(off + sizeof(float) * 4 * (size_t)p->K);
    b.total = off;
    return b;
}

}  // namespace

namespace {

// The calls of one batch of n instances (n = 1 for apsm_train_backward).  mode 1: the tables and
// the forward pass (the tape, kept in the workspace); 2: the reverse sweep over a workspace that
// mode 1 filled; 3: both.
apsm_status train_bwd_run(const apsm_params *p, int n, const float *rx_pilot, const float *sym_pilot, int32_t P,
                          const float *clin0, const float *dgamma, const float *dclin, float *dscalars, float *dclin0,
                          void *workspace, size_t workspace_bytes, void *stream, int mode) {
    size_t dummy = 0;
    apsm_status s = apsm_train_workspace_bytes(p, 0, &dummy);
    if (s != APSM_OK) return s;
    if (n < 1 || n > 65535 || P < 1 || !rx_pilot) return APSM_ERR_INVALID_ARG;
    if ((mode & 1) && !sym_pilot) return APSM_ERR_INVALID_ARG;
    if ((mode & 2) && (!dgamma || !dclin || !dscalars || !dclin0)) return APSM_ERR_INVALID_ARG;
    if (P > 8192) return APSM_ERR_UNSUPPORTED;
    if (p->weights != APSM_Q_UNIFORM) return APSM_ERR_UNSUPPORTED;  // the adjoint of q = 1/|J_n| only
    const BwdLayout b = bwd_layout(p, P);
    if (!workspace || workspace_bytes < b.total * (size_t)n) return APSM_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(workspace) & 255) return APSM_ERR_INVALID_ARG;
    const size_t smem = train_bwd_smem(p->M, p->window, P);
    // four warps per user when the window fits the lanes and the rings of a CTA's users its shared memory
    const size_t smem_w =
        sizeof(float) * (2 * (size_t)((2 * P + 3) & ~3) +
                         (size_t)std::min(p->K, kTeamUsers) * bwd_team_floats(2 * P, p->window, 2 * p->M));
    const size_t smem_1 =
        sizeof(float) * (2 * (size_t)((2 * P + 3) & ~3) + (size_t)p->K * bwd_warp_floats(2 * P, p->window, 2 * p->M));
    const int users = std::min(p->K, kTeamUsers), ctas = (p->K + users - 1) / users;
    const bool one_fits = p->window <= 32 && smem_1 <= 227 * 1024;
    const bool team_fits = p->window <= 30 && smem_w <= 227 * 1024;
    if (!team_fits && !one_fits && smem > 227 * 1024) return APSM_ERR_UNSUPPORTED;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return APSM_ERR_CUDA;
    }
    int major = 0, minor = 0;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
    if (major != 10 || minor != 3) return APSM_ERR_NOT_SM103;
    const int row = 2 * std::min(P, p->dict_cap);  // live centres
    const bool is_long = row > (p->window <= 16 ? kLongRow : kLongRowWide);
    auto team_kern = p->window <= 8    ? (is_long ? train_bwd_team_kernel<8, true> : train_bwd_team_kernel<8, false>)
                     : p->window <= 16 ? (is_long ? train_bwd_team_kernel<16, true> : train_bwd_team_kernel<16, false>)
                                       : (is_long ? train_bwd_team_kernel<30, true> : train_bwd_team_kernel<30, false>);
    bool team_form = team_fits;
    if (team_fits) {
        if (cudaFuncSetAttribute(team_kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_w) != cudaSuccess)
            return APSM_ERR_CUDA;
        if (one_fits) {
            const long long grid = (long long)ctas * n;
            int sms = 0, per_sm = 1;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return APSM_ERR_CUDA;
            if (grid > sms && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, team_kern, kTeamThreads * users,
                                                                            smem_w) != cudaSuccess)
                return APSM_ERR_CUDA;
            const bool two_goes = grid <= 2LL * sms * per_sm && P <= p->dict_cap &&
                                  (p->window <= 16 ? row <= kTeamTwoMax
                                                   : row <= kTeamTwoMaxWide && 4 * p->K >= 3 * users * ctas) &&
                                  (row >= kTeamTwoRow || p->K > kTeamTwoUsers);
            team_form = grid <= (long long)sms * per_sm || two_goes;
        }
    }
    cudaStream_t strm = static_cast<cudaStream_t>(stream);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    TrainBwdArgs a{};
    a.M = p->M;
    a.K = p->K;
    a.W = p->window;
    a.D = p->dict_cap;
    a.P = P;
    a.Sp = (2 * P + 3) & ~3;
    a.sigma = p->sigma;
    a.mu = p->mu;
    a.eps = p->eps;
    a.wL = p->w_L;
    a.wG = 1.f - p->w_L;
    a.k2 = kLog2e / (2.f * p->sigma * p->sigma);
    a.rx = reinterpret_cast<const float2 *>(rx_pilot);
    a.sym = reinterpret_cast<const float2 *>(sym_pilot);
    a.clin0 = reinterpret_cast<const float2 *>(clin0);
    a.dgamma = dgamma;
    a.dclin = reinterpret_cast<const float2 *>(dclin);
    a.ltab = reinterpret_cast<float *>(ws + b.ltab);
    a.gtab = reinterpret_cast<float *>(ws + b.gtab);
    a.gdtab = reinterpret_cast<float *>(ws + b.gdtab);
    a.tape = reinterpret_cast<Tape *>(ws + b.tape);
    a.snap = reinterpret_cast<float *>(ws + b.snap);
    a.scal = reinterpret_cast<float *>(ws + b.scal);
    a.dclin0 = reinterpret_cast<float2 *>(dclin0);
    a.dscalars = dscalars;
    a.st_rx = (size_t)P * p->M;
    a.st_sym = (size_t)P * p->K;
    a.st_clin0 = (size_t)p->M * p->K;
    a.st_dgamma = (size_t)round_up(p->dict_cap, kTileEntries) * 2 * p->K;
    a.st_mk = (size_t)p->M * p->K;
    a.ws_stride = b.total;
    a.mode = mode;
    const bool one_form = !team_form && one_fits;
    const long long pairs = 2LL * P * a.Sp;
    const int blocks = (int)std::min<long long>(std::max(1, 4096 / n), (pairs + 255) / 256);
    if (mode & 1) train_bwd_tables_kernel<<<dim3(blocks, n), 256, 0, strm>>>(a);
    if (team_form) {
        team_kern<<<dim3(ctas, n), kTeamThreads * users, smem_w, strm>>>(a);
    } else if (one_form) {
        auto kern = p->window <= 8 ? train_bwd_warp_kernel<8>
                    : p->window <= 16 ? train_bwd_warp_kernel<16> : train_bwd_warp_kernel<32>;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_1) != cudaSuccess)
            return APSM_ERR_CUDA;
        kern<<<dim3(1, n), 32 * p->K, smem_1, strm>>>(a);
    } else {
        if (cudaFuncSetAttribute(train_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess)
            return APSM_ERR_CUDA;
        train_bwd_kernel<<<dim3(p->K, n), kBwdThreads, smem, strm>>>(a);
    }
    if (mode & 2) train_bwd_sum_kernel<<<dim3(1, n), 32, 0, strm>>>(a);
    g_launches += 1 + (mode & 1) + ((mode & 2) >> 1);
    return cudaGetLastError() == cudaSuccess ? APSM_OK : APSM_ERR_CUDA;
}

}  // namespace

extern "C" {

apsm_status apsm_train_backward_workspace_bytes(const apsm_params *p, int32_t P, size_t *bytes) {
    return apsm_train_backward_batched_workspace_bytes(p, P, 1, bytes);
}

apsm_status apsm_train_backward_batched_workspace_bytes(const apsm_params *p, int32_t P, int32_t n, size_t *bytes) {
    size_t dummy = 0;
    apsm_status s = apsm_train_workspace_bytes(p, 0, &dummy);  // parameter validation
    if (s != APSM_OK) return s;
    if (!bytes || P < 0 || n < 1) return APSM_ERR_INVALID_ARG;
    *bytes = bwd_layout(p, P).total * (size_t)n;
    return APSM_OK;
}

apsm_status apsm_train_backward(const apsm_params *p, const float *rx_pilot, const float *sym_pilot, int32_t P,
                                const float *clin0, const float *dgamma, const float *dclin, float *dscalars,
                                float *dclin0, void *workspace, size_t workspace_bytes, void *stream) {
    return train_bwd_run(p, 1, rx_pilot, sym_pilot, P, clin0, dgamma, dclin, dscalars, dclin0, workspace,
                         workspace_bytes, stream, 3);
}

apsm_status apsm_train_backward_batched(const apsm_params *p, int32_t n, const float *rx_pilot, const float *sym_pilot,
                                        int32_t P, const float *clin0, const float *dgamma, const float *dclin,
                                        float *dscalars, float *dclin0, void *workspace, size_t workspace_bytes,
                                        void *stream) {
    return train_bwd_run(p, n, rx_pilot, sym_pilot, P, clin0, dgamma, dclin, dscalars, dclin0, workspace,
                         workspace_bytes, stream, 3);
}

apsm_status apsm_train_backward_batched_forward(const apsm_params *p, int32_t n, const float *rx_pilot,
                                                const float *sym_pilot, int32_t P, const float *clin0,
                                                void *workspace, size_t workspace_bytes, void *stream) {
    return train_bwd_run(p, n, rx_pilot, sym_pilot, P, clin0, nullptr, nullptr, nullptr, nullptr, workspace,
                         workspace_bytes, stream, 1);
}

apsm_status apsm_train_backward_batched_reverse(const apsm_params *p, int32_t n, const float *rx_pilot, int32_t P,
                                                const float *dgamma, const float *dclin, float *dscalars,
                                                float *dclin0, void *workspace, size_t workspace_bytes,
                                                void *stream) {
    return train_bwd_run(p, n, rx_pilot, nullptr, P, nullptr, dgamma, dclin, dscalars, dclin0, workspace,
                         workspace_bytes, stream, 2);
}

}  // extern "C"
