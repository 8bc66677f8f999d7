// train_bwd_warp.cuh -- the training adjoint with one warp per user, for launches of more users than the
// four-warp teams of train_bwd.cu fill the GPU with twice, and for windows of 31 and 32 slots.
// Included by train_bwd.cu inside its namespace (its argument block and helpers are used here).
//
// ---- one warp per user -------------------------------------------------------------------------
// The same recurrence and adjoint as train_bwd_kernel, for windows of at most 32 slots: one warp
// per user (lane o = window slot o), the users of one instance in one CTA, and no block barrier
// inside the step loop -- each step synchronises one warp only.  The O(S) sums of a step take
// 4 kPfV entries per lane (float4 loads) from registers loaded a step ahead (the rest directly).
constexpr int kWarpUsersMax = 16;  // users (warps) per CTA of train_bwd_warp_kernel

__device__ __forceinline__ float4 ldg4_if(bool c, const float *p) {  // p 16-byte aligned
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t@q ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w)
                 : "l"(p), "r"((int)c));
    return v;
}

// Entries lo4 + 4 (lane + 32 q) + 0..3 (q < kPfV, lo4 = lo rounded down to a multiple of 4, the
// first of the four below hi) of one or two table rows (rows are padded to a multiple of 4 floats).
struct RowPfW {
    float4 g[kPfV], d[kPfV];
};

__device__ __forceinline__ void row_fetch_w(RowPfW &f, const float *grow, const float *drow, int lo, int hi, int lane) {
    const int lo4 = lo & ~3;
#pragma unroll
    for (int q = 0; q < kPfV; ++q) {
        const int i0 = lo4 + 4 * (lane + 32 * q);
        f.g[q] = ldg4_if(i0 < hi, grow + i0);
        f.d[q] = ldg4_if(drow != nullptr && i0 < hi, drow + i0);
    }
}

// band of row r, entries s0 + t for t = lane (and lane + 32 when W = 32), inside [0, S)
template <int NQ>
__device__ __forceinline__ void band_fetch_w(BandPf &b, const TrainBwdArgs &a, int S, int W, int r, int s0, int lane) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int t = lane + 32 * q, j = s0 + t;
        const bool ok = r >= 0 && r < S && t <= W && j >= 0 && j < S;
        const size_t x = ok ? (size_t)r * a.Sp + j : 0;
        b.g[q] = ldg_if(ok, a.gtab + x);
        b.d[q] = ldg_if(ok, a.gdtab + x);
        b.l[q] = ldg_if(ok, a.ltab + x);
    }
}

template <int NQ>
__device__ __forceinline__ void band_store_w(const BandPf &b, float *kg, float *kd, float *kl, int S, int W, int r,
                                             int s0, int sr, int s0r, int lane) {
    const int WR = W + 1;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int t = lane + 32 * q, j = s0 + t;
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

// floats of one warp's region: gamma / R [S rounded up to 4, zero padded], kg, kd, kl [(W+1)^2],
// xw [(W+1)][2M], py, pd, pw, pb, ca, cb [W], w / wbar [2M]
__host__ __device__ inline int bwd_warp_floats(int S, int W, int L2) {
    const int WR = W + 1;
    return (((S + 3) & ~3) + 3 * WR * WR + WR * L2 + 6 * W + L2 + 3) & ~3;
}

// WM: a bound on the window (8, 16 or 32) over which the O(W) loops are unrolled, so that their
// shared-memory loads are independent of one another.
template <int WM>
__global__ void __launch_bounds__(32 * kWarpUsersMax) train_bwd_warp_kernel(const TrainBwdArgs a0) {
    extern __shared__ __align__(16) float sm[];
    const TrainBwdArgs a = for_instance(a0, blockIdx.y);
    constexpr int NQ = WM >= 32 ? 2 : 1;  // band entries per lane (W + 1 <= 32 NQ)
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    const int M = a.M, K = a.K, W = a.W, D = a.D, P = a.P, S = 2 * P, L2 = 2 * M, WR = W + 1;
    float *nrm = sm, *rk = nrm + ((S + 3) & ~3);  // ||x_j||^2 and 1 / kappa_jj, shared by the users
    float *gam = rk + ((S + 3) & ~3) + k * bwd_warp_floats(S, W, L2);
    const int S4 = (S + 3) & ~3;
    float *kg = gam + S4, *kd = kg + WR * WR, *kl = kd + WR * WR, *xw = kl + WR * WR;
    float *py = xw + WR * L2, *pd = py + W, *pw = pd + W, *pb = pw + W, *ca = pb + W, *cb = ca + W, *w = cb + W;
    Tape *tape = a.tape + (size_t)k * S * W;
    float *snap = a.snap + (size_t)k * (P > D ? P - D : 0) * W;
    const float inv_s3 = 1.f / (a.sigma * a.sigma * a.sigma);
    const float mqW = a.mu / (float)W, qW = 1.f / (float)W;
    auto pmod = [](int x, int R) { return ((x % R) + R) % R; };
    int sW = 0, sR = 0;  // slots of the reference sample n - W - 1 (mod W, mod W + 1)
    auto slotW = [&](int n, int j) { return ring_slot(sW, j - (n - W - 1), W); };
    auto slotR = [&](int n, int j) { return ring_slot(sR, j - (n - W - 1), WR); };
    auto first_centre = [&](int n) { return 2 * max(0, (n >> 1) - D + 1); };
    auto evict_step = [&](int i) { return 2 * ((i >> 1) + D); };
    // component m of sample j as stored, and its sign (x_{2t+1}'s upper half is -Re r)
    auto xc = [&](int j, int m) {
        const bool ok = m < L2 && j >= 0 && j < S;
        const bool up = m >= M, odd = j & 1;
        const int mm = up ? m - M : m, comp = up ? (odd ? 0 : 1) : (odd ? 1 : 0);
        return ldg_if(ok, reinterpret_cast<const float *>(a.rx + (ok ? (size_t)(j >> 1) * M + mm : 0)) + comp);
    };
    auto xsign = [&](int j, int m, float v) { return (m >= M && (j & 1)) ? -v : v; };
    auto wrap = [&](int x) { return x >= WR ? x - WR : x; };  // x < 2 (W + 1)
    auto target_at = [&](bool ok, int j) {
        return ldg_if(ok, reinterpret_cast<const float *>(a.sym + (ok ? (size_t)(j >> 1) * K + k : 0)) + (j & 1));
    };

    for (int i = threadIdx.x; i < S; i += blockDim.x) {
        nrm[i] = a.ltab[(size_t)i * a.Sp + i];  // ||x_i||^2
        const float kap = fmaf(a.wL, nrm[i], a.wG);
        rk[i] = kap != 0.f ? 1.f / kap : 0.f;
    }
    __syncthreads();  // the only block barrier: nrm and rk are shared by the users
    for (int i = lane; i < S4; i += 32) gam[i] = 0.f;
    for (int m = lane; m < M; m += 32) {
        const float2 c = a.clin0 ? a.clin0[m * K + k] : make_float2(0.f, 0.f);
        w[m] = c.x;
        w[M + m] = c.y;
    }
    RowPfW pf;
    BandPf bp;
    float xn[4];
    if (a.mode & 1) {
        sW = pmod(-W - 1, W);
        sR = pmod(-W - 1, WR);
        band_fetch_w<NQ>(bp, a, S, W, 0, -W, lane);
        band_store_w<NQ>(bp, kg, kd, kl, S, W, 0, -W, slotR(0, 0), slotR(0, -W), lane);
        band_fetch_w<NQ>(bp, a, S, W, 1, 1 - W, lane);
        if (S > 1) row_fetch_w(pf, a.gtab + a.Sp, a.gdtab + a.Sp, first_centre(1), 1, lane);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int m = lane + 32 * c;
            if (m < L2) xw[slotR(0, 0) * L2 + m] = xcomp(a.rx, M, 0, m);
            xn[c] = xc(1, m);
        }
        float bn = target_at(lane == 0 && S > 1, 1);  // the next arrival's target, a step early
        if (lane == 0) pb[0] = target_at(true, 0);
        __syncwarp();
        {
            float ws = 0.f;
            for (int m = lane; m < L2; m += 32) ws = fmaf(w[m], xw[slotR(0, 0) * L2 + m], ws);
            ws = warp_sum(ws);
            if (lane == 0) {
                py[0] = 0.f;
                pd[0] = 0.f;
                pw[0] = ws;
            }
        }
        __syncwarp();

        // ---- forward ---------------------------------------------------------------------------------------
        for (int n = 0; n < S; ++n, sW = ring_slot(sW, 1, W), sR = ring_slot(sR, 1, WR)) {
            const int jlo = max(0, n - W + 1), nJ = n - jlo + 1, jn = n + 1;
            const float mq = nJ == W ? mqW : a.mu / (float)nJ;
            const float b_jn = bn;
            bn = target_at(lane == 0 && jn + 1 < S, jn + 1);
            float ys = 0.f, ds = 0.f, ws = 0.f;  // the arrival's sums from the state before this step
            if (jn < S) {
                band_store_w<NQ>(bp, kg, kd, kl, S, W, jn, jn - W, slotR(n, jn), slotR(n, jn - W), lane);
                band_fetch_w<NQ>(bp, a, S, W, jn + 1, jn + 1 - W, lane);
                const int sx = slotR(n, jn) * L2;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int m = lane + 32 * c;
                    if (m < L2) {
                        const float x = xsign(jn, m, xn[c]);
                        xw[sx + m] = x;
                        ws = fmaf(w[m], x, ws);
                        xn[c] = xc(jn + 1, m);
                    }
                }
                const int lo = first_centre(jn), lo4 = lo & ~3;
                float y2[2] = {0.f, 0.f}, d2[2] = {0.f, 0.f};  // two chains of sums
                if (lo == 0) {  // nothing evicted yet: gamma is zero from jn on (padding included)
#pragma unroll
                    for (int q = 0; q < kPfV; ++q) {
                        const int i0 = 4 * (lane + 32 * q);
                        if (i0 < jn) {
                            const float4 gm = *reinterpret_cast<const float4 *>(gam + i0);
                            y2[0] = fmaf(gm.x, pf.g[q].x, fmaf(gm.z, pf.g[q].z, y2[0]));
                            y2[1] = fmaf(gm.y, pf.g[q].y, fmaf(gm.w, pf.g[q].w, y2[1]));
                            d2[0] = fmaf(gm.x, pf.d[q].x, fmaf(gm.z, pf.d[q].z, d2[0]));
                            d2[1] = fmaf(gm.y, pf.d[q].y, fmaf(gm.w, pf.d[q].w, d2[1]));
                        }
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < kPfV; ++q) {
                        const int i0 = lo4 + 4 * (lane + 32 * q);
                        if (i0 < jn) {
                            const float4 gm = *reinterpret_cast<const float4 *>(gam + i0);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int i = i0 + e;
                                if (i >= lo && i < jn) {
                                    y2[e & 1] = fmaf(f4(gm, e), f4(pf.g[q], e), y2[e & 1]);
                                    d2[e & 1] = fmaf(f4(gm, e), f4(pf.d[q], e), d2[e & 1]);
                                }
                            }
                        }
                    }
                }
                const float *grow = a.gtab + (size_t)jn * a.Sp, *drow = a.gdtab + (size_t)jn * a.Sp;
                for (int i = max(lo, lo4 + 4 * 32 * kPfV) + lane; i < jn; i += 32) {
                    y2[0] = fmaf(gam[i], __ldg(grow + i), y2[0]);
                    d2[0] = fmaf(gam[i], __ldg(drow + i), d2[0]);
                }
                ys = y2[0] + y2[1];
                ds = d2[0] + d2[1];
                if (jn + 1 < S)
                    row_fetch_w(pf, a.gtab + (size_t)(jn + 1) * a.Sp, a.gdtab + (size_t)(jn + 1) * a.Sp,
                                first_centre(jn + 1), jn + 1, lane);
                ys = warp_sum(ys);
                ds = warp_sum(ds);
                ws = warp_sum(ws);
            }
            if (lane < nJ) {  // the window's projections (Eq. beta), all from f_n
                const int j = jlo + lane, r = slotW(n, j);
                const float dw = pw[r], yg = py[r], gd = pd[r];
                const float y = fmaf(a.wL, dw, a.wG * yg);
                const float e = y - pb[r];
                const float kap = fmaf(a.wL, nrm[j], a.wG), r_k = rk[j];
                float beta = 0.f, s = 0.f;
                if (kap != 0.f) {
                    if (e < -a.eps) { s = 1.f; beta = (-e - a.eps) * r_k; }
                    else if (e > a.eps) { s = -1.f; beta = (-e + a.eps) * r_k; }
                }
                tape[(size_t)n * W + lane] = Tape{beta, s, kap, dw, yg, gd};
                ca[lane] = mq * beta;
                cb[lane] = gam[j] + mq * beta;  // the coefficient after the step
            }
            __syncwarp();
            // Eq. apsm: coefficients, linear part, carried predictions of J_{n+1} (2D = W + 1: the oldest
            // centre of J_n leaves before step n+1)
            if (lane < nJ) gam[jlo + lane] = cb[lane];
            if (lane == 0 && jn < S) pb[slotW(n, jn)] = b_jn;
            const int s_lo = slotR(n, jlo);
            for (int m = lane; m < L2; m += 32) {
                float acc = w[m];
#pragma unroll
                for (int o = 0; o < WM; ++o)
                    if (o < nJ) acc = fmaf(ca[o], xw[wrap(s_lo + o) * L2 + m], acc);
                w[m] = acc;
            }
            const int t_lo = max(0, n - W + 2), n_t = jn < S ? jn - t_lo + 1 : 0;
            const int e_lo = first_centre(n), e_hi = jn < S ? first_centre(jn) : e_lo;
            if (lane < n_t) {
                const int j = t_lo + lane, r = slotW(n, j), sj = slotR(n, j) * WR;
                float ay, ad, aw;
                if (j == jn) {
                    ay = ys;
                    ad = ds;
                    aw = ws;
                } else {
                    ay = py[r];
                    ad = pd[r];
                    aw = pw[r];
                }
                const int o_lo = j == jn ? max(0, e_hi - jlo) : 0;
#pragma unroll
                for (int o = 0; o < WM; ++o) {
                    if (o < nJ) {
                        const int si = sj + wrap(s_lo + o);
                        const float c = ca[o];
                        aw = fmaf(c, kl[si], aw);
                        if (o >= o_lo) {
                            ay = fmaf(c, kg[si], ay);
                            ad = fmaf(c, kd[si], ad);
                        }
                    }
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
            __syncwarp();
        }

    }  // forward
    if (!(a.mode & 2)) return;

    // ---- reverse sweep ---------------------------------------------------------------------------------
    {  // kernel values and components of the last W + 1 samples (as the forward left them)
        const int j0 = max(0, S - W - 1), nr = S - j0;
        for (int t = lane; t < nr * nr; t += 32) {
            const int i = j0 + t / nr, j = j0 + t % nr;
            const size_t x = (size_t)i * a.Sp + j;
            const int u = (i % WR) * WR + j % WR;
            kg[u] = a.gtab[x];
            kl[u] = a.ltab[x];
        }
        for (int t = lane; t < nr * L2; t += 32) {
            const int j = j0 + t / L2, m = t % L2;
            xw[(j % WR) * L2 + m] = xcomp(a.rx, M, j, m);
        }
    }
    __syncwarp();
    for (int i = lane; i < S4; i += 32) gam[i] = 0.f;  // R
    for (int m = lane; m < M; m += 32) {
        const float2 d = a.dclin[m * K + k];
        w[m] = d.x;
        w[M + m] = d.y;
    }
    const int alive0 = max(0, P - D);
    auto final_at = [&](int j) {
        const bool ok = j >= 0 && (j >> 1) >= alive0;
        int t = j >> 1;  // its ring slot: t mod D (t < D unless entries were evicted)
        if (P > D) t %= D;
        return ldg_if(ok, a.dgamma + (ok ? ((size_t)t * 2 + (j & 1)) * K + k : 0));
    };
    auto pull_hi = [&](int n) {
        const int e = evict_step(n - W);
        return e > n + 1 ? min(e, S) : n - W + 2;
    };
    __syncwarp();
    for (int j = max(0, S - W) + lane; j < S; j += 32) {  // abar of the last window (xw holds them)
        float d = 0.f;
        const int sx = pmod(j, WR) * L2;
        for (int m = 0; m < L2; ++m) d = fmaf(w[m], xw[sx + m], d);
        py[j % W] = d + final_at(j);
    }
    const int je0 = S - 1 - W;
    if (je0 >= 0) row_fetch_w(pf, a.gtab + (size_t)je0 * a.Sp, nullptr, je0 + 2, pull_hi(S - 1), lane);
    band_fetch_w<NQ>(bp, a, S, W, je0, je0, lane);
#pragma unroll
    for (int c = 0; c < 4; ++c) xn[c] = xc(je0, lane + 32 * c);
    float fa = final_at(je0);  // every lane: the entrant's final adjoint, a step early
    Tape tnext;
    auto tape_at = [&](Tape &t, bool ok, int n) {
        const float *f = reinterpret_cast<const float *>(tape + (ok ? (size_t)n * W + lane : 0));
        const float2 u0 = ld2_if(ok, f), u1 = ld2_if(ok, f + 2), u2 = ld2_if(ok, f + 4);
        t = Tape{u0.x, u0.y, u1.x, u1.y, u2.x, u2.y};
    };
    tape_at(tnext, lane < S - max(0, S - W), S - 1);
    sW = pmod(S - 1 - W - 1, W);
    sR = pmod(S - 1 - W - 1, WR);
    __syncwarp();
    float sig_bar = 0.f, mu_bar = 0.f, eps_bar = 0.f, wl_bar = 0.f;  // lane o: window slot o's terms
    for (int n = S - 1; n >= 0; --n, sW = ring_slot(sW, W - 1, W), sR = ring_slot(sR, WR - 1, WR)) {
        const int jlo = max(0, n - W + 1), nJ = n - jlo + 1, je = n - W;
        const float q = nJ == W ? qW : 1.f / (float)nJ;
        const float fa_je = fa;
        fa = final_at(je - 1);
        if (((n + 1) & 1) == 0 && n + 1 <= S - 1 && ((n + 1) >> 1) >= D && lane < W - 1) {
            const int e = n + 1;  // R after the steps >= e, for the centres whose entry leaves at e
            snap[(size_t)((e >> 1) - D) * W + lane] = gam[e - W + 1 + lane];
        }
        float gs = 0.f, ls = 0.f;
        if (je >= 0) {
            band_store_w<NQ>(bp, kg, kd, kl, S, W, je, je, slotR(n, je), slotR(n, je), lane);
            band_fetch_w<NQ>(bp, a, S, W, je - 1, je - 1, lane);
            const int sx = slotR(n, je) * L2;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int m = lane + 32 * c;
                if (m < L2) {
                    const float x = xsign(je, m, xn[c]);
                    xw[sx + m] = x;
                    ls = fmaf(w[m], x, ls);
                    xn[c] = xc(je - 1, m);
                }
            }
            const int lo = je + 2, hi = pull_hi(n), e = evict_step(je);
            const int s_lo = e <= S - 1 ? e - W + 1 : S;
            const float *sv = snap + (size_t)((e >> 1) - D) * W;
            const float *grow = a.gtab + (size_t)je * a.Sp;
            const int lo4 = lo & ~3;
            float g2[2] = {0.f, 0.f};
            if (hi == S && s_lo >= S) {  // no eviction after the entrant: R is zero below lo and past S
#pragma unroll
                for (int qq = 0; qq < kPfV; ++qq) {
                    const int i0 = lo4 + 4 * (lane + 32 * qq);
                    if (i0 < hi) {
                        const float4 rm = *reinterpret_cast<const float4 *>(gam + i0);
                        g2[0] = fmaf(rm.x, pf.g[qq].x, fmaf(rm.z, pf.g[qq].z, g2[0]));
                        g2[1] = fmaf(rm.y, pf.g[qq].y, fmaf(rm.w, pf.g[qq].w, g2[1]));
                    }
                }
            } else {
#pragma unroll
                for (int qq = 0; qq < kPfV; ++qq) {
                    const int i0 = lo4 + 4 * (lane + 32 * qq);
                    if (i0 < hi) {
                        const float4 rm = *reinterpret_cast<const float4 *>(gam + i0);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int i = i0 + e;
                            if (i >= lo && i < hi) {
                                const float r = i >= s_lo ? f4(rm, e) - sv[i - s_lo] : f4(rm, e);
                                g2[e & 1] = fmaf(r, f4(pf.g[qq], e), g2[e & 1]);
                            }
                        }
                    }
                }
            }
            for (int i = max(lo, lo4 + 4 * 32 * kPfV) + lane; i < hi; i += 32)
                g2[0] = fmaf(i >= s_lo ? gam[i] - sv[i - s_lo] : gam[i], __ldg(grow + i), g2[0]);
            gs = g2[0] + g2[1];
            if (je - 1 >= 0) row_fetch_w(pf, a.gtab + (size_t)(je - 1) * a.Sp, nullptr, je + 1, pull_hi(n - 1), lane);
            gs = warp_sum(gs);
            ls = warp_sum(ls);
        }
        if (lane < nJ) {
            const Tape tp = tnext;
            tape_at(tnext, n > 0 && lane < n - max(0, n - W), n - 1);
            const int j = jlo + lane;
            const float ab = py[slotW(n, j)];
            mu_bar += q * tp.beta * ab;
            const float bbar = a.mu * q * ab;
            float cwo = 0.f, cgo = 0.f;
            if (tp.s != 0.f) {
                const float ybar = -bbar * rk[j];
                eps_bar += tp.s * ybar;
                wl_bar += (ybar * tp.beta) * (nrm[j] - 1.f);
                wl_bar += ybar * (tp.dotw - tp.gauss);
                sig_bar += ybar * a.wG * tp.gd2 * inv_s3;
                cwo = ybar * a.wL;
                cgo = ybar * a.wG;
            }
            ca[lane] = cwo;
            cb[lane] = cgo;
        }
        __syncwarp();
        if (lane < nJ) gam[jlo + lane] += cb[lane];
        const int s_lo = slotR(n, jlo);
        for (int m = lane; m < L2; m += 32) {
            float acc = w[m];
#pragma unroll
            for (int o = 0; o < WM; ++o)
                if (o < nJ) acc = fmaf(ca[o], xw[wrap(s_lo + o) * L2 + m], acc);
            w[m] = acc;
        }
        const int t_lo = max(0, n - W), n_t = n - t_lo;
        if (lane < n_t) {
            const int j = t_lo + lane, r = slotW(n, j), sj = slotR(n, j) * WR;
            float acc;
            bool alive = true;
            if (j == je) {
                acc = fa_je + gs + ls;
                alive = n < evict_step(j);
            } else {
                acc = py[r];
            }
#pragma unroll
            for (int o = 0; o < WM; ++o) {
                if (o < nJ) {
                    const int si = sj + wrap(s_lo + o);
                    acc = fmaf(ca[o], kl[si], acc);
                    if (alive) acc = fmaf(cb[o], kg[si], acc);
                }
            }
            py[r] = acc;
        }
        __syncwarp();
    }

    for (int m = lane; m < M; m += 32) a.dclin0[m * K + k] = make_float2(w[m], w[M + m]);
    // slot partials combined in slot order
    float *red = py;  // py, pd, pw, pb: 4 W floats
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
