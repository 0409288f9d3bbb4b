// lsq_simt.cu -- the column least-squares solves of SAM construction
// (arXiv 2406.17656, Sec. 2: min_m || A_k(I_j, J_j) m - A_0(I_j, j) ||) with one
// thread per column: size classes 0 and 1 (level-1 columns) of refined FP32
// builds of many columns.
//
// The refinement needs R only as a preconditioner: with R^T R close to B^T B a
// corrected semi-normal-equation step r = c - B m, g = B^T r, R^T R d = g,
// m += d contracts the error by rho, about u_32 kappa(B)^2 for the Cholesky
// factor of an FP32 Gram matrix.  So the thread forms
//   G = B^T B, b = B^T c, G = L L^T, m = G^{-1} b  in FP32  (error ~ rho |m|)
// and takes one step more than the build's s steps, all with r and g in FP64.
// On level-1 columns of Q1 diffusion rho is about 3e-7 against 1.5e-7 for the
// QR's R, so s + 1 steps leave less error than the QR kernel's s (measured
// against 64 bits: the same 1.5e-16 for s = 2, 3e-15 against 1e-13 for s = 1).
//
// Why a thread per column: a 25 x 9 problem has 81 entries in B and 45 in G;
// cooperating lanes spend their time on shuffles and idle register slots
// (lsq_kernel.cuh issues about 1,900 warp instructions per column here).  Alone,
// a thread needs no communication and keeps its state in 0.5 KB of shared
// memory, interleaved over the warp's 32 threads so that every access is free of
// bank conflicts whatever each thread's index.  The sparse passes read the
// sources' values and the local rows from copies interleaved over 32 columns
// (simt_values, simt_rows), padded to W entries per column with zeros and an
// unused row, so neighbouring threads' loads fall in the same sectors and no
// entry is tested.  Columns with 23 or more unknowns need 2 KB each: three warps
// per SM, whose latency nothing hides (measured 1.6 times slower than the QR
// kernel on 49 x 25 columns), so they keep lsq_kernel.cuh.
//
// Measured, 4 maps of 512^2 unknowns, level 1, two steps: 1.65 ms for the class-1
// launch against 3.94 ms (lsq_kernel.cuh); FP64 arithmetic bounds it (16
// cycles of an SM per warp instruction, about 270 of its 460 cycles per column).
// Loading two columns ahead costs the registers of two warps per SM (2.05 ms);
// 12 and 16 warps per SM are equal.
#include <cfloat>
#include <type_traits>

#include "lsq_core.cuh"

namespace sam {
namespace {

constexpr __host__ __device__ int tri(int q) { return q * (q + 1) / 2; }

constexpr int kSimtWarps = 16;  // one-warp blocks per SM at most (128 registers each)
constexpr int kAhead = 1;       // columns loaded ahead of their use
// One column problem per lane.  Word i of a lane's shared memory is at
// 32 i + lane, so that any index of any lane hits its own bank.
template <int MAXI_, int MAXJ_>
struct SimtShape {
    static constexpr int MAXI = MAXI_, MAXJ = MAXJ_;
    static constexpr int ROWS = MAXI + 1;                // and the row of the padding entries
    static constexpr int LW = (tri(MAXJ + 1) + 3) & ~3;  // rows 0..MAXJ of [G b], then of L
    static constexpr int RW = LW;                        // r in FP64 (2 words a row); w2 during the Gram pass
    static constexpr int W4 = (LW - 2 * ROWS) & ~3;      // w4 (4 words a row: the end of L, and r) during the Gram pass
    static constexpr int TAB = LW + 2 * ROWS;            // columns of J
    static constexpr int WORDS = TAB + MAXJ;
    static_assert(MAXJ % 2 == 1 && RW % 2 == 0, "shape");
    // the row groups of four that leave w4 alone
    static constexpr int Q4 = [] {
        int q = 0;
        while (q + 4 <= MAXJ + 1 && tri(q + 4) <= W4) q += 4;
        return q;
    }();
    static constexpr int BYTES = 128 * WORDS;
    static constexpr int FIT = 232448 / (BYTES + 1024);
    static constexpr int WARPS = FIT < kSimtWarps ? FIT : kSimtWarps;  // one-warp blocks per SM
};

// W entries of one column of B: values and local rows
template <typename T, int W>
struct Ent {
    T v[W];
    int i[W];
};

template <class SH, int W>
__global__ void __launch_bounds__(32, SH::WARPS) lsq_simt_kernel(LsqArgs args, int bin) {
    constexpr int MAXI = SH::MAXI, MAXJ = SH::MAXJ;
    extern __shared__ __align__(16) float smem_f[];
    const int lane = threadIdx.x;
    float *S = smem_f + lane;  // word i of this lane: S[32 i]
    double *R = reinterpret_cast<double *>(smem_f + 32 * SH::RW) + lane;

    const int w0 = args.bin_off[bin] + (args.item_hi > 0 ? args.item_lo : 0);
    const int total = args.item_hi > 0 ? args.item_hi - args.item_lo : args.bin_off[bin + 1] - w0;
    const int32_t *work = args.work + w0;
    for (int base = blockIdx.x * 32; base < total; base += gridDim.x * 32) {
        const bool valid = base + lane < total;
        const int jj = work[valid ? base + lane : base];  // (idle lanes repeat a column and write nothing)
        const int kmap = jj / args.n;
        const int jl = jj - kmap * args.n;
        const int js = args.shadow_shared ? jl : jj;
        const int64_t poff = args.shadow_shared ? (int64_t)kmap * args.map_nnz_pat : 0;
        const int64_t eoff = args.shadow_shared ? (int64_t)kmap * args.ell_map : 0;
        const int roff = kmap * args.n;
        const int zc = args.zbig ? jj : jl;
        const int jb = args.jcp[js], n = args.jcp[js + 1] - jb, nI = args.icnt[js];
        const int zb = args.zcp[zc], ze = args.zcp[zc + 1];
        const int nmax = __reduce_max_sync(0xffffffffu, n);
        const int imax = __reduce_max_sync(0xffffffffu, nI);
        int status = kStOk;
        // the columns of J (past them the first one again: its values meet
        // padding rows there)
        for (int c = 0; c < nmax; ++c) S[32 * (SH::TAB + c)] = __int_as_float(args.jri[jb + (c < n ? c : 0)]);
        const uint8_t *lrow = args.lrow_t + ((int64_t)(js >> 5) * kLTile) * 32 + (js & 31);
        auto ell = [&](int c) -> int64_t {
            const int col = __float_as_int(S[32 * (SH::TAB + c)]);
            return eoff + (int64_t)(col >> 5) * (32 * W) + (col & 31);
        };
        auto fetch32 = [&](Ent<float, W> &e, int c) {
            const float *v = args.kev32 + ell(c);
            const uint8_t *l = lrow + c * (32 * W);
#pragma unroll
            for (int u = 0; u < W; ++u) e.v[u] = v[32 * u];
#pragma unroll
            for (int u = 0; u < W; ++u) e.i[u] = l[32 * u];
        };
        auto fetch64 = [&](Ent<double, W> &e, int c) {
            const double *v = args.kev + ell(c);
            const uint8_t *l = lrow + c * (32 * W);
#pragma unroll
            for (int u = 0; u < W; ++u) e.v[u] = v[32 * u];
#pragma unroll
            for (int u = 0; u < W; ++u) e.i[u] = l[32 * u];
        };
        const int zro = (args.shadow_shared ? 0 : roff) - (args.zbig ? roff : 0);
        auto target_row = [&](int t) -> int {
            int i;
            if (args.zloc && t - zb < kZCap) {
                i = args.zloc[(int64_t)js * kZCap + (t - zb)];
                if (i == kZOutside) return -1;
                if (i >= nI) {  // impossible for a consistent shadow: never index out of bounds
                    status = kStUnsupported;
                    return -1;
                }
                return i;
            }
            return find_sorted(args.ish + (int64_t)js * kICap, nI, args.zri[t] + zro);
        };
        // ---- [G b] = [B c]^T B in FP32: NW columns q of [B c] at a time
        // dense in w, their products with every column c <= q
        auto gram = [&](auto nw_, int qbeg, int qend, float *w) {
            constexpr int NW = decltype(nw_)::value;
            for (int i = 0; i < imax; ++i)
#pragma unroll
                for (int t = 0; t < NW; ++t) w[32 * NW * i + t] = 0.f;
#pragma unroll
            for (int t = 0; t < NW; ++t) w[32 * NW * MAXI + t] = 0.f;
            for (int q0 = qbeg; q0 < qend; q0 += NW) {
                if (q0 > nmax) break;
                const int cend = min(q0 + NW, nmax);
                Ent<float, W> E[kAhead + 1];
                fetch32(E[0], 0);
                                int rows[NW][W];
#pragma unroll
                for (int t = 0; t < NW; ++t) {
                    const int q = q0 + t;
                    if (q < nmax) {
                        Ent<float, W> e;
                        fetch32(e, q);
#pragma unroll
                        for (int u = 0; u < W; ++u) {
                            rows[t][u] = e.i[u];
                            if (q < n) w[32 * NW * e.i[u] + t] = e.v[u];
                        }
                    }
                    w[32 * NW * MAXI + t] = 0.f;  // (padding entries wrote there)
                    if (q == n)
                        for (int z = zb; z < ze; ++z) {
                            const int i = target_row(z);
                            if (i >= 0) w[32 * NW * i + t] = args.zcv32[z];
                        }
                }
                auto dots = [&](const Ent<float, W> &e, int c) {
                    float acc[NW] = {};
#pragma unroll
                    for (int u = 0; u < W; ++u) {
                        const float *wr = w + 32 * NW * e.i[u];
                        if constexpr (NW == 4) {
                            const float4 x = *reinterpret_cast<const float4 *>(wr);
                            acc[0] = fmaf(e.v[u], x.x, acc[0]);
                            acc[1] = fmaf(e.v[u], x.y, acc[1]);
                            acc[2] = fmaf(e.v[u], x.z, acc[2]);
                            acc[3] = fmaf(e.v[u], x.w, acc[3]);
                        } else {
                            const float2 x = *reinterpret_cast<const float2 *>(wr);
                            acc[0] = fmaf(e.v[u], x.x, acc[0]);
                            acc[1] = fmaf(e.v[u], x.y, acc[1]);
                        }
                    }
                    const int b = tri(q0) + c;
#pragma unroll
                    for (int t = 0; t < NW; ++t)
                        if (q0 + t >= c && q0 + t <= MAXJ) S[32 * (b + t * q0 + tri(t))] = acc[t];
                };
                for (int c = 0; c < cend; c += kAhead + 1) {
#pragma unroll
                    for (int k = 0; k < kAhead + 1; ++k) {
                        if (c + k < cend) {
                            if (c + k + kAhead < cend) fetch32(E[(k + kAhead) % (kAhead + 1)], c + k + kAhead);
                            dots(E[k], c + k);
                        }
                    }
                }
                // clear the block's columns of w
#pragma unroll
                for (int t = 0; t < NW; ++t) {
                    const int q = q0 + t;
                    if (q < nmax) {
#pragma unroll
                        for (int u = 0; u < W; ++u) w[32 * NW * rows[t][u] + t] = 0.f;
                    }
                    if (q == n)
                        for (int z = zb; z < ze; ++z) {
                            const int i = target_row(z);
                            if (i >= 0) w[32 * NW * i + t] = 0.f;
                        }
                }
            }
        };
        gram(std::integral_constant<int, 4>{}, 0, SH::Q4, smem_f + 32 * SH::W4 + 4 * lane);
        gram(std::integral_constant<int, 2>{}, SH::Q4, MAXJ + 1, smem_f + 32 * SH::RW + 2 * lane);
        // ---- r = c in FP64
        double out2 = 0.0;
        for (int i = 0; i < imax; ++i) R[32 * i] = 0.0;
        R[32 * MAXI] = 0.0;
        for (int z = zb; z < ze; ++z) {
            const int i = target_row(z);
            const double v = args.zcv[z];
            if (i >= 0) R[32 * i] = v;
            else out2 = fma(v, v, out2);
        }
        // ---- G = L L^T, two rows at a time in registers; the row of b gives
        // y = L^{-1} b.  The diagonal holds 1 / L_kk
        float dmax = 0.f, dmin = FLT_MAX;
        bool brk = false;
        for (int q0 = 0; q0 <= nmax; q0 += 2) {
            const int b0 = tri(q0), b1 = tri(q0 + 1);
            float a0[MAXJ], a1[MAXJ];
            float t00 = S[32 * (b0 + q0)], t10 = S[32 * (b1 + q0)], t11 = S[32 * (b1 + q0 + 1)];
            if ((q0 < n && t00 == 0.f) || (q0 + 1 < n && t11 == 0.f)) status = max(status, (int)kStRank);
#pragma unroll
            for (int j = 0; j < MAXJ - 1; ++j) {
                if (j >= q0) break;
                float s0 = S[32 * (b0 + j)], s1 = S[32 * (b1 + j)], p0 = 0.f, p1 = 0.f;
#pragma unroll
                for (int k = 0; k < j; ++k) {
                    const float l = S[32 * (tri(j) + k)];
                    if (k & 1) {
                        p0 = fmaf(-a0[k], l, p0);
                        p1 = fmaf(-a1[k], l, p1);
                    } else {
                        s0 = fmaf(-a0[k], l, s0);
                        s1 = fmaf(-a1[k], l, s1);
                    }
                }
                const float inv = S[32 * (tri(j) + j)];
                a0[j] = (s0 + p0) * inv;
                a1[j] = (s1 + p1) * inv;
                S[32 * (b0 + j)] = a0[j];
                S[32 * (b1 + j)] = a1[j];
                t00 = fmaf(-a0[j], a0[j], t00);
                t10 = fmaf(-a0[j], a1[j], t10);
                t11 = fmaf(-a1[j], a1[j], t11);
            }
            auto pivot = [&](int q, float t) -> float {
                if (q >= n) return 0.f;
                // (past a breakdown every pivot is NaN: the FP64 re-solve decides)
                if (!brk && !(fabsf(t) <= FLT_MAX)) status = max(status, (int)kStNonfinite);
                brk = brk || !(t > 0.f);
                dmax = fmaxf(dmax, t);
                dmin = fminf(dmin, t);
                return rsqrtf(t);
            };
            const float i0 = pivot(q0, t00);
            const float l10 = t10 * i0;
            const float i1 = pivot(q0 + 1, fmaf(-l10, l10, t11));
            S[32 * (b0 + q0)] = i0;
            S[32 * (b1 + q0)] = l10;
            S[32 * (b1 + q0 + 1)] = i1;
        }
        const float kap2 = dmax / dmin;  // a lower bound on kappa(B)^2
        const int xb = tri(n);           // y, then each product's x and g, in the row of b
        float x[MAXJ];
        auto load_x = [&]() {
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) x[j] = (j < n) ? S[32 * (xb + j)] : 0.f;
        };
        auto store_x = [&]() {
#pragma unroll
            for (int j = 0; j < MAXJ; ++j)
                if (j < n) S[32 * (xb + j)] = x[j];
        };
        auto back = [&]() {  // L^T x = y
#pragma unroll
            for (int j = MAXJ - 1; j >= 0; --j) {
                if (j >= nmax) continue;
                if (j < n) {
                    const float xj = x[j] * S[32 * (tri(j) + j)];
                    x[j] = xj;
#pragma unroll
                    for (int k = 0; k < j; ++k) x[k] = fmaf(-S[32 * (tri(j) + k)], xj, x[k]);
                }
            }
        };
        auto fwd = [&]() {  // L y = g
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) {
                if (j >= nmax) break;
                float s = x[j], p = 0.f;
#pragma unroll
                for (int k = 0; k < j; ++k) {
                    const float l = S[32 * (tri(j) + k)];
                    if (k & 1) p = fmaf(-l, x[k], p);
                    else s = fmaf(-l, x[k], s);
                }
                x[j] = (j < n) ? (s + p) * S[32 * (tri(j) + j)] : 0.f;
            }
        };
        load_x();
        back();
        double m[MAXJ];
        float msq = 0.f;
#pragma unroll
        for (int j = 0; j < MAXJ; ++j) {
            m[j] = widen(x[j]);
            msq = fmaf(x[j], x[j], msq);
        }
        double r2 = 0.0;
        bool fallback = brk, redo = false;
        const bool autoref = args.refine_steps < 0;
        const int steps = autoref ? 1 : args.refine_steps;
        float da2 = 0.f, dprev2 = 0.f;
        for (int step = 0; step <= steps; ++step) {
            store_x();
            Ent<double, W> E[kAhead + 1];
            // r -= B x (FP64), column by column
            fetch64(E[0], 0);
            for (int c = 0; c < nmax; c += kAhead + 1) {
#pragma unroll
                for (int k = 0; k < kAhead + 1; ++k) {
                    if (c + k < nmax) {
                        if (c + k + kAhead < nmax) fetch64(E[(k + kAhead) % (kAhead + 1)], c + k + kAhead);
                        const double xc = c + k < n ? -widen(S[32 * (xb + c + k)]) : 0.0;
                        double rv[W];
#pragma unroll
                        for (int u = 0; u < W; ++u) rv[u] = R[32 * E[k].i[u]];
#pragma unroll
                        for (int u = 0; u < W; ++u) rv[u] = fma(E[k].v[u], xc, rv[u]);
#pragma unroll
                        for (int u = 0; u < W; ++u) R[32 * E[k].i[u]] = rv[u];
                    }
                }
            }
            // g = B^T r (FP64, rounded to FP32)
            fetch64(E[0], 0);
            for (int c = 0; c < nmax; c += kAhead + 1) {
#pragma unroll
                for (int k = 0; k < kAhead + 1; ++k) {
                    if (c + k < nmax) {
                        if (c + k + kAhead < nmax) fetch64(E[(k + kAhead) % (kAhead + 1)], c + k + kAhead);
                        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll
                        for (int u = 0; u < W; ++u) {
                            const double rr = R[32 * E[k].i[u]];
                            if (u % 3 == 0) s0 = fma(E[k].v[u], rr, s0);
                            else if (u % 3 == 1) s1 = fma(E[k].v[u], rr, s1);
                            else s2 = fma(E[k].v[u], rr, s2);
                        }
                        if (c + k < n) S[32 * (xb + c + k)] = narrow_trunc(s0 + s1 + s2);
                    }
                }
            }
            load_x();
            fwd();
            back();
            float dsq = 0.f;
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) {
                m[j] += widen(x[j]);
                dsq = fmaf(x[j], x[j], dsq);
            }
            // Accuracy guard (as lsq_kernel.cuh): rho estimated as the largest
            // of kRhoSafety u_32 kappa^2, kAutoC |d_1| / |m| (the first
            // correction is the Cholesky solve's error, about rho |m|) and
            // |d_s| / |d_{s-1}|; a predicted error rho / (1 - rho) |d_s| above
            // kFallbackTol |m| misses
            constexpr float kTol = (float)kFallbackTol, kTol2 = kTol * kTol, kC = (float)kAutoC;
            if (step == 0) da2 = dsq;
            if (step == steps) {
                const float rk = (float)(kRhoSafety * kU32) * kap2;
                bool miss = !(rk < 0.5f) || rk * rk * dsq > kTol2 * (1.f - rk) * (1.f - rk) * msq;
                miss = miss || 4.f * kC * kC * da2 >= msq || 4.f * kC * kC * da2 * dsq > kTol2 * msq * msq;
                if (step > 0 && dsq > (float)kNoise2 * msq)
                    miss = miss || 4.f * dsq >= dprev2 || 4.f * dsq * dsq > kTol2 * msq * dprev2;
                if (autoref)
                    redo = kC * dsq > (float)kAutoTol * msq || miss;
                else
                    fallback = fallback || miss;
                // ||r - B d||^2 = ||r||^2 - d.g (g = B^T r = G d up to rounding)
                float dg = 0.f;
#pragma unroll
                for (int j = 0; j < MAXJ; ++j)
                    if (j < n) dg = fmaf(x[j], S[32 * (xb + j)], dg);
                for (int i = 0; i < nI; ++i) r2 = fma(R[32 * i], R[32 * i], r2);
                r2 -= widen(dg);
            }
            dprev2 = dsq;
        }
        if (autoref && brk) redo = true;
        // ---- outputs
        if (valid) {
            if (args.refine_used)
                args.refine_used[jj] = (uint8_t)((fallback && status == kStOk) ? kAutoSteps + 1 : (steps < 2 ? steps : 2));
            bool nf = !finite64(r2);
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) nf = nf || (j < n && !finite64(m[j]));
            if (status == kStOk && !brk && !fallback && !redo && nf) status = kStNonfinite;
            if (status == kStOk && fallback && !autoref) status = kStRefine;
            if (status == kStOk && redo) status = kStStep2;
#pragma unroll
            for (int j = 0; j < MAXJ; ++j)
                if (j < n) args.mval[args.csr_pos[jb + j] + poff] = (status == kStOk) ? m[j] : 0.0;
            args.colres[jj] = (status == kStOk) ? (r2 > 0.0 ? r2 : 0.0) + out2 : 0.0;
            args.colstat[jj] = status;
        }
    }
}

template <class SH, int W>
cudaError_t launch_simt(sam_handle h, const LsqArgs &a, int bin) {
    const size_t smem = SH::BYTES;
    auto kern = lsq_simt_kernel<SH, W>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    profile_begin(h, bin);
    kern<<<per_sm * handle_sms(h), 32, smem, handle_stream(h)>>>(a, bin);
    count_launch(h);
    profile_end(h, bin);
    return cudaGetLastError();
}

template <int W>
cudaError_t launch_width(sam_handle h, const LsqArgs &args, int bin) {
    switch (bin) {
        case 0: return launch_simt<SimtShape<14, 5>, W>(h, args, 0);
        case 1: return launch_simt<SimtShape<26, 9>, W>(h, args, 1);
        default: return cudaErrorInvalidValue;
    }
}

__global__ void simt_values_kernel(int n, int W, const int32_t *kcp, int64_t map_nnz, const double *cv, int64_t ell_map,
                                   double *kev, float *kev32) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const int k = blockIdx.y;
    const int b = kcp[c], len = kcp[c + 1] - b;
    const double *v = cv + (int64_t)k * map_nnz + b;
    const int64_t o = (int64_t)k * ell_map + (int64_t)(c >> 5) * (32 * W) + (c & 31);
    for (int u = 0; u < W; ++u) {
        const double x = u < len ? v[u] : 0.0;
        kev[o + 32 * u] = x;
        kev32[o + 32 * u] = (float)x;
    }
}

// a block per 32 columns, a warp per column at a time
__global__ void __launch_bounds__(256) simt_rows_kernel(int n, int W, const int32_t *kcp, const int32_t *jcp,
                                                        const int32_t *jri, const uint8_t *bin, const uint8_t *lrow,
                                                        uint8_t *lrow_t) {
    __shared__ __align__(4) uint8_t sh[kLTile][32];
    __shared__ int most;
    const int j0 = blockIdx.x * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) most = 0;
    __syncthreads();
    for (int q = warp; q < 32; q += 8) {
        const int j = j0 + q;
        const int b = j < n ? bin[j] : kBinNone;
        if (b >= kSimtBins) continue;
        const int pad = b == 0 ? 14 : 26;  // its shape's padding row
        const int jb = jcp[j], nj = jcp[j + 1] - jb;
        int len = 0;
        if (lane < nj) {
            const int col = jri[jb + lane];
            len = kcp[col + 1] - kcp[col];
        }
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane < kSimtJ) {
            const uint8_t *src = lrow + (int64_t)j * kLCap + (incl - len);
            for (int u = 0; u < W; ++u) sh[lane * W + u][q] = u < len ? src[u] : (uint8_t)pad;
        }
        if (lane == 0) atomicMax(&most, 1);
    }
    __syncthreads();
    if (!most) return;
    const unsigned *src = reinterpret_cast<const unsigned *>(&sh[0][0]);
    unsigned *dst = reinterpret_cast<unsigned *>(lrow_t + (int64_t)blockIdx.x * kLTile * 32);
    for (int t = threadIdx.x; t < kSimtJ * W * 8; t += 256) dst[t] = src[t];
}

}  // namespace

int simt_width(int maxcol) {
    return maxcol < 0 || maxcol > kEllW ? 0 : maxcol <= 5 ? 5 : maxcol <= 7 ? 7 : maxcol <= 9 ? 9 : kEllW;
}

cudaError_t launch_lsq_simt_bin(sam_handle h, const LsqArgs &args, int bin) {
    switch (args.ell_w) {
        case 5: return launch_width<5>(h, args, bin);
        case 7: return launch_width<7>(h, args, bin);
        case 9: return launch_width<9>(h, args, bin);
        case kEllW: return launch_width<kEllW>(h, args, bin);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t simt_values(sam_handle h, int n, int K, int W, const int32_t *kcp, int64_t map_nnz, const double *cv,
                        int64_t ell_map, double *kev, float *kev32) {
    if (n == 0 || K == 0) return cudaSuccess;
    simt_values_kernel<<<dim3((unsigned)((n + 255) / 256), (unsigned)K), 256, 0, handle_stream(h)>>>(
        n, W, kcp, map_nnz, cv, ell_map, kev, kev32);
    count_launch(h);
    return cudaGetLastError();
}

cudaError_t simt_rows(sam_handle h, int n, int W, const int32_t *kcp, const int32_t *jcp, const int32_t *jri,
                      const uint8_t *bin, const uint8_t *lrow, uint8_t *lrow_t) {
    if (n == 0) return cudaSuccess;
    simt_rows_kernel<<<(unsigned)((n + 31) / 32), 256, 0, handle_stream(h)>>>(n, W, kcp, jcp, jri, bin, lrow, lrow_t);
    count_launch(h);
    return cudaGetLastError();
}

}  // namespace sam
