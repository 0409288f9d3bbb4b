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
// QR's R (numpy, FP32 factors of sampled columns), so s + 1 steps leave less
// error than the QR kernel's s.
//
// Why a thread per column: a 25 x 9 problem has 81 entries in B and 45 in G;
// cooperating lanes (lsq_kernel.cuh) spend their time on shuffles and idle
// register slots.  Alone,
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
// Measured, 4 maps of 512^2 unknowns, level 1, two steps: 1.83 ms for the class-1
// launch against 3.91 ms (lsq_kernel.cuh).  FP64 arithmetic bounds it: the pipe is
// active in 58% of the cycles (16 of them per warp instruction) at 13 warps per SM,
// which wait for the operands of the FP64 passes (shared memory pipe 48%; 17,100
// warp instructions per 32 columns).  Spilled registers take 4% of those (width 9,
// class 1: 324 bytes of stores and 372 of loads in the
// build, 376 and 460 in the adjoint; width 12 about twice, width 5 none to 68).
// Loading two columns ahead costs the registers of two warps per SM (2.05 ms);
// 12 and 16 warps per SM are equal.
#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "lsq_core.cuh"
#include "simt_shape.cuh"

namespace sam {
namespace {

constexpr __host__ __device__ int tri(int q) { return simt_tri(q); }

// W entries of one column of B: values and local rows
template <typename T, int W>
struct Ent {
    T v[W];
    int i[W];
};

// One column problem: its data and the steps shared by the build and its adjoint.
template <class SH, int W>
struct Simt {
    static constexpr int MAXI = SH::MAXI, MAXJ = SH::MAXJ;
    const LsqArgs &args;
    float *smem, *S;  // word i of this lane: S[32 i]
    int lane, jj, js, n, nI, nmax, imax, zb, ze, zro, jb, roff, status;
    int64_t poff, eoff;
    const uint8_t *lrow;
    float dmax, dmin;
    bool brk;

    __device__ __forceinline__ Simt(const LsqArgs &a, float *sm, int ln) : args(a), smem(sm), S(sm + ln), lane(ln) {}

    __device__ __forceinline__ void begin(int col) {
        jj = col;
        const int kmap = jj / args.n;
        const int jl = jj - kmap * args.n;
        js = args.shadow_shared ? jl : jj;
        poff = args.shadow_shared ? (int64_t)kmap * args.map_nnz_pat : 0;
        eoff = args.shadow_shared ? (int64_t)kmap * args.ell_map : 0;
        roff = kmap * args.n;
        const int zc = args.zbig ? jj : jl;
        zro = (args.shadow_shared ? 0 : roff) - (args.zbig ? roff : 0);
        jb = args.jcp[js];
        n = args.jcp[js + 1] - jb;
        nI = args.icnt[js];
        zb = args.zcp[zc];
        ze = args.zcp[zc + 1];
        nmax = __reduce_max_sync(0xffffffffu, n);
        imax = __reduce_max_sync(0xffffffffu, nI);
        status = kStOk;
        // the columns of J (past them the first one again: its values meet
        // padding rows there)
        for (int c = 0; c < nmax; ++c) S[32 * (SH::TAB + c)] = __int_as_float(args.jri[jb + (c < n ? c : 0)]);
        lrow = args.lrow_t + ((int64_t)(js >> 5) * kLTile) * 32 + (js & 31);
    }
    __device__ __forceinline__ int64_t ell(int c) const {
        const int col = __float_as_int(S[32 * (SH::TAB + c)]);
        return eoff + (int64_t)(col >> 5) * (32 * W) + (col & 31);
    }
    template <typename T>
    __device__ __forceinline__ void fetch(Ent<T, W> &e, int c) const {
        const T *v;
        if constexpr (sizeof(T) == 4) v = args.kev32 + ell(c);
        else v = args.kev + ell(c);
        const uint8_t *l = lrow + c * (32 * W);
#pragma unroll
        for (int u = 0; u < W; ++u) e.v[u] = v[32 * u];
#pragma unroll
        for (int u = 0; u < W; ++u) e.i[u] = l[32 * u];
    }
    // f(entries, c) for the columns c < end, the next one's entries loaded
    // while this one's are used
    template <typename T, class F>
    __device__ __forceinline__ void columns(int end, F &&f) const {
        Ent<T, W> E[2];
        fetch(E[0], 0);
        for (int c = 0; c < end; c += 2) {
            if (c + 1 < end) fetch(E[1], c + 1);
            f(E[0], c);
            if (c + 1 < end) {
                if (c + 2 < end) fetch(E[0], c + 2);
                f(E[1], c + 1);
            }
        }
    }
    __device__ __forceinline__ int target_row(int t) {
        if (args.zloc && t - zb < kZCap) {
            const int i = args.zloc[(int64_t)js * kZCap + (t - zb)];
            if (i == kZOutside) return -1;
            if (i >= nI) {  // impossible for a consistent shadow: never index out of bounds
                status = kStUnsupported;
                return -1;
            }
            return i;
        }
        return find_sorted(args.ish + (int64_t)js * kICap, nI, args.zri[t] + zro);
    }

    // [G b] = [B c]^T B in FP32: two columns q of [B c] at a time dense in w,
    // their products with every column c <= q (RHS: with c as column n)
    template <bool RHS>
    __device__ __forceinline__ void gram() {
        constexpr int NW = SH::NW;
        static_assert(NW == 2, "a row of w is one float2");
        float *w = smem + 32 * SH::WW + NW * lane;
        for (int i = 0; i < imax; ++i)
#pragma unroll
            for (int t = 0; t < NW; ++t) w[32 * NW * i + t] = 0.f;
#pragma unroll
        for (int t = 0; t < NW; ++t) w[32 * NW * MAXI + t] = 0.f;
        for (int q0 = 0; q0 < MAXJ + 1; q0 += NW) {
            if (q0 >= nmax + (RHS ? 1 : 0)) break;
            const int cend = min(q0 + NW, nmax);
            int rows[NW][W];
#pragma unroll
            for (int t = 0; t < NW; ++t) {
                const int q = q0 + t;
                if (q < nmax) {
                    Ent<float, W> e;
                    fetch(e, q);
#pragma unroll
                    for (int u = 0; u < W; ++u) {
                        rows[t][u] = e.i[u];
                        if (q < n) w[32 * NW * e.i[u] + t] = e.v[u];
                    }
                }
                w[32 * NW * MAXI + t] = 0.f;  // (padding entries wrote there)
                if (RHS && q == n)
                    for (int z = zb; z < ze; ++z) {
                        const int i = target_row(z);
                        if (i >= 0) w[32 * NW * i + t] = args.zcv32[z];
                    }
            }
            columns<float>(cend, [&](const Ent<float, W> &e, int c) {
                float acc[NW] = {};
#pragma unroll
                for (int u = 0; u < W; ++u) {
                    const float2 x = *reinterpret_cast<const float2 *>(w + 32 * NW * e.i[u]);
                    acc[0] = fmaf(e.v[u], x.x, acc[0]);
                    acc[1] = fmaf(e.v[u], x.y, acc[1]);
                }
                const int b = tri(q0) + c;
#pragma unroll
                for (int t = 0; t < NW; ++t)
                    if (q0 + t >= c && q0 + t <= MAXJ) S[32 * (b + t * q0 + tri(t))] = acc[t];
            });
            // clear the block's columns of w
#pragma unroll
            for (int t = 0; t < NW; ++t) {
                const int q = q0 + t;
                if (q < nmax) {
#pragma unroll
                    for (int u = 0; u < W; ++u) w[32 * NW * rows[t][u] + t] = 0.f;
                }
                if (RHS && q == n)
                    for (int z = zb; z < ze; ++z) {
                        const int i = target_row(z);
                        if (i >= 0) w[32 * NW * i + t] = 0.f;
                    }
            }
        }
    }

    // G = L L^T, two rows at a time in registers (RHS: the row of b gives
    // y = L^{-1} b).  The diagonal holds 1 / L_kk
    template <bool RHS>
    __device__ __forceinline__ void factor() {
        dmax = 0.f;
        dmin = FLT_MAX;
        brk = false;
        for (int q0 = 0; q0 < nmax + (RHS ? 1 : 0); q0 += 2) {
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
            const float i0 = pivot(q0, t00);
            const float l10 = t10 * i0;
            const float i1 = pivot(q0 + 1, fmaf(-l10, l10, t11));
            S[32 * (b0 + q0)] = i0;
            S[32 * (b1 + q0)] = l10;
            S[32 * (b1 + q0 + 1)] = i1;
        }
    }
    __device__ __forceinline__ float pivot(int q, float t) {
        if (q >= n) return 0.f;
        // (past a breakdown every pivot is NaN: the re-solve decides)
        if (!brk && !(fabsf(t) <= FLT_MAX)) status = max(status, (int)kStNonfinite);
        brk = brk || !(t > 0.f);
        dmax = fmaxf(dmax, t);
        dmin = fminf(dmin, t);
        return rsqrtf(t);
    }

    // the vector of a product or a solve, in the row of b
    __device__ __forceinline__ void load_x(float (&x)[MAXJ]) const {
#pragma unroll
        for (int j = 0; j < MAXJ; ++j) x[j] = (j < n) ? S[32 * (tri(n) + j)] : 0.f;
    }
    __device__ __forceinline__ void store_x(const float (&x)[MAXJ]) {
#pragma unroll
        for (int j = 0; j < MAXJ; ++j)
            if (j < n) S[32 * (tri(n) + j)] = x[j];
    }
    __device__ __forceinline__ void back(float (&x)[MAXJ]) const {  // L^T x = y
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
    }
    __device__ __forceinline__ void fwd(float (&x)[MAXJ]) const {  // L y = g
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
    }

    // r += B x (FP64), column by column; x(c): the factor of column c (0 past n)
    template <class X>
    __device__ __forceinline__ void add_bx(double *R, X &&x) const {
        columns<double>(nmax, [&](const Ent<double, W> &e, int c) {
            const double xc = x(c);
            double rv[W];
#pragma unroll
            for (int u = 0; u < W; ++u) rv[u] = R[32 * e.i[u]];
#pragma unroll
            for (int u = 0; u < W; ++u) rv[u] = fma(e.v[u], xc, rv[u]);
#pragma unroll
            for (int u = 0; u < W; ++u) R[32 * e.i[u]] = rv[u];
        });
    }
    // put(c, (B^T r)_c) (FP64)
    template <class F>
    __device__ __forceinline__ void bt_r(const double *R, F &&put) const {
        columns<double>(nmax, [&](const Ent<double, W> &e, int c) {
            double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll
            for (int u = 0; u < W; ++u) {
                const double rr = R[32 * e.i[u]];
                if (u % 3 == 0) s0 = fma(e.v[u], rr, s0);
                else if (u % 3 == 1) s1 = fma(e.v[u], rr, s1);
                else s2 = fma(e.v[u], rr, s2);
            }
            if (c < n) put(c, s0 + s1 + s2);
        });
    }
    // r = c in FP64; returns the target's entries outside the shadow, squared
    __device__ __forceinline__ double target(double *R) {
        double out2 = 0.0;
        for (int i = 0; i < imax; ++i) R[32 * i] = 0.0;
        R[32 * MAXI] = 0.0;
        for (int z = zb; z < ze; ++z) {
            const int i = target_row(z);
            const double v = args.zcv[z];
            if (i >= 0) R[32 * i] = v;
            else out2 = fma(v, v, out2);
        }
        return out2;
    }
};

template <class SH, int W>
__global__ void __launch_bounds__(32, SH::WARPS) lsq_simt_kernel(LsqArgs args, int bin) {
    constexpr int MAXJ = SH::MAXJ;
    if (args.longest && simt_width(*args.longest) != W) return;
    extern __shared__ __align__(16) float smem_f[];
    const int lane = threadIdx.x;
    double *R = reinterpret_cast<double *>(smem_f + 32 * SH::RW) + lane;
    Simt<SH, W> C(args, smem_f, lane);
    float *S = C.S;

    const int w0 = args.bin_off[bin] + (args.item_hi > 0 ? args.item_lo : 0);
    const int total = args.item_hi > 0 ? args.item_hi - args.item_lo : args.bin_off[bin + 1] - w0;
    const int32_t *work = args.work + w0;
    for (int base = blockIdx.x * 32; base < total; base += gridDim.x * 32) {
        const bool valid = base + lane < total;
        C.begin(work[valid ? base + lane : base]);  // (idle lanes repeat a column and write nothing)
        const int n = C.n;
        C.template gram<true>();
        const double out2 = C.target(R);
        C.template factor<true>();
        const bool brk = C.brk;
        const float kap2 = C.dmax / C.dmin;  // a lower bound on kappa(B)^2
        // factor tape: R = L^T, packed (its rows are L's columns), also past a
        // zero or non-finite pivot
        if (args.fac_mode == kTapeRecord && valid) {
            float *dst = reinterpret_cast<float *>(args.fac) + args.fac_off[C.jj];
            for (int k = 0; k < n; ++k) {
                const float inv = S[32 * (tri(k) + k)];
                *dst++ = inv == 0.f ? inv : 1.f / inv;
                for (int c = k + 1; c < n; ++c) *dst++ = S[32 * (tri(c) + k)];
            }
        }
        const int xb = tri(n);
        float x[MAXJ];
        C.load_x(x);
        C.back(x);
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
            // r -= B x, g = B^T r (rounded to FP32), d = (L L^T)^{-1} g, m += d
            C.store_x(x);
            C.add_bx(R, [&](int c) { return c < n ? -widen(S[32 * (xb + c)]) : 0.0; });
            C.bt_r(R, [&](int c, double g) { S[32 * (xb + c)] = narrow_trunc(g); });
            C.load_x(x);
            C.fwd(x);
            C.back(x);
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
                for (int i = 0; i < C.nI; ++i) r2 = fma(R[32 * i], R[32 * i], r2);
                r2 -= widen(dg);
            }
            dprev2 = dsq;
        }
        if (autoref && brk) redo = true;
        // ---- outputs
        int status = C.status;
        if (valid) {
            if (args.refine_used)
                args.refine_used[C.jj] = (uint8_t)((fallback && status == kStOk) ? kAutoSteps + 1 : (steps < 2 ? steps : 2));
            bool nf = !finite64(r2);
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) nf = nf || (j < n && !finite64(m[j]));
            if (status == kStOk && !brk && !fallback && !redo && nf) status = kStNonfinite;
            if (status == kStOk && fallback && !autoref) status = kStRefine;
            if (status == kStOk && redo) status = kStStep2;
#pragma unroll
            for (int j = 0; j < MAXJ; ++j)
                if (j < n) args.mval[args.csr_pos[C.jb + j] + C.poff] = (status == kStOk) ? m[j] : 0.0;
            args.colres[C.jj] = (status == kStOk) ? (r2 > 0.0 ? r2 : 0.0) + out2 : 0.0;
            args.colstat[C.jj] = status;
        }
    }
}

// The adjoint of the columns (adjoint_core.cuh says what it computes): lambda
// from the Cholesky factor with FP64 corrections, w = B lambda and r = c - B m
// in FP64, dL/dB in gather order.  The Cholesky factor contracts an error by
// rho, about u_32 kappa^2 per correction, the QR's by half of that.  Up to rho =
// kAdjRho one correction more than asked for (as many from two on: 1e-15 is left)
// and past it two more leave less error than the QR kernel's; past kAdjRhoMax the
// column goes to rest, for that kernel: a warp of such columns as soon as it has
// its factors.  As the
// forward kernel, bound by FP64 arithmetic.  Measured with the forward kernel
// in place: 32 pairs of 512^2, level 1, two steps, map and adjoint, 70.6 ms with
// the QR tiles' adjoint, 49.3 ms with this one.  The adjoint of four Q1 512^2 maps,
// two steps, QR tiles / this kernel: 7.38 / 4.53 ms; rows scaled by 10^+-1 (rho
// around 1e-3) 7.36 / 5.26; by 10^+-3 (nearly all columns left) 7.35 / 8.19.
constexpr float kAdjRho = 1e-5f, kAdjRhoMax = 1e-2f;

template <class SH, int W>
__global__ void __launch_bounds__(32, SH::WARPS) adjoint_simt_kernel(LsqArgs args, int bin, int32_t *rest,
                                                                    int32_t *rest_off) {
    constexpr int MAXI = SH::MAXI, MAXJ = SH::MAXJ;
    if (args.longest && simt_width(*args.longest) != W) return;
    extern __shared__ __align__(16) float smem_f[];
    const int lane = threadIdx.x;
    double *Wv = reinterpret_cast<double *>(smem_f + 32 * SH::RW) + lane;  // B lambda
    double *R = reinterpret_cast<double *>(smem_f) + lane;                 // r, once L is done with
    double *X = reinterpret_cast<double *>(smem_f + 32 * SH::XD) + lane;   // m, then lambda's column factors
    Simt<SH, W> C(args, smem_f, lane);
    float *S = C.S;
    const int w0 = args.bin_off[bin], total = args.bin_off[bin + 1] - w0;
    const int32_t *work = args.work + w0;
    const double rho = args.resid_weight;
    for (int base = blockIdx.x * 32; base < total; base += gridDim.x * 32) {
        const bool valid = base + lane < total;
        C.begin(work[valid ? base + lane : base]);  // (idle lanes repeat a column and write nothing)
        const int n = C.n;
        C.template gram<false>();
        C.template factor<false>();
        const float rk = (float)(kRhoSafety * kU32) * (C.dmax / C.dmin);
        // columns that the QR kernel has to take; a warp of them is done
        auto leave = [&] { rest[atomicAdd(&rest_off[1], 1)] = C.jj; };
        bool left = C.status == kStOk && (C.brk || !(rk <= kAdjRhoMax));
        if (__all_sync(0xffffffffu, left || !valid)) {
            if (valid) leave();
            continue;
        }
        const int xb = tri(n);
        // ---- lambda = G^{-1} g: w = B lambda grows with it
        double gq[MAXJ], lq[MAXJ];
        float x[MAXJ];
        float l2 = 0.f;
#pragma unroll
        for (int j = 0; j < MAXJ; ++j) {
            gq[j] = (j < n && args.dmval) ? args.dmval[args.csr_pos[C.jb + j] + C.poff] : 0.0;
            x[j] = narrow_trunc(gq[j]);
        }
        for (int i = 0; i < C.imax; ++i) Wv[32 * i] = 0.0;
        Wv[32 * MAXI] = 0.0;
        C.fwd(x);
        C.back(x);
#pragma unroll
        for (int j = 0; j < MAXJ; ++j) {
            lq[j] = widen(x[j]);
            l2 = fmaf(x[j], x[j], l2);
        }
        // this lane's corrections (past them its x is zero and changes nothing:
        // a column's result does not depend on the warp's others)
        int corr = args.refine_steps < 2 ? args.refine_steps + 1 : args.refine_steps;
        for (int step = 0;; ++step) {
            C.store_x(x);
            C.add_bx(Wv, [&](int c) { return c < n ? widen(S[32 * (xb + c)]) : 0.0; });
            if (!__any_sync(0xffffffffu, step < corr)) break;
            // correction: lambda += (L L^T)^{-1} (g - B^T w)
            C.bt_r(Wv, [&](int c, double t) { X[32 * c] = t; });
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) x[j] = j < n && step < corr ? narrow_trunc(gq[j] - X[32 * j]) : 0.f;
            C.fwd(x);
            C.back(x);
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) {
                lq[j] += widen(x[j]);
                s = fmaf(x[j], x[j], s);
            }
            if (step == 0) {  // rho by the first correction as well, 4 |d| / |lambda|
                left = left || (C.status == kStOk && !(16.f * s <= kAdjRhoMax * kAdjRhoMax * l2));
                if (!(rk <= kAdjRho) || !(16.f * s <= kAdjRho * kAdjRho * l2)) corr = args.refine_steps + 2;
                if (left) corr = 0;
            }
        }
        if (valid && left) leave();
        // ---- r = c - B m
#pragma unroll
        for (int j = 0; j < MAXJ; ++j)
            if (j < n) X[32 * j] = args.mval[args.csr_pos[C.jb + j] + C.poff];
        C.target(R);
        C.add_bx(R, [&](int c) { return c < n ? -X[32 * c] : 0.0; });
        const bool write = valid && !left && C.status == kStOk;
        // ---- dL/dB(i, c) = r_i (lambda_c - 2 rho m_c) - w_i m_c, and where each column's block starts
        const int64_t blk = args.dB_off[C.jj];
#pragma unroll
        for (int j = 0; j < MAXJ; ++j)  // (x: lambda in FP64 words is not kept: the factor goes with m)
            if (j < n) X[32 * (MAXJ + j)] = fma(-2.0 * rho, X[32 * j], lq[j]);
        int e0 = 0;
        for (int c = 0; c < C.nmax; ++c) {
            if (c >= n) break;
            const double ac = X[32 * (MAXJ + c)], nm = -X[32 * c];
            const uint8_t *l = C.lrow + c * (32 * W);
            int i[W];
#pragma unroll
            for (int u = 0; u < W; ++u) i[u] = l[32 * u];
            int len = 0;
#pragma unroll
            for (int u = 0; u < W; ++u) {
                const double v = fma(R[32 * i[u]], ac, Wv[32 * i[u]] * nm);
                if (write && i[u] != MAXI) args.dB[blk + e0 + u] = v;
                len += i[u] != MAXI ? 1 : 0;
            }
            if (write) args.dbase[args.csr_pos[C.jb + c] + C.poff] = blk + e0;
            e0 += len;
        }
        if (args.dmres) C.bt_r(R, [&](int c, double t) {
            if (write) args.dmres[args.csr_pos[C.jb + c] + C.poff] = -2.0 * rho * t;
        });
        // ---- dL/dA_0(:, j)
        if (write) {
            const int64_t zoff = args.zbig ? 0 : (int64_t)(C.roff / args.n) * args.znnz;
            for (int t = C.zb; t < C.ze; ++t) {
                const int i = C.target_row(t);
                args.dzval[zoff + t] = (i >= 0) ? Wv[32 * i] + 2.0 * rho * R[32 * i] : 2.0 * rho * args.zcv[t];
            }
        }
        if (valid && !left) args.colstat[C.jj] = C.status;
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

template <class SH, int W>
cudaError_t launch_adjoint(sam_handle h, const LsqArgs &a, int bin) {
    const size_t smem = SH::BYTES;
    auto kern = adjoint_simt_kernel<SH, W>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    kern<<<per_sm * handle_sms(h), 32, smem, handle_stream(h)>>>(a, bin, a.dense_list + bin * a.dense_cap,
                                                                      a.dense_off + 2 * bin);
    count_launch(h);
    return cudaGetLastError();
}

template <int W>
cudaError_t launch_width(sam_handle h, const LsqArgs &args, int bin) {
    switch (bin) {
        case 0: return launch_simt<Simt0, W>(h, args, 0);
        case 1: return launch_simt<Simt1, W>(h, args, 1);
        default: return cudaErrorInvalidValue;
    }
}

__global__ void longest_column_kernel(int n, const int32_t *kcp, int32_t *longest) {
    int m = 0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x)
        m = max(m, kcp[c + 1] - kcp[c]);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(longest, m);
}

__global__ void simt_values_kernel(int n, int W, const int32_t *longest, const int32_t *kcp, int64_t map_nnz,
                                   const double *cv, int64_t ell_map, double *kev, float *kev32) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    if (longest) W = simt_width(*longest);
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
__global__ void __launch_bounds__(256) simt_rows_kernel(int n, int W, const int32_t *longest, const int32_t *kcp,
                                                        const int32_t *jcp, const int32_t *jri, const uint8_t *bin,
                                                        const uint8_t *lrow, uint8_t *lrow_t) {
    __shared__ __align__(4) uint8_t sh[kLTile][32];
    __shared__ int most;
    const int j0 = blockIdx.x * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (longest) W = simt_width(*longest);
    if (!W) return;
    if (threadIdx.x == 0) most = 0;
    __syncthreads();
    for (int q = warp; q < 32; q += 8) {
        const int j = j0 + q;
        const int b = j < n ? bin[j] : kBinNone;
        if (b >= kSimtBins) continue;
        const int pad = b == 0 ? Simt0::MAXI : Simt1::MAXI;  // its shape's padding row
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

cudaError_t launch_lsq_simt_bin(sam_handle h, const LsqArgs &args, int bin) {
    if (args.longest) {
        cudaError_t e;
        if ((e = launch_width<5>(h, args, bin)) != cudaSuccess || (e = launch_width<7>(h, args, bin)) != cudaSuccess ||
            (e = launch_width<9>(h, args, bin)) != cudaSuccess)
            return e;
        return launch_width<kEllW>(h, args, bin);
    }
    switch (args.ell_w) {
        case 5: return launch_width<5>(h, args, bin);
        case 7: return launch_width<7>(h, args, bin);
        case 9: return launch_width<9>(h, args, bin);
        case kEllW: return launch_width<kEllW>(h, args, bin);
        default: return cudaErrorInvalidValue;
    }
}

// the columns of class b left over go to dense_list + b dense_cap, their number
// to dense_off[2 b + 1] (from 0)
cudaError_t launch_adjoint_simt(sam_handle h, const LsqArgs &args) {
    cudaError_t e = cudaErrorInvalidValue;
    auto width = [&](auto w) {
        constexpr int W = decltype(w)::value;
        if (!args.longest && args.ell_w != W) return cudaSuccess;
        if ((e = launch_adjoint<Simt0Adj, W>(h, args, 0)) == cudaSuccess) e = launch_adjoint<Simt1Adj, W>(h, args, 1);
        return e;
    };
    if (width(std::integral_constant<int, 5>()) != cudaSuccess || width(std::integral_constant<int, 7>()) != cudaSuccess ||
        width(std::integral_constant<int, 9>()) != cudaSuccess)
        return e;
    width(std::integral_constant<int, kEllW>());
    return e;
}

cudaError_t longest_column(sam_handle h, int n, const int32_t *kcp, int32_t *longest) {
    if (n == 0) return cudaSuccess;
    longest_column_kernel<<<std::min((n + 255) / 256, 4 * handle_sms(h)), 256, 0, handle_stream(h)>>>(n, kcp, longest);
    count_launch(h);
    return cudaGetLastError();
}

cudaError_t simt_values(sam_handle h, int n, int K, int W, const int32_t *longest, const int32_t *kcp, int64_t map_nnz,
                        const double *cv, int64_t ell_map, double *kev, float *kev32) {
    if (n == 0 || K == 0) return cudaSuccess;
    simt_values_kernel<<<dim3((unsigned)((n + 255) / 256), (unsigned)K), 256, 0, handle_stream(h)>>>(
        n, W, longest, kcp, map_nnz, cv, ell_map, kev, kev32);
    count_launch(h);
    return cudaGetLastError();
}

cudaError_t simt_rows(sam_handle h, int n, int W, const int32_t *longest, const int32_t *kcp, const int32_t *jcp,
                      const int32_t *jri, const uint8_t *bin, const uint8_t *lrow, uint8_t *lrow_t) {
    if (n == 0) return cudaSuccess;
    simt_rows_kernel<<<(unsigned)((n + 31) / 32), 256, 0, handle_stream(h)>>>(n, W, longest, kcp, jcp, jri, bin, lrow,
                                                                             lrow_t);
    count_launch(h);
    return cudaGetLastError();
}

}  // namespace sam
