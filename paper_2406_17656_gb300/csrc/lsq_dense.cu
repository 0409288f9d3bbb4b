// lsq_dense.cu -- the column least-squares solves of SAM construction
// (arXiv 2406.17656, Sec. 2: min_m || A_k(I_j, J_j) m - A_0(I_j, j) ||) of the
// large class in refined FP32 builds (level-3 patterns, sources with many
// entries per column), by an FP32 Cholesky factor of the normal equations: one
// block per column, everything in shared memory.
//
// The refinement needs R only as a preconditioner (lsq_simt.cu): G = B^T B,
// b = B^T c and G = L L^T in FP32, then one corrected step more than the
// build's s, all with r and g in FP64.  Against the Householder QR
// (lsq_big.cu) the dense work drops from 2 n^2 (m - n / 3) to about
// nnz(B) n / 2 + n^3 / 6 multiply-adds, since G's rows are sums over the stored
// entries of B alone, and no reflector waits for another's norm.
#include <cfloat>
#include <climits>

#include "lsq_core.cuh"

namespace sam {
namespace {

__host__ __device__ __forceinline__ int tri(int q) { return q * (q + 1) / 2; }

template <typename V>
__device__ __forceinline__ V wsum(V v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct __align__(16) DenseHdr {
    long long colA[kBigJCap];     // value offset of column c of B (this map's values)
    int kcol[kBigJCap];           // structure offset of column c
    unsigned short cb[kBigJCap + 2];  // first entry of column c in gather order
    float colk[kBigJCap + 4];     // column k of L during the factorisation
    float inv[kBigJCap];          // 1 / L_kk
    float g[kBigJCap];            // B^T r, then the correction
    double x[kBigJCap];           // the vector of the next product B x
    double m[kBigJCap];           // the solution
    double part[32];              // partial sums of the warps
    int scan[32];
    int status, nB, lo, hi, nI, brk, redo, fallback;
    float kap2, msq, da2, dprev2;
    double out2, r2;
};

// The arrays of one column after the header; bytes() is what they take.
struct DenseLayout {
    int nI, n, nB, words, nw, ldb;
    unsigned *bm;            // row bitmap over the span [words]
    unsigned short *pre;     // rows before each word [words]
    unsigned *mask;          // columns present in each row [nI][nw]
    double *r;               // c, then the residual [nI]
    unsigned short *rowstart;  // [nI + 1]
    unsigned short *row;     // local row of every entry, by columns [nB]
    unsigned short *pl;      // entries by rows: their index by columns [nB]
    unsigned char *cl;       // and their column [nB]
    float *L;                // rows 0..n of [G b], then of L, packed
    float *B;                // [B c] dense, rows of ldb floats, until G is formed
    double *val;             // then B's entries by columns [nB], when they fit there
    bool vals;
    __device__ size_t set(unsigned char *base, int nI_, int n_, int nB_, int words_, size_t room) {
        nI = nI_, n = n_, nB = nB_, words = words_;
        nw = (n + 31) >> 5;
        ldb = ((n + 1) + 3) & ~3;
        size_t o = 0;
        auto take = [&](size_t bytes) {
            unsigned char *p = base + o;
            o += (bytes + 15) & ~(size_t)15;
            return p;
        };
        r = (double *)take(sizeof(double) * nI);
        const size_t dense = sizeof(float) * (size_t)nI * ldb, all = sizeof(double) * (size_t)nB;
        B = (float *)take(all > dense && all <= room ? all : dense);
        val = (double *)B;
        vals = all <= room || all <= dense;
        L = (float *)take(sizeof(float) * tri(n + 1));
        bm = (unsigned *)take(sizeof(unsigned) * words);
        pre = (unsigned short *)take(sizeof(unsigned short) * words);
        mask = (unsigned *)take(sizeof(unsigned) * nI * nw);
        rowstart = (unsigned short *)take(sizeof(unsigned short) * (nI + 1));
        row = (unsigned short *)take(sizeof(unsigned short) * nB);
        pl = (unsigned short *)take(sizeof(unsigned short) * nB);
        cl = (unsigned char *)take(nB);
        return o;
    }
};

// One column per block of NT threads.  Columns whose arrays take more than
// `cap` bytes (or whose rows span too far) are appended to rest for the next kernel.
template <int NT>
__global__ void __launch_bounds__(NT) lsq_dense_kernel(LsqArgs args, int bin, unsigned cap, int32_t *rest,
                                                       int32_t *rest_off) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DenseHdr &H = *reinterpret_cast<DenseHdr *>(smem_raw);
    unsigned char *base = smem_raw + sizeof(DenseHdr);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    const int w0 = args.bin_off[bin] + (args.item_hi > 0 ? args.item_lo : 0);
    const int items = args.item_hi > 0 ? args.item_hi - args.item_lo : args.bin_off[bin + 1] - w0;
    const bool sh = args.shadow_shared != 0;
    // a column this launch cannot hold: to the next one, or to the FP64 re-solve
    auto leave = [&](int jj) {
        if (tid != 0) return;
        if (rest) {
            rest[atomicAdd(&rest_off[1], 1)] = jj;
        } else {
            args.colstat[jj] = kStRefine;
            if (args.refine_used) args.refine_used[jj] = kAutoSteps + 1;
        }
    };
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        __syncthreads();  // the last column's shared memory is done with
        const int jj = args.work[w0 + item];
        const int kmap = jj / args.n;
        const int jl = jj - kmap * args.n;
        const int js = sh ? jl : jj;
        const int64_t aoff = sh ? (int64_t)kmap * args.map_nnz_src : 0;
        const int64_t poff = sh ? (int64_t)kmap * args.map_nnz_pat : 0;
        const int roff = kmap * args.n;
        const int zc = args.zbig ? jj : jl;
        const int zro = (sh ? 0 : roff) - (args.zbig ? roff : 0);
        const int jb = args.jcp[js], n = args.jcp[js + 1] - jb;
        const int zb = args.zcp[zc], ze = args.zcp[zc + 1];
        const int nI = args.icnt[js];
        // ---- the columns of J, their first entries and the span of the rows
        if (warp == 0) {
            int run = 0, lo = INT_MAX, hi = -1;
            for (int c0 = 0; c0 < n; c0 += 32) {
                const int c = c0 + lane;
                int len = 0;
                if (c < n && n <= kBigJCap) {
                    const int col = args.jri[jb + c];
                    const int a0 = args.kcp[col];
                    len = args.kcp[col + 1] - a0;
                    H.kcol[c] = a0;
                    H.colA[c] = (long long)a0 + aoff;
                    if (len > 0) {
                        lo = min(lo, args.kri[a0]);
                        hi = max(hi, args.kri[a0 + len - 1]);
                    }
                }
                int incl = len;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (c < n && n <= kBigJCap) H.cb[c + 1] = (unsigned short)min(run + incl, 65535);
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0) {
                H.cb[0] = 0;
                H.nB = run;
                H.lo = lo;
                H.hi = hi;
                H.status = kStOk;
                H.brk = 0;
            }
        }
        __syncthreads();
        const int nB = H.nB, lo = H.lo;
        const int64_t span = (int64_t)H.hi - lo + 1;
        const int words = (int)((span + 31) >> 5);
        DenseLayout D;
        bool take = n <= kBigJCap && nI >= n && nI <= kBigICap && nB <= kBigLCap && words <= (int)cap;
        if (take) {
            // the values stay in shared memory when there is room for them
            const size_t least = D.set(base, nI, n, nB, words, 0);
            take = least <= cap;
            if (take) D.set(base, nI, n, nB, words, cap - least + sizeof(float) * (size_t)nI * D.ldb);
            // (a small block leaves a column whose values do not fit to the large ones)
            take = take && (D.vals || !rest);
        }
        if (!take) {
            leave(jj);
            continue;
        }
        // ---- bitmap of the rows, rows before each word
        for (int w = tid; w < words; w += NT) D.bm[w] = 0u;
        for (int q = tid; q < nI * D.nw; q += NT) D.mask[q] = 0u;
        for (int q = tid; q < nI * D.ldb / 4; q += NT) reinterpret_cast<float4 *>(D.B)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = tid; i < nI; i += NT) D.r[i] = 0.0;
        __syncthreads();
        for (int c = warp; c < n; c += NW) {
            const int a0 = H.kcol[c], len = H.cb[c + 1] - H.cb[c];
            for (int e = lane; e < len; e += 32) {
                const int x = args.kri[a0 + e] - lo;
                atomicOr(&D.bm[x >> 5], 1u << (x & 31));
            }
        }
        __syncthreads();
        if (warp == 0) {
            int run = 0;
            for (int q = 0; q < words; q += 32) {
                const int cnt = q + lane < words ? __popc(D.bm[q + lane]) : 0;
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (q + lane < words) D.pre[q + lane] = (unsigned short)(run + incl - cnt);
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0 && run != nI) H.status = kStUnsupported;  // impossible for a consistent shadow
        }
        __syncthreads();
        if (H.status != kStOk) {
            leave(jj);
            continue;
        }
        auto rank = [&](int x) { return (int)D.pre[x >> 5] + __popc(D.bm[x >> 5] & ((1u << (x & 31)) - 1u)); };
        // ---- [B c] dense in FP32, local rows, row masks; c in FP64
        for (int c = warp; c < n; c += NW) {
            const int a0 = H.kcol[c], p0 = H.cb[c], len = H.cb[c + 1] - p0;
            for (int e = lane; e < len; e += 32) {
                const int i = rank(args.kri[a0 + e] - lo);
                D.row[p0 + e] = (unsigned short)i;
                D.B[i * D.ldb + c] = args.kcv32[H.colA[c] + e];
                atomicOr(&D.mask[i * D.nw + (c >> 5)], 1u << (c & 31));
            }
        }
        if (warp == NW - 1) {
            double o2 = 0.0;
            for (int t = zb + lane; t < ze; t += 32) {
                const int x = args.zri[t] + zro - lo;
                const double v = args.zcv[t];
                const bool in = x >= 0 && x < span && ((D.bm[x >> 5] >> (x & 31)) & 1u);
                if (in) {
                    const int i = rank(x);
                    D.r[i] = v;
                    D.B[i * D.ldb + n] = args.zcv32[t];
                } else {
                    o2 = fma(v, v, o2);
                }
            }
            o2 = wsum(o2);
            if (lane == 0) H.out2 = o2;
        }
        __syncthreads();
        // ---- G = B^T B (its lower triangle) and b = B^T c, row c of G from the
        // dense rows of column c's entries: lanes take four columns each
        {
            const int HW = n + 1 <= 64 ? 16 : 32;  // lanes per row of G
            const int sub = lane / HW, k4 = lane % HW, per = 32 / HW;
            for (int c = warp * per + sub; c <= n; c += NW * per) {
                const int p0 = c < n ? H.cb[c] : 0, len = c < n ? H.cb[c + 1] - p0 : nI;
                if (4 * k4 <= c && 4 * k4 < n) {
                    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                    for (int e = 0; e < len; ++e) {
                        const float *b = D.B + (c < n ? (int)D.row[p0 + e] : e) * D.ldb;
                        const float v = b[c];
                        const float4 w = *reinterpret_cast<const float4 *>(b + 4 * k4);
                        a.x = fmaf(v, w.x, a.x);
                        a.y = fmaf(v, w.y, a.y);
                        a.z = fmaf(v, w.z, a.z);
                        a.w = fmaf(v, w.w, a.w);
                    }
                    float *g = D.L + tri(c) + 4 * k4;
                    const int m = min(c, n - 1) - 4 * k4;  // columns up to min(c, n - 1)
                    g[0] = a.x;
                    if (m >= 1) g[1] = a.y;
                    if (m >= 2) g[2] = a.z;
                    if (m >= 3) g[3] = a.w;
                    if (c < n && 4 * k4 + 3 >= c) {  // the diagonal: a zero column is rank deficient
                        const float d = c - 4 * k4 == 0 ? a.x : c - 4 * k4 == 1 ? a.y : c - 4 * k4 == 2 ? a.z : a.w;
                        if (d == 0.f) atomicMax(&H.status, (int)kStRank);
                    }
                }
            }
        }
        __syncthreads();
        // ---- entries by rows; values in FP64 in the place of the dense rows
        if (warp == 0) {
            int run = 0;
            for (int q = 0; q < nI; q += 32) {
                int cnt = 0;
                if (q + lane < nI)
                    for (int w = 0; w < D.nw; ++w) cnt += __popc(D.mask[(q + lane) * D.nw + w]);
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (q + lane < nI) D.rowstart[q + lane] = (unsigned short)(run + incl - cnt);
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) D.rowstart[nI] = (unsigned short)run;
        }
        __syncthreads();
        for (int c = warp; c < n; c += NW) {
            const int p0 = H.cb[c], len = H.cb[c + 1] - p0;
            for (int e = lane; e < len; e += 32) {
                const int i = D.row[p0 + e];
                int pos = D.rowstart[i] + __popc(D.mask[i * D.nw + (c >> 5)] & ((1u << (c & 31)) - 1u));
                for (int w = 0; w < (c >> 5); ++w) pos += __popc(D.mask[i * D.nw + w]);
                D.pl[pos] = (unsigned short)(p0 + e);
                D.cl[pos] = (unsigned char)c;
                if (D.vals) D.val[p0 + e] = args.kcv[H.colA[c] + e];
            }
        }
        // ---- G = L L^T; the row of b becomes y = L^{-1} b
        float dmax = 0.f, dmin = FLT_MAX;
        bool brk = false;
        for (int k = 0; k < n; ++k) {
            const float d = D.L[tri(k) + k];
            if (!brk && !(fabsf(d) <= FLT_MAX) && tid == 0) atomicMax(&H.status, (int)kStNonfinite);
            brk = brk || !(d > 0.f);
            dmax = fmaxf(dmax, d);
            dmin = fminf(dmin, d);
            const float inv = rsqrtf(d);
            for (int i = k + 1 + tid; i <= n; i += NT) {
                const float v = D.L[tri(i) + k] * inv;
                D.L[tri(i) + k] = v;
                H.colk[i] = v;
            }
            if (tid == 0) H.inv[k] = inv;
            __syncthreads();
            float lj[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int j = k + 1 + lane + 32 * t;
                lj[t] = j < n ? H.colk[j] : 0.f;
            }
            for (int i = k + 1 + warp; i <= n; i += NW) {
                const float li = H.colk[i];
                float *Li = D.L + tri(i);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int j = k + 1 + lane + 32 * t;
                    if (j <= i && j < n) Li[j] = fmaf(-li, lj[t], Li[j]);
                }
            }
            __syncthreads();
        }
        const float kap2 = dmax / dmin;
        // triangular solves by warp 0: entries c = lane + 32 t in x[]
        float x[4];
        auto back = [&]() {  // L^T x = y
            for (int k = n - 1; k >= 0; --k) {
                const int t0 = k >> 5;
                float xk = (t0 == 0 ? x[0] : t0 == 1 ? x[1] : t0 == 2 ? x[2] : x[3]) * H.inv[k];
                xk = __shfl_sync(0xffffffffu, xk, k & 31);
                const float *Lk = D.L + tri(k);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = lane + 32 * t;
                    if (c < k) x[t] = fmaf(-Lk[c], xk, x[t]);
                    else if (c == k) x[t] = xk;
                }
            }
        };
        auto fwd = [&]() {  // L y = g
            for (int k = 0; k < n; ++k) {
                const int t0 = k >> 5;
                float yk = (t0 == 0 ? x[0] : t0 == 1 ? x[1] : t0 == 2 ? x[2] : x[3]) * H.inv[k];
                yk = __shfl_sync(0xffffffffu, yk, k & 31);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = lane + 32 * t;
                    if (c > k && c < n) x[t] = fmaf(-D.L[tri(c) + k], yk, x[t]);
                    else if (c == k) x[t] = yk;
                }
            }
        };
        if (warp == 0) {
            float m2 = 0.f;
#pragma unroll
            for (int t = 0; t < 4; ++t) x[t] = lane + 32 * t < n ? D.L[tri(n) + lane + 32 * t] : 0.f;
            back();
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int c = lane + 32 * t;
                if (c < n) {
                    H.x[c] = H.m[c] = widen(x[t]);
                    m2 = fmaf(x[t], x[t], m2);
                }
            }
            m2 = wsum(m2);
            if (lane == 0) {
                H.msq = m2;
                H.fallback = brk ? 1 : 0;
                H.redo = 0;
            }
        }
        const bool autoref = args.refine_steps < 0;
        // (automatic: the second step in place: it costs the block alone)
        const int steps = autoref ? kAutoSteps : args.refine_steps;
        int used = 0;
        for (int step = 0; step <= steps; ++step) {
            __syncthreads();
            // r -= B x (FP64), a row per thread, its entries by columns
            double rs = 0.0;
            for (int i = tid; i < nI; i += NT) {
                double ri = D.r[i];
                const int e1 = D.rowstart[i + 1];
                if (D.vals) {
#pragma unroll 4
                    for (int e = D.rowstart[i]; e < e1; ++e) ri = fma(-D.val[D.pl[e]], H.x[D.cl[e]], ri);
                } else {
                    for (int e = D.rowstart[i]; e < e1; ++e) {
                        const int c = D.cl[e];
                        ri = fma(-args.kcv[H.colA[c] + (D.pl[e] - H.cb[c])], H.x[c], ri);
                    }
                }
                D.r[i] = ri;
                rs = fma(ri, ri, rs);
            }
            rs = wsum(rs);
            if (lane == 0) H.part[warp] = rs;
            __syncthreads();
            // g = B^T r (FP64, rounded to FP32), eight lanes per column
            for (int c = tid >> 3; c < ((n + 3) & ~3); c += NT / 8) {
                double a0 = 0.0;
                if (c < n) {
                    const int p1 = H.cb[c + 1];
                    const int p0 = H.cb[c];
                    if (D.vals)
                        for (int p = p0 + (lane & 7); p < p1; p += 8) a0 = fma(D.val[p], D.r[D.row[p]], a0);
                    else
                        for (int p = p0 + (lane & 7); p < p1; p += 8)
                            a0 = fma(args.kcv[H.colA[c] + (p - p0)], D.r[D.row[p]], a0);
                }
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                if (c < n && (lane & 7) == 0) H.g[c] = narrow_trunc(a0);
            }
            __syncthreads();
            if (warp == 0) {
#pragma unroll
                for (int t = 0; t < 4; ++t) x[t] = lane + 32 * t < n ? H.g[lane + 32 * t] : 0.f;
                fwd();
                back();
                float dsq = 0.f, dg = 0.f;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = lane + 32 * t;
                    if (c < n) {
                        H.x[c] = widen(x[t]);
                        H.m[c] += H.x[c];
                        dsq = fmaf(x[t], x[t], dsq);
                        dg = fmaf(x[t], H.g[c], dg);
                    }
                }
                dsq = wsum(dsq);
                dg = wsum(dg);
                if (lane == 0) {
                    constexpr float kTol = (float)kFallbackTol, kTol2 = kTol * kTol, kC = (float)kAutoC;
                    const float msq = H.msq;
                    if (step == 0) H.da2 = dsq;
                    const float da2 = H.da2;
                    const float rk = (float)(kRhoSafety * kU32) * kap2;
                    bool miss = !(rk < 0.5f) || rk * rk * dsq > kTol2 * (1.f - rk) * (1.f - rk) * msq;
                    miss = miss || 4.f * kC * kC * da2 >= msq || 4.f * kC * kC * da2 * dsq > kTol2 * msq * msq;
                    if (step > 0 && dsq > (float)kNoise2 * msq) {
                        const float dprev2 = H.dprev2;
                        miss = miss || 4.f * dsq >= dprev2 || 4.f * dsq * dsq > kTol2 * msq * dprev2;
                    }
                    H.dprev2 = dsq;
                    // automatic: the second step when the first left too much
                    const bool more = autoref && step == 1 && (kC * dsq > (float)kAutoTol * msq || miss);
                    H.redo = step < (autoref ? 1 : steps) || more;
                    if (!H.redo) {
                        H.fallback = H.fallback || miss;
                        double r2 = 0.0;
                        for (int w = 0; w < NW; ++w) r2 += H.part[w];
                        H.r2 = r2 - widen(dg);  // ||r - B d||^2 = ||r||^2 - d.g (g = B^T r = G d up to rounding)
                    }
                }
            }
            __syncthreads();
            used = step;
            if (!H.redo) break;
        }
        // ---- outputs
        if (warp == 0) {
            int status = H.status;
            int nf = !finite64(H.r2);
            for (int c = lane; c < n; c += 32) nf |= !finite64(H.m[c]);
            nf = __any_sync(0xffffffffu, nf);
            const bool fallback = H.fallback != 0;
            if (status == kStOk && !fallback && nf) status = kStNonfinite;
            if (status == kStOk && fallback) status = kStRefine;  // re-solved by the FP64 kernel
            for (int c = lane; c < n; c += 32)
                args.mval[(int64_t)args.csr_pos[jb + c] + poff] = status == kStOk ? H.m[c] : 0.0;
            if (lane == 0) {
                args.colres[jj] = status == kStOk ? (H.r2 > 0.0 ? H.r2 : 0.0) + H.out2 : 0.0;
                args.colstat[jj] = status;
                if (args.refine_used)
                    args.refine_used[jj] = (uint8_t)(status == kStRefine ? kAutoSteps + 1 : (used < 2 ? used : 2));
            }
        }
    }
}

template <int NT>
cudaError_t launch_dense(sam_handle h, const LsqArgs &a, int bin, int per_sm, int32_t *rest, int32_t *rest_off) {
    // the shared memory of an SM split over per_sm blocks (1 KB of each is the system's)
    const size_t smem = (size_t)((per_sm == 1 ? 232448 : 233472 / per_sm - 1024) & ~127);
    auto kern = lsq_dense_kernel<NT>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<handle_sms(h) * per_sm, NT, smem, handle_stream(h)>>>(a, bin, (unsigned)(smem - sizeof(DenseHdr)), rest, rest_off);
    count_launch(h);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_lsq_dense(sam_handle h, const LsqArgs &args, int bin) {
    // small columns by small blocks, the others by one block per SM
    cudaError_t e = cudaMemsetAsync(args.dense_off, 0, sizeof(int32_t) * 2, handle_stream(h));
    if (e != cudaSuccess) return e;
    profile_begin(h, bin);
    if ((e = launch_dense<128>(h, args, bin, 7, args.dense_list, args.dense_off)) != cudaSuccess) return e;
    LsqArgs a = args;
    a.item_lo = a.item_hi = 0;
    a.work = args.dense_list;
    a.bin_off = args.dense_off;
    if ((e = launch_dense<512>(h, a, 0, 1, nullptr, nullptr)) != cudaSuccess) return e;
    profile_end(h, bin);
    return cudaSuccess;
}

}  // namespace sam
