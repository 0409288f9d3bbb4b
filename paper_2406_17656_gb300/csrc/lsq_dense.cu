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
//
// Where the time goes (clock64 timers in an instrumented copy, 81 x 49 columns of
// Q1 level-3 maps, seven blocks per SM): factorisation 28%, triangular solves 16%,
// row index and scatter 16%, Gram matrix 9%, the FP64 passes 14%.  The
// factorisation is one warp's for up to 52 unknowns: it needs no block barrier
// per pivot, as a tile over four warps did, and repeats no warp's bookkeeping.
// Shared memory decides the blocks per SM: the dense FP32 rows of [B c] live
// only until G exists, then the row lists and B's FP64 values take their place.
// 128 threads per small block: 96 cost 1%, 64 cost 23%.  Counters of one launch
// (small blocks, 81 x 49 columns): 32,000 warp instructions per column, issue 42%,
// shared memory pipe 43%, FP64 pipe 19%, 7.5 of a warp's 15.3 cycles per instruction
// at a block barrier, which is the warps that wait for the one that factors.
//
// Measured: Q1 256^2, 2 maps, level 3, the whole call: 60.1 -> 8.6 ms; 7,700
// columns of up to 201 x 96 with 7,300 entries, 2 maps: 47.8 -> 15.3 ms.
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

template <int MAXJ>
struct __align__(16) DenseHdr {
    long long colA[MAXJ];     // value offset of column c of B (this map's values)
    int kcol[MAXJ];           // structure offset of column c
    unsigned short cb[MAXJ + 2];  // first entry of column c in gather order
    float inv[MAXJ];          // 1 / L_kk
    double g[MAXJ];           // B^T r
    double x[MAXJ];           // the vector of the next product B x
    double m[MAXJ];           // the solution
    int status, nB, lo, hi, nI, brk, redo, fallback, gexp;
    float kap2, msq, da2, dprev2;
    double out2, r2;
};

// A column whose rows span at most this finds their ranks in a bitmap (6 bytes
// per 32 rows of the span, 6 KB at most); past it the rows are sorted, 4 bytes
// each, so that the footprint does not grow with the numbering (the shadow pass
// takes at most 1024 entries there).  With the bitmap alone a permuted Q1 512^2,
// level 3 (span 262,144), filled a block's memory with it: 141.6 ms, sorted
// 24.9; 128^3 27-point, level 1 (span 65,700): 659 ms, sorted 214.
constexpr int kBitmapRows = 32768;

// The arrays of one column after the header; bytes() is what they take.
struct DenseLayout {
    int nI, n, nB, words, nw, ldb;
    unsigned *bm;            // row bitmap over the span [words]
    unsigned short *pre;     // rows before each word [words]
    int *I;                  // or (wide) the sorted rows [nI]
    unsigned *mask;          // columns present in each row [nI][nw]
    double *r;               // c, then the residual [nI]
    unsigned short *rowstart;  // [nI + 1]
    unsigned short *row;     // local row of every entry, by columns [nB]
    float *L;                // rows 0..n of [G b], then of L, packed
    float *B;                // [B c] dense, rows of ldb floats, until G is formed; then there
    unsigned short *pl;      // the entries by rows: their index by columns [nB]
    unsigned char *cl;       // their column [nB]
    double *val;             // and, when there is room (vals), B's entries by columns [nB]
    int *keys;               // (wide) and before B the entries' rows, padded to a power of two [p2]
    bool vals;
    size_t least;            // bytes of that place without the values
    // words = 0: wide
    __device__ size_t set(unsigned char *base, int nI_, int n_, int nB_, int words_, int p2, size_t room) {
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
        const size_t dense = sizeof(float) * (size_t)nI * ldb, v8 = sizeof(double) * (size_t)nB;
        const size_t lists = ((3 * (size_t)nB + 15) & ~(size_t)15), all = v8 + lists;
        least = dense > lists ? dense : lists;
        if (words == 0 && least < sizeof(int) * (size_t)p2) least = sizeof(int) * (size_t)p2;
        vals = all <= (least > room ? least : room);
        unsigned char *u = take(vals && all > least ? all : least);
        B = (float *)u;
        keys = (int *)u;
        pl = (unsigned short *)u;
        cl = u + 2 * nB;
        val = (double *)(u + lists);
        L = (float *)take(sizeof(float) * tri(n + 1));
        bm = (unsigned *)take(sizeof(unsigned) * (words ? words : nI));
        I = (int *)bm;
        pre = (unsigned short *)take(sizeof(unsigned short) * words);
        mask = (unsigned *)take(sizeof(unsigned) * nI * nw);
        rowstart = (unsigned short *)take(sizeof(unsigned short) * (nI + 1));
        row = (unsigned short *)take(sizeof(unsigned short) * nB);
        return o;
    }
};

// Blocks of NT threads, BLOCKS per SM.  The factorisation runs on the first GT
// threads as a TY x TX grid over RS TY rows (G's and b) and CS TX columns.
template <int NT_, int BLOCKS_, int GT_, int TX_, int RS_, int CS_>
struct DenseShape {
    static constexpr int NT = NT_, BLOCKS = BLOCKS_, GT = GT_, TX = TX_, TY = GT_ / TX_, RS = RS_, CS = CS_;
    static constexpr int MAXJ = TY * RS - 1 < TX * CS ? TY * RS - 1 : TX * CS;
    static constexpr int XS = (MAXJ + 31) / 32;  // unknowns per lane in the solves
    // the pivot column in shared memory, once by rows and once by columns: a
    // thread's values are contiguous (padded to whole 16-byte chunks)
    static constexpr int RP = (RS + 3) & ~3, CP = (CS + 3) & ~3, UW = TY * RP + TX * CP;
};
using DenseSmall = DenseShape<128, 7, 32, 4, 7, 13>;   // up to 52 unknowns
using DenseMedium = DenseShape<128, 3, 128, 8, 9, 16>;  // up to 128
using DenseHalf = DenseShape<256, 2, 32, 4, 7, 13>;    // up to 52
using DenseLarge = DenseShape<512, 1, 128, 8, 9, 16>;  // up to 128
static_assert(DenseSmall::UW % 4 == 0 && DenseLarge::UW % 4 == 0, "alignment");
static_assert(DenseSmall::MAXJ == 52 && DenseLarge::MAXJ == kBigJCap, "shapes");

// the threads of the factorisation (named barrier 1 when they are several warps)
template <class SH>
__device__ __forceinline__ void group_sync() {
    if constexpr (SH::GT == 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"n"(SH::GT) : "memory");
}

struct Pivots {
    float dmax, dmin;
    bool brk;
    int status;
};

// Pivots k = TX T0 .. TX T0 + TX - 1 and on: right-looking, thread (ty, tx)
// holding rows ty + TY q of columns tx + TX t (the blocks that reach the
// lower triangle).  The pivot column goes unscaled through ub (double-buffered),
// one barrier per pivot; row n is b.  Elements past row or column n are never
// used, so nothing tests for them; a finished column keeps its unscaled values.
template <class SH, int T0>
__device__ __forceinline__ void factor_from(float (&a)[SH::RS][SH::CS], float *ub, float *invs, int n, int tx, int ty,
                                            Pivots &pv) {
    constexpr int TX = SH::TX, TY = SH::TY, RS = SH::RS, CS = SH::CS, RP = SH::RP, CP = SH::CP, Q0 = TX * T0 / TY;
    if constexpr (T0 < CS) {
        if (TX * T0 >= n) return;
        for (int kk = 0; kk < TX; ++kk) {
            const int k = TX * T0 + kk;
            if (k >= n) return;
            float *ur = ub + (k & 1) * SH::UW, *uc = ur + TY * RP;
            if (tx == kk) {
#pragma unroll
                for (int q = Q0; q < RS; ++q) {
                    const int i = ty + TY * q;
                    ur[ty * RP + q] = a[q][T0];
                    if (i < TX * CS) uc[(i % TX) * CP + i / TX] = a[q][T0];
                }
            }
            group_sync<SH>();
            const float d = uc[kk * CP + T0];
            if (!pv.brk && !(fabsf(d) <= FLT_MAX)) pv.status = kStNonfinite;  // (past a breakdown every pivot is NaN)
            pv.brk = pv.brk || !(d >= FLT_MIN);  // (1 / d of a subnormal d overflows: the re-solve decides)
            pv.dmax = fmaxf(pv.dmax, d);
            pv.dmin = fminf(pv.dmin, d);
            const float inv = rsqrtf(d), ninv2 = -inv * inv;
            if (tx == kk && ty == 0) invs[k] = inv;
            float ui[RP], uj[CP];
#pragma unroll
            for (int q = Q0 / 4; q < RP / 4; ++q) *reinterpret_cast<float4 *>(ui + 4 * q) = *reinterpret_cast<const float4 *>(ur + ty * RP + 4 * q);
#pragma unroll
            for (int t = T0 / 4; t < CP / 4; ++t) *reinterpret_cast<float4 *>(uj + 4 * t) = *reinterpret_cast<const float4 *>(uc + tx * CP + 4 * t);
#pragma unroll
            for (int q = Q0; q < RS; ++q) ui[q] *= ninv2;
            // (rows and columns up to k keep their values)
            if (ty + TY * Q0 <= k) ui[Q0] = 0.f;
            if constexpr (Q0 + 1 < RS && TY < TX) {
                if (ty + TY * (Q0 + 1) <= k) ui[Q0 + 1] = 0.f;
            }
            if (tx <= kk) uj[T0] = 0.f;
#pragma unroll
            for (int t = T0; t < CS; ++t)
#pragma unroll
                for (int q = Q0; q < RS; ++q)
                    if (TY * q + TY - 1 >= TX * t) a[q][t] = fmaf(ui[q], uj[t], a[q][t]);
        }
        factor_from<SH, T0 + 1>(a, ub, invs, n, tx, ty, pv);
    }
}

// One column per block of NT threads.  Columns whose arrays take more than
// `cap` bytes are appended to rest for the next launch.
template <class SH>
__global__ void __launch_bounds__(SH::NT, SH::BLOCKS) lsq_dense_kernel(LsqArgs args, int bin, unsigned cap, int32_t *rest,
                                                       int32_t *rest_off) {
    constexpr int NT = SH::NT, NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using Hdr = DenseHdr<SH::MAXJ>;
    Hdr &H = *reinterpret_cast<Hdr *>(smem_raw);
    float *ub = reinterpret_cast<float *>(smem_raw + sizeof(Hdr));  // the factorisation's pivot column
    unsigned char *base = smem_raw + sizeof(Hdr) + 8 * SH::UW;
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
                if (c < n && n <= SH::MAXJ) {
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
                if (c < n && n <= SH::MAXJ) H.cb[c + 1] = (unsigned short)min(run + incl, 65535);
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
        const bool wide = span > kBitmapRows;
        const int words = wide ? 0 : (int)((span + 31) >> 5);
        int p2 = 1;
        if (wide)
            while (p2 < nB) p2 <<= 1;
        DenseLayout D;
        bool take = n <= SH::MAXJ && nI >= n && nI <= kBigICap && nB <= kBigLCap;
        if (take) {
            // the values stay in shared memory when there is room for them
            const size_t least = D.set(base, nI, n, nB, words, p2, 0);
            take = least <= cap;
            if (take) D.set(base, nI, n, nB, words, p2, cap - least + D.least);
            // (a small block leaves a column whose values do not fit to the large ones)
            take = take && (D.vals || !rest);
        }
        if (!take) {
            leave(jj);
            continue;
        }
        if (wide) {
            // ---- the rows sorted (bitonic), each once
            for (int c = warp; c < n; c += NW) {
                const int a0 = H.kcol[c], p0 = H.cb[c], len = H.cb[c + 1] - p0;
                for (int e = lane; e < len; e += 32) D.keys[p0 + e] = args.kri[a0 + e];
            }
            for (int q = nB + tid; q < p2; q += NT) D.keys[q] = INT_MAX;
            __syncthreads();
            for (int k = 2; k <= p2; k <<= 1)
                for (int j = k >> 1; j > 0; j >>= 1) {
                    for (int q = tid; q < p2 / 2; q += NT) {
                        const int a = 2 * q - (q & (j - 1)), b = a + j;  // the pair's elements
                        const int x = D.keys[a], y = D.keys[b];
                        if ((x > y) == ((a & k) == 0)) {
                            D.keys[a] = y;
                            D.keys[b] = x;
                        }
                    }
                    __syncthreads();
                }
            if (warp == 0) {
                int run = 0;
                for (int q0 = 0; q0 < p2; q0 += 32) {
                    const int q = q0 + lane;
                    const int x = q < p2 ? D.keys[q] : INT_MAX;
                    const bool first = x != INT_MAX && (q == 0 || D.keys[q - 1] != x);
                    const unsigned m = __ballot_sync(0xffffffffu, first);
                    const int pos = run + __popc(m & ((1u << lane) - 1u));
                    if (first && pos < nI) D.I[pos] = x;
                    run += __popc(m);
                }
                if (lane == 0 && run != nI) H.status = kStUnsupported;  // impossible for a consistent shadow
            }
            __syncthreads();
        }
        for (int w = tid; w < words; w += NT) D.bm[w] = 0u;
        for (int q = tid; q < nI * D.nw; q += NT) D.mask[q] = 0u;
        for (int q = tid; q < nI * D.ldb / 4; q += NT) reinterpret_cast<float4 *>(D.B)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = tid; i < nI; i += NT) D.r[i] = 0.0;
        __syncthreads();
        if (!wide) {
            // ---- bitmap of the rows, rows before each word
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
        }
        if (H.status != kStOk) {
            leave(jj);
            continue;
        }
        // the local row of a row of the shadow; of any row, -1 when it is none
        auto rank = [&](int row) {
            if (wide) return find_sorted(D.I, nI, row);
            const int x = row - lo;
            return (int)D.pre[x >> 5] + __popc(D.bm[x >> 5] & ((1u << (x & 31)) - 1u));
        };
        auto find = [&](int row) {
            const int x = row - lo;
            return wide || (x >= 0 && x < span && ((D.bm[x >> 5] >> (x & 31)) & 1u)) ? rank(row) : -1;
        };
        // ---- [B c] dense in FP32, local rows, row masks; c in FP64
        for (int c = warp; c < n; c += NW) {
            const int a0 = H.kcol[c], p0 = H.cb[c], len = H.cb[c + 1] - p0;
            for (int e = lane; e < len; e += 32) {
                const int i = rank(args.kri[a0 + e]);
                D.row[p0 + e] = (unsigned short)i;
                D.B[i * D.ldb + c] = args.kcv32[H.colA[c] + e];
                atomicOr(&D.mask[i * D.nw + (c >> 5)], 1u << (c & 31));
            }
        }
        if (warp == NW - 1) {
            double o2 = 0.0;
            for (int t = zb + lane; t < ze; t += 32) {
                const int i = find(args.zri[t] + zro);
                const double v = args.zcv[t];
                if (i >= 0) {
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
                    if (c < n && 4 * k4 + 3 >= c) {
                        // the diagonal: a column of zeros is rank deficient; one
                        // whose squares vanish in FP32 breaks the factor down
                        const float d = c - 4 * k4 == 0 ? a.x : c - 4 * k4 == 1 ? a.y : c - 4 * k4 == 2 ? a.z : a.w;
                        if (d == 0.f) {
                            bool zero = true;
                            for (int e = 0; e < len; ++e) zero = zero && D.B[(int)D.row[p0 + e] * D.ldb + c] == 0.f;
                            if (zero) atomicMax(&H.status, (int)kStRank);
                        }
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
        __syncthreads();
        if (tid < SH::GT) {
            constexpr int TX = SH::TX, TY = SH::TY, RS = SH::RS, CS = SH::CS;
            const int tx = tid % TX, ty = tid / TX;
            float a[RS][CS];
#pragma unroll
            for (int q = 0; q < RS; ++q)
#pragma unroll
                for (int t = 0; t < CS; ++t) {
                    const int i = ty + TY * q, j = tx + TX * t;
                    a[q][t] = TY * q + TY - 1 >= TX * t && i <= n && j <= i && j < n ? D.L[tri(i) + j] : 0.f;
                }
            Pivots pv{0.f, FLT_MAX, false, kStOk};
            factor_from<SH, 0>(a, ub, H.inv, n, tx, ty, pv);
            group_sync<SH>();
#pragma unroll
            for (int t = 0; t < CS; ++t) {
                const int j = tx + TX * t;
                const float inv = j < n ? H.inv[j] : 0.f;
#pragma unroll
                for (int q = 0; q < RS; ++q) {
                    const int i = ty + TY * q;
                    if (TY * q + TY - 1 >= TX * t && i <= n && j < i && j < n) D.L[tri(i) + j] = a[q][t] * inv;
                }
            }
            if (tid == 0) {
                if (pv.status != kStOk) H.status = max(H.status, pv.status);
                H.brk = pv.brk ? 1 : 0;
                H.kap2 = pv.dmax / pv.dmin;  // a lower bound on kappa(B)^2
                H.gexp = ((__float_as_int(pv.dmax) >> 23) & 0xff) - 127;
            }
            group_sync<SH>();
        }
        // triangular solves by warp 0: entries c = lane + 32 t in x[].  The
        // chain of a step is a product, a shuffle and a multiply-add; L's
        // elements are loaded a step ahead
        constexpr int XS = SH::XS;
        float x[XS], iv[XS];
        auto back = [&]() {  // L^T x = y
#pragma unroll
            for (int t0 = XS - 1; t0 >= 0; --t0) {
                if (32 * t0 >= n) continue;
                const int kh = min(32 * t0 + 31, n - 1);
                float l[XS], ln[XS];
#pragma unroll
                for (int t = 0; t <= t0; ++t) l[t] = lane + 32 * t < kh ? D.L[tri(kh) + lane + 32 * t] : 0.f;
#pragma unroll 4
                for (int k = kh; k >= 32 * t0; --k) {
                    const int k1 = max(k - 1, 0);
#pragma unroll
                    for (int t = 0; t <= t0; ++t) ln[t] = lane + 32 * t < k1 ? D.L[tri(k1) + lane + 32 * t] : 0.f;
                    const float xk = __shfl_sync(0xffffffffu, x[t0] * iv[t0], k & 31);
#pragma unroll
                    for (int t = 0; t <= t0; ++t) {
                        x[t] = fmaf(-l[t], xk, x[t]);
                        l[t] = ln[t];
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < XS; ++t) x[t] *= iv[t];
        };
        auto fwd = [&]() {  // L y = g
            int b[XS];
#pragma unroll
            for (int t = 0; t < XS; ++t) b[t] = tri(lane + 32 * t);
#pragma unroll
            for (int t0 = 0; t0 < XS; ++t0) {
                if (32 * t0 >= n) continue;
                const int ke = min(32 * t0 + 32, n);
                float l[XS], ln[XS];
                auto load = [&](float (&o)[XS], int k) {
#pragma unroll
                    for (int t = t0; t < XS; ++t) o[t] = lane + 32 * t > k && lane + 32 * t < n ? D.L[b[t] + k] : 0.f;
                };
                load(l, 32 * t0);
#pragma unroll 4
                for (int k = 32 * t0; k < ke; ++k) {
                    load(ln, k + 1);
                    const float yk = __shfl_sync(0xffffffffu, x[t0] * iv[t0], k & 31);
#pragma unroll
                    for (int t = t0; t < XS; ++t) {
                        x[t] = fmaf(-l[t], yk, x[t]);
                        l[t] = ln[t];
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < XS; ++t) x[t] *= iv[t];
        };
        if (warp == 0) {
            float m2 = 0.f;
#pragma unroll
            for (int t = 0; t < XS; ++t) iv[t] = lane + 32 * t < n ? H.inv[lane + 32 * t] : 0.f;
#pragma unroll
            for (int t = 0; t < XS; ++t) x[t] = lane + 32 * t < n ? D.L[tri(n) + lane + 32 * t] : 0.f;
            back();
#pragma unroll
            for (int t = 0; t < XS; ++t) {
                const int c = lane + 32 * t;
                if (c < n) {
                    H.x[c] = H.m[c] = widen(x[t]);
                    m2 = fmaf(x[t], x[t], m2);
                }
            }
            m2 = wsum(m2);
            if (lane == 0) {
                H.msq = m2;
                H.fallback = H.brk;
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
            }
            __syncthreads();
            // g = B^T r (FP64), eight lanes per column
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
                if (c < n && (lane & 7) == 0) H.g[c] = a0;
            }
            __syncthreads();
            if (warp == 0) {
                // g rounded to FP32, scaled by the power of two that takes it to
                // the size of G's pivots: on its own g is far smaller than G
                // (by |r| / |B|) and below FP32's range where G is not yet
                unsigned top = 0u;
#pragma unroll
                for (int t = 0; t < XS; ++t) {
                    const int c = lane + 32 * t;
                    if (c < n) top = max(top, (unsigned)__double2hiint(H.g[c]) & 0x7fffffffu);
                }
                top = __reduce_max_sync(0xffffffffu, top) >> 20;
                const int up = top == 0u || top == 0x7ffu ? 0 : min(max(H.gexp - 1 - ((int)top - 1023), -1000), 1000);
                const double sup = __hiloint2double((1023 + up) << 20, 0), sdown = __hiloint2double((1023 - up) << 20, 0);
#pragma unroll
                for (int t = 0; t < XS; ++t) x[t] = lane + 32 * t < n ? narrow_trunc(H.g[lane + 32 * t] * sup) : 0.f;
                fwd();
                back();
                float dsq = 0.f;
                double dg = 0.0;
#pragma unroll
                for (int t = 0; t < XS; ++t) {
                    const int c = lane + 32 * t;
                    if (c < n) {
                        const double d = widen(x[t]) * sdown;
                        x[t] = narrow_trunc(d);
                        H.x[c] = d;
                        H.m[c] += d;
                        dsq = fmaf(x[t], x[t], dsq);
                        dg = fma(d, H.g[c], dg);
                    }
                }
                dsq = wsum(dsq);
                constexpr float kTol = (float)kFallbackTol, kTol2 = kTol * kTol, kC = (float)kAutoC;
                const float msq = H.msq, da2 = step == 0 ? dsq : H.da2, dprev2 = H.dprev2;
                const float rk = (float)(kRhoSafety * kU32) * H.kap2;
                bool miss = !(rk < 0.5f) || rk * rk * dsq > kTol2 * (1.f - rk) * (1.f - rk) * msq;
                miss = miss || 4.f * kC * kC * da2 >= msq || 4.f * kC * kC * da2 * dsq > kTol2 * msq * msq;
                if (step > 0 && dsq > (float)kNoise2 * msq)
                    miss = miss || 4.f * dsq >= dprev2 || 4.f * dsq * dsq > kTol2 * msq * dprev2;
                // automatic: the second step when the first left too much
                const bool more = autoref && step == 1 && (kC * dsq > (float)kAutoTol * msq || miss);
                const bool redo = step < (autoref ? 1 : steps) || more;
                // ||r - B d||^2 = ||r||^2 - d.g (g = B^T r = G d up to rounding), by
                // one warp: the sum's order is that of every block shape
                double r2 = -dg;
                if (!redo) {
                    for (int i = lane; i < nI; i += 32) r2 = fma(D.r[i], D.r[i], r2);
                    r2 = wsum(r2);
                }
                __syncwarp();
                if (lane == 0) {
                    H.da2 = da2;
                    H.dprev2 = dsq;
                    H.redo = redo;
                    H.r2 = r2;
                    if (!redo) H.fallback = H.fallback || miss;
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

template <class SH>
cudaError_t launch_dense(sam_handle h, const LsqArgs &a, int bin, int32_t *rest, int32_t *rest_off) {
    constexpr int per_sm = SH::BLOCKS;
    // the shared memory of an SM split over per_sm blocks (1 KB of each is the system's)
    const size_t smem = (size_t)((per_sm == 1 ? 232448 : 233472 / per_sm - 1024) & ~127);
    auto kern = lsq_dense_kernel<SH>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<handle_sms(h) * per_sm, SH::NT, smem, handle_stream(h)>>>(a, bin, (unsigned)(smem - sizeof(DenseHdr<SH::MAXJ>) - 8 * SH::UW), rest, rest_off);
    count_launch(h);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_lsq_dense(sam_handle h, const LsqArgs &args, int bin) {
    // Small columns by small blocks, each next launch those that are left.  The
    // class is where most columns are when map 0 has more than 27 unknowns per
    // column on average (the register tiles' limit), or more than 256 entries in
    // the mean B (as many rows at most, where the tiles end at 64; stencils that
    // fit the tiles have up to 225).  Then the shapes of three and two blocks per SM
    // come between: 20,000 columns of 5 unknowns and 950 rows 11.4 ms with them,
    // 15.4 without; of 14 unknowns and 840 rows (80 KB each) 4.3, 7.3 with three
    // blocks per SM alone.  Otherwise the class's columns are few or none, and two
    // launches less are worth more (three empty ones cost small builds 10 to 15 us
    // of 390 to 1,200; two per SM with a handful of columns, where the mean is past
    // its 52 unknowns, 100 us of 15.3 ms).  Which shape solves a column does not change its bits.
    const int64_t n = args.n;
    const bool middle = args.map_nnz_pat > 27 * n ||
                        (double)args.map_nnz_pat * (double)args.map_nnz_src > 256.0 * (double)n * (double)n;
    cudaError_t e;
    if (args.item_hi > 0 && (e = cudaMemsetAsync(args.dense_off, 0, sizeof(int32_t) * 6, handle_stream(h))) != cudaSuccess)
        return e;  // (a chunk of a batch: the counters are used again)
    profile_begin(h, bin);
    if ((e = launch_dense<DenseSmall>(h, args, bin, args.dense_list, args.dense_off)) != cudaSuccess) return e;
    LsqArgs a = args;
    a.item_lo = a.item_hi = 0;
    a.work = args.dense_list;
    a.bin_off = args.dense_off;
    if (middle) {
        // (the two lists in turn: what one launch leaves, the next reads)
        if ((e = launch_dense<DenseMedium>(h, a, 0, args.dense_list + args.dense_cap, args.dense_off + 2)) != cudaSuccess)
            return e;
        a.work = args.dense_list + args.dense_cap;
        a.bin_off = args.dense_off + 2;
        if (args.map_nnz_pat <= DenseHalf::MAXJ * n) {
            if ((e = launch_dense<DenseHalf>(h, a, 0, args.dense_list, args.dense_off + 4)) != cudaSuccess) return e;
            a.work = args.dense_list;
            a.bin_off = args.dense_off + 4;
        }
    }
    if ((e = launch_dense<DenseLarge>(h, a, 0, nullptr, nullptr)) != cudaSuccess) return e;
    profile_end(h, bin);
    return cudaSuccess;
}

}  // namespace sam
