// residual_row.cuh -- one row of R = A_k M - A_0 (Eq. (res)), summed in a
// fixed order by one warp.  Shared by sam_residual (misc.cu) and the
// allocation-free sam_residual_static (noalloc.cu), so that both compute
// the same bits.
#pragma once

#include <climits>

#include "common.cuh"

namespace sam {

constexpr int kResRowBuf = 1024;  // candidate entries of one row of R a warp can hold

// A row is summed through its columns' ranks where it has more candidates than a
// warp (those take 15 rounds of the sort, less than a bitmap of any span) and at
// most kResFastCnt, over at most kResFastWords words of 32 columns.  Per call, sort /
// ranks: 30 candidates, 200,000 rows, over 63 words 0.593 / 0.603 ms, over 938
// 0.591 / 0.688; 56 candidates over 129 words (32,768 rows) 0.222 / 0.186, over 969
// (681,472 rows) 3.21 / 2.94; 234 candidates over 33 (65,536 rows) 1.11 / 0.36.
constexpr int kResSortCnt = 32, kResFastCnt = 768;
constexpr int kResFastWords = 1024;

// ||R(i, :)||^2 for R = A_k M - A_0, computed by the calling warp.  The row's
// entries are the products A_k(i, c) M(c, :) and -A_0(i, :).  In long rows whose
// columns span at most 32 kResFastWords (every stencil and mesh in a banded
// numbering), a bitmap of the columns in K gives each its rank, and the
// products are added to V[rank] in the order of the row of A_k (the columns of
// one row of M are distinct, so its entries are added side by side).
// Otherwise they are collected as (column, value) pairs in K / V (kResRowBuf
// entries of the warp's own shared memory), sorted by column with a fixed
// bitonic network and summed per column.  The sort took 36 rounds over 256
// pairs for a row of 234 candidates: 1.04 ms for 65,536 rows of a level-2 Q1
// map (a build, residual, apply and adjoint of it 4.87 ms; with the ranks 4.14).
// Every lane returns the same value.  Returns a negative value, having written
// nothing, when the row has more than kResRowBuf candidate entries.
__device__ __forceinline__ double residual_row_sq(int64_t i, int lane, const int32_t *krp, const int32_t *kci,
                                                  const double *kv, const int32_t *mrp, const int32_t *mci,
                                                  const double *mv, const int32_t *zrp, const int32_t *zci,
                                                  const double *zv, int *K, double *V) {
    // count the candidates
    int cnt = zrp[i + 1] - zrp[i];
    for (int base = krp[i]; base < krp[i + 1]; base += 32) {
        const int e = base + lane;
        int len = (e < krp[i + 1]) ? mrp[kci[e] + 1] - mrp[kci[e]] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) len += __shfl_xor_sync(0xffffffffu, len, o);
        cnt += len;
    }
    if (cnt > kResRowBuf) return -1.0;
    const int zb = zrp[i], ze = zrp[i + 1];
    if (cnt > kResSortCnt && cnt <= kResFastCnt) {
        // the span of the columns (rows are sorted: their ends)
        int lo = INT_MAX, hi = -1;
        for (int e = krp[i] + lane; e < krp[i + 1]; e += 32) {
            const int mb = mrp[kci[e]], me = mrp[kci[e] + 1];
            if (me > mb) {
                lo = min(lo, mci[mb]);
                hi = max(hi, mci[me - 1]);
            }
        }
        if (ze > zb) {
            lo = min(lo, zci[zb]);
            hi = max(hi, zci[ze - 1]);
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (hi < 0) return 0.0;
        const int64_t span = (int64_t)hi - lo + 1;
        if (span <= 32 * kResFastWords) {
            const int words = (int)((span + 31) >> 5);
            unsigned *bm = reinterpret_cast<unsigned *>(K);
            unsigned short *pre = reinterpret_cast<unsigned short *>(V + kResFastCnt);  // columns before each word
            for (int w = lane; w < words; w += 32) bm[w] = 0u;
            __syncwarp();
            // A row out of order (an unvalidated input) is left to the sort:
            // it may leave the window or name a column twice.
            bool fit = true;
            auto mark = [&](const int32_t *ci, int t, int b) {
                const int x = ci[t] - lo;
                if (x < 0 || x >= span || (t > b && ci[t - 1] >= ci[t]))
                    fit = false;
                else
                    atomicOr(&bm[x >> 5], 1u << (x & 31));
            };
            for (int t = zb + lane; t < ze; t += 32) mark(zci, t, zb);
            for (int e0 = krp[i]; e0 < krp[i + 1]; e0 += 32) {
                const int e = e0 + lane, ne = min(32, krp[i + 1] - e0);
                const int c = lane < ne ? kci[e] : 0;
                const int mb_ = lane < ne ? mrp[c] : 0, me_ = lane < ne ? mrp[c + 1] : 0;
                for (int q = 0; q < ne; ++q) {
                    const int mb = __shfl_sync(0xffffffffu, mb_, q), me = __shfl_sync(0xffffffffu, me_, q);
                    for (int t = mb + lane; t < me; t += 32) mark(mci, t, mb);
                }
            }
            __syncwarp();
            if (__all_sync(0xffffffffu, fit)) {
                const int wpl = (words + 31) >> 5, w0 = min(words, lane * wpl), w1 = min(words, w0 + wpl);
                int own = 0;
                for (int w = w0; w < w1; ++w) own += __popc(bm[w]);
                int incl = own;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int distinct = __shfl_sync(0xffffffffu, incl, 31);
                int run = incl - own;
                for (int w = w0; w < w1; ++w) {
                    pre[w] = (unsigned short)run;
                    run += __popc(bm[w]);
                }
                for (int t = lane; t < distinct; t += 32) V[t] = 0.0;
                __syncwarp();
                auto at = [&](int col) {
                    const int x = col - lo;
                    return (int)pre[x >> 5] + __popc(bm[x >> 5] & ((1u << (x & 31)) - 1u));
                };
                for (int t = zb + lane; t < ze; t += 32) V[at(zci[t])] = -zv[t];
                __syncwarp();
                for (int e0 = krp[i]; e0 < krp[i + 1]; e0 += 32) {
                    const int e = e0 + lane, ne = min(32, krp[i + 1] - e0);
                    const int c = lane < ne ? kci[e] : 0;
                    const int mb_ = lane < ne ? mrp[c] : 0, me_ = lane < ne ? mrp[c + 1] : 0;
                    const double a_ = lane < ne ? kv[e] : 0.0;
                    for (int q = 0; q < ne; ++q) {
                        const int me = __shfl_sync(0xffffffffu, me_, q);
                        const double a = __shfl_sync(0xffffffffu, a_, q);
                        for (int t = __shfl_sync(0xffffffffu, mb_, q) + lane; t < me; t += 32) {
                            const int r = at(mci[t]);
                            V[r] = fma(a, mv[t], V[r]);
                        }
                        __syncwarp();
                    }
                }
                double r2 = 0.0;
                for (int t = lane; t < distinct; t += 32) r2 = fma(V[t], V[t], r2);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
                __syncwarp();
                return r2;
            }
            __syncwarp();
        }
    }
    // target entries first, then the products, in a fixed order
    for (int t = zb + lane; t < ze; t += 32) {
        K[t - zb] = zci[t];
        V[t - zb] = -zv[t];
    }
    int off = ze - zb;
    for (int e = krp[i]; e < krp[i + 1]; ++e) {
        const int c = kci[e];
        const double a = kv[e];
        const int mb = mrp[c], me = mrp[c + 1];
        for (int t = mb + lane; t < me; t += 32) {
            K[off + t - mb] = mci[t];
            V[off + t - mb] = a * mv[t];
        }
        off += me - mb;
    }
    __syncwarp();
    int p2 = 32;
    while (p2 < cnt) p2 <<= 1;
    for (int t = cnt + lane; t < p2; t += 32) {
        K[t] = INT_MAX;
        V[t] = 0.0;
    }
    __syncwarp();
    for (int k = 2; k <= p2; k <<= 1)
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            for (int t = lane; t < p2; t += 32) {
                const int u = t ^ jj;
                if (u > t) {
                    const bool up = (t & k) == 0;
                    const int a = K[t], b = K[u];
                    if ((a > b) == up) {
                        K[t] = b;
                        K[u] = a;
                        const double va = V[t];
                        V[t] = V[u];
                        V[u] = va;
                    }
                }
            }
            __syncwarp();
        }
    // segmented sums: the lane holding the first entry of a column sums it
    double r2 = 0.0;
    for (int t = lane; t < cnt; t += 32) {
        if (t == 0 || K[t - 1] != K[t]) {
            double s = 0.0;
            for (int q = t; q < cnt && K[q] == K[t]; ++q) s += V[q];
            r2 = fma(s, s, r2);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    __syncwarp();
    return r2;
}

}  // namespace sam
