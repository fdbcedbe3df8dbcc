// 64 x 64 tile of the FP64 contraction on the CUDA cores, shared by its own kernel and
// by the tensor-core form's fallback.
#pragma once

#include "ppl_internal.h"

namespace {

constexpr int GBM = 64, GBN = 64, GBK = 16;

__device__ __forceinline__ long long ixd(const Idx2& x, int i) {
    return (long long)(i / x.div) * x.hi + (long long)(i % x.div) * x.lo;
}

// barrier `bar` over the 256 threads of the tile (a caller's block may have more)
__device__ __forceinline__ void block_sync256(int bar) { asm volatile("bar.sync %0, 256;" ::"r"(bar) : "memory"); }

// Rows m0 .., columns n0 .. of batch entry b over kbeg .. kend - 1: 256 threads (tid), 4 x 4
// outputs per thread at (ty + 16 i, tx + 16 j), sm: GBK (GBM + GBN) doubles of shared
// memory, bar: a barrier of their own.  Operands are read through Idx2 maps, so every layout of the method is
// served without copies; the FP64 pipe (not the loads) bounds it on GB300.
__device__ __forceinline__ void gemm64_tile(const G64& g, int b, int m0, int n0, int kbeg, int kend, double* sm, int tid,
                                            int bar) {
    double(*As)[GBM] = (double(*)[GBM])sm;
    double(*Bs)[GBN] = (double(*)[GBN])(sm + GBK * GBM);
    const int tx = tid % 16, ty = tid / 16;
    const double* A = g.A + (long long)b * g.ab;
    const double* B = g.B + (long long)b * g.bb;
    const bool a_kfast = (g.ak.lo == 1 && g.ak.div >= (1 << 30));
    const bool b_kfast = (g.bk.lo == 1 && g.bk.div >= (1 << 30));

    // per-thread load coordinates: 4 elements of each 64x16 tile
    int a_ml[4], a_kl[4], b_nl[4], b_kl[4];
    long long a_row[4], b_row[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int e = tid + 256 * q;
        a_ml[q] = a_kfast ? e / GBK : e % GBM;
        a_kl[q] = a_kfast ? e % GBK : e / GBM;
        b_nl[q] = b_kfast ? e / GBK : e % GBN;
        b_kl[q] = b_kfast ? e % GBK : e / GBN;
        const int m = m0 + a_ml[q], n = n0 + b_nl[q];
        a_row[q] = (m < g.M) ? ixd(g.am, m) : -1;
        b_row[q] = (n < g.N) ? ixd(g.bn, n) : -1;
    }

    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;

    for (int k0 = kbeg; k0 < kend; k0 += GBK) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int ka = k0 + a_kl[q], kb = k0 + b_kl[q];
            As[a_kl[q]][a_ml[q]] = (a_row[q] >= 0 && ka < kend) ? A[a_row[q] + ixd(g.ak, ka)] : 0.0;
            Bs[b_kl[q]][b_nl[q]] = (b_row[q] >= 0 && kb < kend) ? B[b_row[q] + ixd(g.bk, kb)] : 0.0;
        }
        block_sync256(bar);
#pragma unroll
        for (int kk = 0; kk < GBK; ++kk) {
            double av[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
        }
        block_sync256(bar);
    }

    double* C = g.C + (long long)b * g.cb;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty + 16 * i;
        if (m >= g.M) continue;
        const long long cr = ixd(g.cm, m);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx + 16 * j;
            if (n >= g.N) continue;
            double* p = C + cr + ixd(g.cn, n);
            if (g.atomic) {
                atomicAdd(p, g.alpha * acc[i][j]);
            } else {
                const double old = (g.beta != 0.0) ? g.beta * *p : 0.0;
                *p = fma(g.alpha, acc[i][j], old);
            }
            if (g.lower && n0 < m0) C[ixd(g.cm, n) + ixd(g.cn, m)] = *p;     // the mirrored tile
        }
    }
}

}  // namespace
