// One ALS mode update in a single cooperative FP64 kernel (Optimizing the
// CP-PPL tensor-network section: W as the Hadamard product of the other
// three Gram matrices, a Cholesky solve of the normal equations, column
// normalisation; then the new factor's Gram matrix for the next updates).
//
//   P0  V = G1 .* G2 .* G3 (lower triangle), Z = M, tol = max(2^-52 R max V_kk, 1e-300)
//   P1  right-looking blocked Cholesky of V (32-wide blocks, pivots clamped at tol;
//       panels by warp-per-row triangular solves with the column-scaled diagonal block)
//       with the rows of Z appended below V, so the same panel and trailing updates
//       carry out the forward substitution Z <- M L^-T; the next diagonal block is
//       updated by five blocks and factored by block 0 while the others update the rest
//   P2  back substitution U~ L = Z: the rows are independent, so every block solves
//       its own rows over all column blocks with no grid barrier (one warp per
//       column block in turn, all eight warps for the updates left of it)
//   P3  lam_r = ||U~[:, r]||, U = U~ / lam (a zero column keeps lam = 0)
//   P4  G = U^T U
//
// GB300 executes about two FP64 FMAs per clock per SM, so every phase is
// spread over all SMs in 32 x 32 tiles and 8-row panels; phases are separated
// by grid barriers (a cooperative launch guarantees co-residency).  Every
// barrier wait is bounded: on expiry the kernel raises an abort flag that
// all blocks observe, records the error and returns.
#include "ppl_internal.h"

#include <algorithm>

#include <cmath>

namespace {

constexpr int NB = 32;
constexpr int NT = 256;
constexpr unsigned long long BAR_NS = 1000ull * 1000ull * 1000ull;   // 1 s per barrier wait

// The block's shared memory (at file scope, so that the factorisation below can be
// a function of its own and still address it as shared memory).
__shared__ double Ls[NB][NB + 1];   // the diagonal block being factored; staging in the back substitution
__shared__ double Li[NB][NB + 1];   // its column-scaled factor; staging in the back substitution
__shared__ double Ta[NB][NB + 1];   // tiles
__shared__ double Tb[NB][NB + 1];
__shared__ double rd[NB];           // 1 / L_jj
__shared__ unsigned short tri[NB * (NB + 1) / 2];   // (row << 8) | col of the lower triangle, row-major

struct SolveP {
    const double* G1;
    const double* G2;
    const double* G3;
    double* V;
    double* Linv;
    const double* M;
    double* Z;
    double* U;
    double* lam;
    double* G;
    unsigned int* sync;              // barrier words (see gsync), zero between launches
    unsigned long long* nclamp;
    unsigned int* err;
    unsigned int* withhold;          // != 0: block 1 skips its first barrier arrival (once)
    unsigned long long wait_ns;      // bound of every barrier wait
    int R, dim;
};

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned int ld_vol(const unsigned int* p) { return *(volatile const unsigned int*)p; }

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned int atom_add_release(unsigned int* p, unsigned int v) {
    unsigned int old;
    asm volatile("atom.add.release.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// p.sync: [0] arrivals of this launch, counted up over all barriers, with the top
// bit as the abort flag (a waiter learns of an abort from the word it polls
// anyway); [1] blocks that have left; [3] pieces of the next diagonal block.  The
// words are zero between launches: the last block to leave clears them, on the
// abort path too, so no launch needs a memset before it (two memset nodes ahead
// of every solve cost 8 to 11 us of graph time, 40 us per sweep).
constexpr unsigned int SYNC_ABORT = 0x80000000u;

__device__ __forceinline__ void raise_abort(const SolveP& p, unsigned int code) {
    atomicOr(&p.sync[0], SYNC_ABORT);
    atomicOr(p.err, code);
}

// wait (bounded) until *w >= target; false when the wait ran out or a block aborted.
// The clock is read on every 32nd poll only: a poll is one L2 round trip and the
// barriers are on the critical path.
__device__ __forceinline__ bool poll_until(const SolveP& p, const unsigned int* w, unsigned int target, unsigned int code) {
    unsigned long long t0 = 0;
    for (unsigned int n = 1;; ++n) {
        const unsigned int v = ld_acquire(w);
        if (w == &p.sync[0] && (v & SYNC_ABORT)) return false;
        if ((v & ~SYNC_ABORT) >= target) return true;
        if ((n & 31u) == 0u) {
            const unsigned long long t = gtimer();
            if (t0 == 0) t0 = t;
            if (t - t0 > p.wait_ns) {
                raise_abort(p, code);
                return false;
            }
            if (ld_vol(&p.sync[0]) & SYNC_ABORT) return false;
        }
    }
}

// grid-wide barrier; false when the wait expired or another block aborted.
// The block's writes are ordered before its arrival by __syncthreads and the
// release of the arrival; the waiters' acquire loads order what follows.  The
// waiters poll the arrival counter itself (target counts G more per barrier), so
// the last arrival releases them with no second word to write: 1.5 us on 152
// blocks, against 2.5 us with a separate generation word and a clock read per poll.
__device__ bool gsync(const SolveP& p, unsigned int& target, int* s_flag, int bid, int G) {
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        target += (unsigned int)G;
        // the test of the bounded waits: block 1 withholds its first arrival, so
        // the other blocks' wait runs out; it waits (bounded) for their abort
        const bool withhold =
            bid == 1 && p.withhold && ld_vol(p.withhold) != 0u && atomicExch(p.withhold, 0u) != 0u;
        if (withhold) {
            const unsigned long long t0 = gtimer();
            while (!(ld_vol(&p.sync[0]) & SYNC_ABORT) && gtimer() - t0 < 4 * p.wait_ns) {
            }
            ok = 0;
        } else {
            const unsigned int old = atom_add_release(&p.sync[0], 1u);
            ok = (old & SYNC_ABORT) ? 0 : (poll_until(p, &p.sync[0], target, 16u) ? 1 : 0);
        }
        *s_flag = ok;
    }
    __syncthreads();
    return *s_flag != 0;
}

// every block passes here once per launch, whatever happened before: the last one
// leaves the barrier words at zero for the next launch
__device__ void leave_sync(const SolveP& p, int G) {
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int old;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(&p.sync[1]) : "memory");
        if (old == (unsigned int)G - 1u) {
            p.sync[0] = 0u;
            p.sync[3] = 0u;
            p.sync[1] = 0u;
        }
    }
}

__device__ __forceinline__ void tri_index(int t, int& I, int& J) {
    // t -> (I, J), I >= J, row-major over the lower triangle (an FP32 estimate,
    // corrected exactly below: the FP64 pipe is the solve's bottleneck)
    int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= t) ++i;
    while (i * (i + 1) / 2 > t) --i;
    I = i;
    J = t - i * (i + 1) / 2;
}

// 1/d for a positive normal d: the PTX approximate reciprocal refined by two
// Newton-Raphson steps x <- x + x (1 - d x), each squaring the relative error
// (within an ulp or two of the correctly rounded quotient).  Four FP64 FMAs
// instead of the longer IEEE division sequence on the factorisation's
// critical path.  (One third-order step is three, 64 clocks less per pivot, but its
// last bits differ; the tensor-core forms split the factors into operands, and a
// last bit at a rounding boundary of an operand changes every later sweep by the
// split precision's noise.)
__device__ __forceinline__ double recip_nr(double d) {
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(d));
    double e = fma(-d, x, 1.0);
    x = fma(x, e, x);
    e = fma(-d, x, 1.0);
    return fma(x, e, x);
}

// Factor the kb x kb diagonal block held in Ls (lower) and leave in Li the
// column-scaled factor the panel and back substitution solve with: Li[i][j] =
// L[i][j] / L[j][j] below the diagonal, 1 / L[i][i] on it, 0 elsewhere.  Pivots
// not above tol are replaced by tol and counted.  Li is also written to Linv, where
// the other blocks read it.  All NT threads.
//
// Right-looking on unscaled columns: with d_j the pivot and s_i = a_ij (1 / d_j),
// a_ic -= s_i a_cj; the scalings by 1 / sqrt(d_j) follow at the end, all at once.  An FP64 instruction occupies its SM
// sub-partition's pipe for 64 clocks however many lanes are active, so the work
// is laid out by sub-partitions.  Warp 0 alone, on its own sub-partition, owns the
// chain pivot -> reciprocal -> column -> next pivot: at step j it scales column j
// (which it hands to the others), updates column j + 1 and inverts the next pivot,
// six dependent FP64 instructions, while the six warps of the other three
// sub-partitions apply column j to columns j + 2 ..; one block barrier per step.
// The pivot test is an integer comparison (an FP64 one is one more instruction).
// Measured on one 32 x 32 block: 16.3 us with the whole triangle updated by all
// warps, two instructions per element, the reciprocal after it in the same step
// and separate passes for square roots and scaling; 10.5 us so.
__device__ __noinline__ void factor_block(double* Linv, int kb, double tol, unsigned long long* nclamp) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    // the helpers: the six warps that do not share sub-partition 0 with warp 0
    const int hw = warp < 4 ? warp - 1 : warp - 2;            // 1, 2, 3, 5, 6, 7 -> 0 .. 5
    const bool helper = (warp & 3) != 0;
    for (int e = threadIdx.x; e < NB * NB; e += NT) Li[e / NB][e % NB] = 0.0;
    __syncthreads();
    double a = 0.0;        // warp 0: a_ij of column j, i = lane
    double dl = 1.0;       // the pivot of column `lane`
    double r = 0.0;        // 1 / d_j
    const long long tol_bits = __double_as_longlong(tol);
    auto pivot = [&](int j) {             // d_j from column j, clamped, and its reciprocal (every lane)
        double d = __shfl_sync(0xffffffffu, a, j);
        // d > tol for tol > 0: positive doubles order as their bits; negative and NaN fail
        const long long bits = __double_as_longlong(d);
        if (!(bits > tol_bits && bits <= 0x7ff0000000000000ll)) {
            d = tol;
            if (lane == 0) atomicAdd(nclamp, 1ull);
        }
        if (lane == j) dl = d;
        r = recip_nr(d);
    };
    if (warp == 0) {
        a = lane < kb ? Ls[lane][0] : 0.0;
        pivot(0);
    }
    for (int j = 0; j < kb; ++j) {
        if (warp == 0) {
            const double s = a * r;
            double x = (j + 1 < kb && lane > j && lane < kb) ? Ls[lane][j + 1] : 0.0;
            const double aj1 = __shfl_sync(0xffffffffu, a, (j + 1) & 31);
            if (lane > j && lane < kb) Li[lane][j] = s;
            // the column is published: the helpers may start
            asm volatile("bar.arrive 1, 224;" ::: "memory");
            if (j + 1 < kb) {
                x = fma(-s, aj1, x);
                if (lane > j && lane < kb) Ls[lane][j + 1] = x;
                a = x;
                pivot(j + 1);
            }
        } else if (helper) {
            asm volatile("bar.sync 1, 224;" ::: "memory");
            const int m = kb - j - 2;          // columns j + 2 .. kb - 1
            const int nel = m > 0 ? m * (m + 1) / 2 : 0;
            for (int e = hw * 32 + lane; e < nel; e += 6 * 32) {
                const unsigned short ic = tri[e];
                const int i = j + 2 + (ic >> 8), c = j + 2 + (ic & 0xff);
                Ls[i][c] = fma(-Li[i][j], Ls[c][j], Ls[i][c]);
            }
        }
        __syncthreads();
    }
    // L_jj = sqrt(d_j), L_ij = a_ij / L_jj, Li_ij = L_ij / L_jj
    if (warp == 0) rd[lane] = lane < kb ? recip_nr(sqrt(dl)) : 0.0;
    __syncthreads();
    for (int e = threadIdx.x; e < kb * (kb + 1) / 2; e += NT) {
        const int i = tri[e] >> 8, j = tri[e] & 0xff;
        Li[i][j] = i == j ? rd[i] : Ls[i][j] * rd[j] * rd[j];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NB * NB; e += NT) Linv[e] = Li[e / NB][e % NB];
    __syncthreads();
}

constexpr int RB = 4;   // rows of U~ per back-substitution pass
// pieces of the next diagonal block's update, of PIECE elements of its lower triangle
constexpr int NPIECE = 5, PIECE = (NB * (NB + 1) / 2 + NPIECE - 1) / NPIECE;

// asynchronous global -> shared copies (cp.async), waited for by the issuing thread
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// one warp copies rows 0 .. rows-1 of an NB-wide block (row stride ld) into dst
__device__ __forceinline__ void stage_block(const double* src, long long ld, int rows, double (*dst)[NB + 1], int lane) {
#pragma unroll 8
    for (int q = 0; q < rows; ++q) cp_async8(&dst[q][lane], src + q * ld + lane);
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Zl[r][c + bs b] -= sum_q x[r][q] L[j0 + q][lane + c + bs b] for the NR rows and
// CB column blocks b of one warp (Zl and Ll point at the lane's column: Zl at
// Z[r0][lane], Ll at L[j0][lane]).
template <int NR, int CB>
__device__ __forceinline__ void back_update(double* Zl, int R, const double* Ll, const double (*x)[NB], int c, int kb,
                                            int bs, double (*acc)[NR]) {
#pragma unroll
    for (int b = 0; b < CB; ++b)
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[b][r] = __ldcg(Zl + (long long)r * R + c + b * bs);
#pragma unroll 4
    for (int q = 0; q < kb; ++q) {
        double l[CB];
#pragma unroll
        for (int b = 0; b < CB; ++b) l[b] = __ldcg(Ll + (long long)q * R + c + b * bs);
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const double xv = x[r][q];
#pragma unroll
            for (int b = 0; b < CB; ++b) acc[b][r] = fma(-xv, l[b], acc[b][r]);
        }
    }
#pragma unroll
    for (int b = 0; b < CB; ++b)
#pragma unroll
        for (int r = 0; r < NR; ++r) Zl[(long long)r * R + c + b * bs] = acc[b][r];
}

// The kb unknowns of one column block for NR rows (one warp, lane = column):
// w holds the block of Z with every block to its right already subtracted; with
// the column-scaled diagonal block Ld (L_qt / L_tt below the diagonal, 1 / L_tt
// on it), x_q is final once the columns right of q are subtracted, then
// w_t -= x_q L_qt / L_tt for t < q.
template <int NR>
__device__ __forceinline__ void back_diag(const double (*Ld)[NB + 1], int kb, int lane, double* w) {
    const double dinv = (lane < kb) ? Ld[lane][lane] : 0.0;
#pragma unroll
    for (int r = 0; r < NR; ++r) w[r] = (lane < kb) ? w[r] * dinv : 0.0;
    for (int q = kb - 1; q > 0; --q) {
        const double lq = (lane < q) ? Ld[q][lane] : 0.0;
#pragma unroll
        for (int r = 0; r < NR; ++r) w[r] = fma(-__shfl_sync(0xffffffffu, w[r], q), lq, w[r]);
    }
}

// Rows r0 .. r0+NR-1 of the back substitution U~ L = Z, all NT threads of the
// block, column blocks from the last one down.  At step J the unknowns x_J are
// published in shared memory; warp (J-1) mod 8 subtracts x_J L[rows of J][block
// J-1] from block J-1, keeps the result in registers and solves it at once
// (x_{J-1}), while the seven other warps subtract x_J from blocks 0 .. J-2; one
// block barrier per step.  The diagonal block of J-1 and the block L[rows of J]
// [block J-1] were copied to shared memory (cp.async) by the same warp one step
// earlier; the published values and the staged blocks alternate between two
// buffers (one row per SM, R = 250: 26 us against 40 us with L[J][J-1] read from L2
// inside the owner's chain of 32 FMAs).
template <int NR>
__device__ void back_rows(const SolveP& p, int r0, double (*xs)[RB][NB], double (*lb0)[NB + 1], double (*lb1)[NB + 1],
                          double (*lo0)[NB + 1], double (*lo1)[NB + 1]) {
    constexpr int NW = NT / 32, NO = NW - 1;
    // CB blocks per pass, so that a pass keeps 4 sums and CB loads per step of q
    // in flight also when NR is small
    constexpr int CB = (NR == 1) ? 4 : (NR == 2 ? 2 : 1);
    const int R = p.R;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nt = (R + NB - 1) / NB;
    double* Zr = p.Z + (long long)r0 * R;
    auto publish = [&](int J, const double* w) {
        const int j0 = J * NB, kb = min(NB, R - j0);
        if (lane < kb) {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                xs[J & 1][r][lane] = w[r];
                p.U[(long long)(r0 + r) * R + j0 + lane] = w[r];
            }
        }
    };
    // what the owner of block J needs one step later: its diagonal block and L[rows of J+1][block J]
    auto stage = [&](int J) {
        stage_block(p.Linv + (long long)J * NB * NB, NB, NB, (J & 1) ? lb1 : lb0, lane);
        const int j1 = (J + 1) * NB;
        stage_block(p.V + (long long)j1 * R + J * NB, R, min(NB, R - j1), (J & 1) ? lo1 : lo0, lane);
    };
    {   // the last block has nothing to its right
        const int J = nt - 1, j0 = J * NB, kb = min(NB, R - j0);
        if (warp == J % NW) {
            stage_block(p.Linv + (long long)J * NB * NB, NB, NB, (J & 1) ? lb1 : lb0, lane);
            cp_async_wait_all();
            __syncwarp();
            double w[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) w[r] = (lane < kb) ? __ldcg(Zr + (long long)r * R + j0 + lane) : 0.0;
            back_diag<NR>((J & 1) ? lb1 : lb0, kb, lane, w);
            publish(J, w);
        }
        if (J >= 1 && warp == (J - 1) % NW) stage(J - 1);
        __syncthreads();
    }
    for (int J = nt - 1; J >= 1; --J) {
        const int j0 = J * NB, kb = min(NB, R - j0);
        const double (*x)[NB] = xs[J & 1];
        const double* Ll = p.V + (long long)j0 * R + lane;     // L[j0 + q][lane + c] at q * R + c
        const int ow = (J - 1) % NW;
        if (warp == ow) {
            double w[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) w[r] = __ldcg(Zr + (long long)r * R + (J - 1) * NB + lane);
            cp_async_wait_all();
            __syncwarp();
            const double (*lo)[NB + 1] = ((J - 1) & 1) ? lo1 : lo0;
#pragma unroll 8
            for (int q = 0; q < kb; ++q) {
                const double l = lo[q][lane];
#pragma unroll
                for (int r = 0; r < NR; ++r) w[r] = fma(-x[r][q], l, w[r]);
            }
            back_diag<NR>(((J - 1) & 1) ? lb1 : lb0, NB, lane, w);
            publish(J - 1, w);
        } else {
            if (J >= 2 && warp == (J - 2) % NW) stage(J - 2);
            const int w7 = (warp - ow - 1 + NW) % NW;
            int Jc = w7;
            double acc[CB][NR];
            for (; Jc + NO * (CB - 1) < J - 1; Jc += NO * CB) back_update<NR, CB>(Zr + lane, R, Ll, x, Jc * NB, kb, NO * NB, acc);
            for (; Jc < J - 1; Jc += NO) back_update<NR, 1>(Zr + lane, R, Ll, x, Jc * NB, kb, NO * NB, acc);
        }
        __syncthreads();
    }
}

// One 32 x 32 tile of a block step's trailing update: C -= Pa Pb^T over the kb
// columns of the panel, C in the lower triangle of V (tiles below the next
// diagonal) or in Z (the appended rows).
struct TrailTile {
    const double* Pa;
    const double* Pb;
    double* C;
    int arows, brows;
    bool diag;      // a diagonal tile of V: only j <= i is updated
};

__device__ __forceinline__ TrailTile trail_tile(const SolveP& p, int tile, int k0, int kb, int ntri, int Tk, int dim) {
    const int R = p.R;
    TrailTile t;
    int i0, j0;
    if (tile < ntri) {
        int I, J;
        tri_index(tile, I, J);
        i0 = k0 + kb + I * NB;
        j0 = k0 + kb + J * NB;
        t.Pa = p.V + (long long)i0 * R + k0;
        t.arows = R - i0;
        t.C = p.V + (long long)i0 * R + j0;
        t.diag = (I == J);
    } else {
        const int tz = tile - ntri;
        const int Mb = tz / Tk, J = tz % Tk;
        i0 = Mb * NB;
        j0 = k0 + kb + J * NB;
        t.Pa = p.Z + (long long)i0 * R + k0;
        t.arows = dim - i0;
        t.C = p.Z + (long long)i0 * R + j0;
        t.diag = false;
    }
    t.brows = R - j0;
    t.Pb = p.V + (long long)j0 * R + k0;
    return t;
}

__device__ __forceinline__ bool trail_owns(const TrailTile& t, int i, int j) {
    return i < t.arows && j < t.brows && (!t.diag || j <= i);
}

// this thread's four elements of each operand tile and its four C values
__device__ __forceinline__ void trail_fetch(const TrailTile& t, int R, int kb, int tid, int tx, int ty, double* pa,
                                            double* pb, double* pc) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int e = tid + u * NT;
        const int i = e / NB, s2 = e % NB;
        pa[u] = (i < t.arows && s2 < kb) ? __ldcg(t.Pa + (long long)i * R + s2) : 0.0;
        pb[u] = (i < t.brows && s2 < kb) ? __ldcg(t.Pb + (long long)i * R + s2) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = ty + 16 * (u >> 1), j = tx + 16 * (u & 1);
        pc[u] = trail_owns(t, i, j) ? __ldcg(t.C + (long long)i * R + j) : 0.0;
    }
}

// this thread's two elements of each 32 x 16 operand of the Gram tile at (i0, j0)
// (16 x 16 tiles of the lower triangle), rows x0 .. x0+31 of U
__device__ __forceinline__ void gram_fetch(const SolveP& p, int i0, int j0, int x0, int tid, double* qa, double* qb) {
    constexpr int T16 = 16;
    const int R = p.R, dim = p.dim;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int e = tid + u * NT;
        const int x = e / T16, c = e % T16;
        const bool okx = (x0 + x < dim);
        qa[u] = (okx && i0 + c < R) ? __ldcg(p.U + (long long)(x0 + x) * R + i0 + c) : 0.0;
        qb[u] = (okx && j0 + c < R) ? __ldcg(p.U + (long long)(x0 + x) * R + j0 + c) : 0.0;
    }
}

// One mode update of one instance, run by blocks bid = 0 .. G-1 (of one launch,
// or of one instance's share of a batched launch); the barriers count G blocks.
__device__ __forceinline__ void solve_body(const SolveP& p, const int bid, const int G) {
    __shared__ double red[NT / 32];
    __shared__ int s_flag;

    const int R = p.R, dim = p.dim;
    const int tid = threadIdx.x;
    const long long gtid = (long long)bid * NT + tid;
    const long long gthreads = (long long)G * NT;
    for (int i = 0, e = 0; i < NB; ++i)
        for (int c = 0; c <= i; ++c, ++e)
            if (e % NT == tid) tri[e] = (unsigned short)((i << 8) | c);
    unsigned int target = 0;   // arrivals of the next barrier; meaningful in thread 0 only
    const int kb0 = min(NB, R);

    // ---- P0 --------------------------------------------------------------------
    // every block forms the pivot tolerance from the diagonal of V itself
    double mx = 0.0;
    for (int i = tid; i < R; i += NT) {
        const long long d = (long long)i * R + i;
        mx = fmax(mx, p.G1[d] * p.G2[d] * p.G3[d]);
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (tid % 32 == 0) red[tid / 32] = mx;
    __syncthreads();
    mx = red[0];
    for (int w = 1; w < NT / 32; ++w) mx = fmax(mx, red[w]);
    const double tol = fmax(ldexp(1.0, -52) * (double)R * mx, 1e-300);
    if (bid == 0) {
        // the first diagonal block straight from the Gram matrices
        for (int e = tid; e < kb0 * kb0; e += NT) {
            const int i = e / kb0, j = e % kb0;
            const long long d = (long long)i * R + j;
            if (j <= i) Ls[i][j] = p.G1[d] * p.G2[d] * p.G3[d];
        }
        __syncthreads();
        factor_block(p.Linv, kb0, tol, p.nclamp);
    }
    // V and Z, row by row (no 64-bit division per element); block 0 is busy with the
    // factor, so it leaves its rows to the others where there are any
    {
        const int nb = G > 1 ? G - 1 : 1, b0 = G > 1 ? bid - 1 : 0;
        if (b0 >= 0) {
            for (int r = kb0 + b0; r < R; r += nb) {
                const long long d = (long long)r * R;
                for (int q = tid; q <= r; q += NT) p.V[d + q] = p.G1[d + q] * p.G2[d + q] * p.G3[d + q];
            }
        }
    }
    for (long long e = gtid; e < (long long)dim * R; e += gthreads) p.Z[e] = p.M[e];
    if (!gsync(p, target, &s_flag, bid, G)) return;

    const int nt = (R + NB - 1) / NB;
    const int D = (dim + NB - 1) / NB;
    const int tx = tid % 16, ty = tid / 16;

    // ---- P1: Cholesky with the forward substitution fused, one block of look-ahead
    for (int k = 0; k < nt; ++k) {
        const int k0 = k * NB, kb = min(NB, R - k0);
        for (int e = tid; e < NB * NB; e += NT) Li[e / NB][e % NB] = __ldcg(p.Linv + (long long)k * NB * NB + e);
        __syncthreads();
        // panel: rows below the block (V) and all rows of Z, 8 rows per task
        const int vrows = R - k0 - kb;
        const int prow = vrows + dim;                // V rows below the block, then the rows of Z
        // one warp per row solves x L^T = a: with val_q final, x_q = val_q / L_qq
        // and val_t -= val_q (L_tq / L_qq), so each column costs one FMA
        const int ntask = (prow + 7) / 8;
        for (int task = bid; task < ntask; task += G) {
            const int rr = task * 8 + tid / NB, t = tid % NB;
            double* row = nullptr;
            if (rr < vrows)
                row = p.V + (long long)(k0 + kb + rr) * R + k0;
            else if (rr < prow)
                row = p.Z + (long long)(rr - vrows) * R + k0;
            if (row) {   // warp-uniform: rr is the same for the 32 lanes
                double val = (t < kb) ? __ldcg(row + t) : 0.0;
                for (int q = 0; q < kb; ++q) {
                    const double yq = __shfl_sync(0xffffffffu, val, q);
                    if (t > q) val = fma(-yq, Li[t][q], val);
                }
                if (t < kb) row[t] = val * Li[t][t];
            }
        }
        if (!gsync(p, target, &s_flag, bid, G)) return;
        // trailing update of V (lower tiles) and of Z.  Tile 0 is the next
        // diagonal block: the blocks 0 .. NPIECE-1 each update a fifth of its lower
        // triangle (one warp per SM sub-partition: 1 us of FP64 issue, against 4.2
        // us on one SM), the others signal block 0, which factors the block while
        // the rest of the grid takes the remaining tiles.  Block 0 takes no other
        // tile; with too few blocks it updates all of tile 0.
        const int Tk = (vrows + NB - 1) / NB;
        const int ntri = Tk * (Tk + 1) / 2;
        const int ntile = ntri + D * Tk;
        const bool pieces = G > NPIECE;
        if (k + 1 < nt && bid < (pieces ? NPIECE : 1)) {
            const int d0 = k0 + kb, nb1 = min(NB, R - d0);
            const double* Pd = p.V + (long long)d0 * R + k0;     // rows of the panel at the next block
            for (int e = tid; e < NB * NB; e += NT) {
                const int i = e / NB, s2 = e % NB;
                Ta[i][s2] = (i < nb1 && s2 < kb) ? __ldcg(Pd + (long long)i * R + s2) : 0.0;
            }
            __syncthreads();
            const int nel = nb1 * (nb1 + 1) / 2;
            const int e0 = pieces ? bid * PIECE : 0, e1 = pieces ? min(nel, e0 + PIECE) : nel;
            for (int e = e0 + tid; e < e1; e += NT) {
                const int i = tri[e] >> 8, j = tri[e] & 0xff;
                double* c = p.V + (long long)(d0 + i) * R + d0 + j;
                const double c0 = __ldcg(c);
                double acc = 0.0;
#pragma unroll 8
                for (int s2 = 0; s2 < NB; ++s2) acc = fma(Ta[i][s2], Ta[j][s2], acc);
                if (bid == 0)
                    Ls[i][j] = c0 - acc;
                else
                    *c = c0 - acc;
            }
            __syncthreads();
            if (bid != 0) {
                if (tid == 0) atom_add_release(&p.sync[3], 1u);
            } else {
                if (pieces) {
                    if (tid == 0)
                        s_flag = poll_until(p, &p.sync[3], (unsigned int)(NPIECE - 1) * (unsigned int)(k + 1), 64u) ? 1 : 0;
                    __syncthreads();
                    for (int e = PIECE + tid; e < nel; e += NT) {
                        const int i = tri[e] >> 8, j = tri[e] & 0xff;
                        Ls[i][j] = __ldcg(p.V + (long long)(d0 + i) * R + d0 + j);
                    }
                    __syncthreads();
                }
                if (!pieces || s_flag) factor_block(p.Linv + (long long)(k + 1) * NB * NB, nb1, tol, p.nclamp);
            }
        }
        // tiles 1 .. of the others (tile 0 is done above whenever there is one)
        const int first = G == 1 ? 1 : (bid == 0 ? ntile : bid), stride = G == 1 ? 1 : G - 1;
        // each block's tiles in turn; the operands and the C values of the next
        // tile are loaded into registers while the current one is multiplied
        TrailTile cur{}, nxt{};
        double pa[4], pb[4], pc[4];
        int tile = first;
        if (tile < ntile) {
            cur = trail_tile(p, tile, k0, kb, ntri, Tk, dim);
            trail_fetch(cur, R, kb, tid, tx, ty, pa, pb, pc);
        }
        for (; tile < ntile; tile += stride) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = tid + u * NT;
                Ta[e / NB][e % NB] = pa[u];
                Tb[e / NB][e % NB] = pb[u];
            }
            double c4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) c4[u] = pc[u];
            __syncthreads();
            if (tile + stride < ntile) {
                nxt = trail_tile(p, tile + stride, k0, kb, ntri, Tk, dim);
                trail_fetch(nxt, R, kb, tid, tx, ty, pa, pb, pc);
            }
            double a00 = 0, a01 = 0, a10 = 0, a11 = 0;
            for (int s2 = 0; s2 < kb; ++s2) {
                const double x0 = Ta[ty][s2], x1 = Ta[ty + 16][s2];
                const double y0 = Tb[tx][s2], y1 = Tb[tx + 16][s2];
                a00 = fma(x0, y0, a00);
                a01 = fma(x0, y1, a01);
                a10 = fma(x1, y0, a10);
                a11 = fma(x1, y1, a11);
            }
            const double acc[4] = {a00, a01, a10, a11};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = ty + 16 * (u >> 1), j = tx + 16 * (u & 1);
                if (trail_owns(cur, i, j)) cur.C[(long long)i * R + j] = c4[u] - acc[u];
            }
            __syncthreads();
            cur = nxt;
        }
        if (!gsync(p, target, &s_flag, bid, G)) return;
    }

    // ---- P2: back substitution U~ L = Z, RB rows at a time ------------------------
    {
        __shared__ double xs[2][RB][NB];
        const int rpc = (dim + G - 1) / G;
        const int rbeg = bid * rpc, rend = min(dim, rbeg + rpc);
        for (int r0 = rbeg; r0 < rend; r0 += RB) {
            switch (min(RB, rend - r0)) {
                case 4: back_rows<4>(p, r0, xs, Ls, Li, Ta, Tb); break;
                case 3: back_rows<3>(p, r0, xs, Ls, Li, Ta, Tb); break;
                case 2: back_rows<2>(p, r0, xs, Ls, Li, Ta, Tb); break;
                default: back_rows<1>(p, r0, xs, Ls, Li, Ta, Tb); break;
            }
        }
    }
    constexpr int T16 = 16;
    const int ty16 = tid / T16, tx16 = tid % T16;
    if (!gsync(p, target, &s_flag, bid, G)) return;

    // ---- P3: normalise: 32 columns per block, 8 row groups, a zero column keeps lam = 0
    {
        const int c = tid % 32, rg = tid / 32;
        for (int cb = bid; cb * 32 < R; cb += G) {
            const int r = cb * 32 + c;
            double s = 0.0;
            if (r < R)
                for (int x = rg; x < dim; x += NT / 32) {
                    const double u = __ldcg(p.U + (long long)x * R + r);
                    s = fma(u, u, s);
                }
            Ta[rg][c] = s;
            __syncthreads();
            if (rg == 0) {
                double t = 0.0;
                for (int q = 0; q < NT / 32; ++q) t += Ta[q][c];
                Tb[0][c] = t;
            }
            __syncthreads();
            if (r < R) {
                const double l = sqrt(Tb[0][c]);
                const double inv = (l > 0.0) ? 1.0 / l : 1.0;
                for (int x = rg; x < dim; x += NT / 32) p.U[(long long)x * R + r] = __ldcg(p.U + (long long)x * R + r) * inv;
                if (rg == 0) p.lam[r] = l;
            }
            __syncthreads();
        }
    }
    if (!gsync(p, target, &s_flag, bid, G)) return;

    // ---- P4: Gram of the new factor, 16 x 16 tiles of the lower triangle ------------
    const int TR = (R + T16 - 1) / T16;
    const int ntri = TR * (TR + 1) / 2;
    // each block's (tile, 32-row step) pairs in turn, the next pair's operands
    // loaded into registers while the current one is multiplied
    {
        const int nx = (dim + NB - 1) / NB;
        int tile = bid, xs = 0;
        int ti0 = 0, tj0 = 0;              // the current tile's corner
        if (tile < ntri) {
            int I, J;
            tri_index(tile, I, J);
            ti0 = I * T16;
            tj0 = J * T16;
        }
        int ni0 = ti0, nj0 = tj0;          // the next pair's tile corner
        double qa[2], qb[2];
        if (tile < ntri) gram_fetch(p, ti0, tj0, 0, tid, qa, qb);
        double acc = 0.0;
        while (tile < ntri) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int e = tid + u * NT;
                Ta[e / T16][e % T16] = qa[u];
                Tb[e / T16][e % T16] = qb[u];
            }
            __syncthreads();
            int ntl = tile, nxs = xs + 1;
            if (nxs == nx) {
                ntl += G;
                nxs = 0;
                if (ntl < ntri) {
                    int I, J;
                    tri_index(ntl, I, J);
                    ni0 = I * T16;
                    nj0 = J * T16;
                }
            }
            if (ntl < ntri) gram_fetch(p, ni0, nj0, nxs * NB, tid, qa, qb);
#pragma unroll 8
            for (int x = 0; x < NB; ++x) acc = fma(Ta[x][ty16], Tb[x][tx16], acc);
            __syncthreads();
            if (nxs == 0) {
                const int i = ti0 + ty16, j = tj0 + tx16;
                if (i < R && j < R) {
                    p.G[(long long)i * R + j] = acc;
                    p.G[(long long)j * R + i] = acc;
                }
                acc = 0.0;
            }
            tile = ntl;
            xs = nxs;
            ti0 = ni0;
            tj0 = nj0;
        }
    }
}

__global__ void __launch_bounds__(NT, 1) k_solve(const __grid_constant__ SolveP p) {
    solve_body(p, blockIdx.x, gridDim.x);
    leave_sync(p, gridDim.x);
}

// Several instances' mode updates in one cooperative launch.  The blocks form
// lanes: lane l is blocks lane_blk0[l] .. lane_blk0[l+1]-1 and solves the
// instances order[lane_inst0[l]] .. order[lane_inst0[l+1]-1] one after the
// other, each with its own barrier words, so the lanes proceed independently
// and only share the SMs.
constexpr int MAX_BATCH = 64;
struct SolveBatch {
    int n, nl;
    int lane_blk0[MAX_BATCH + 1];
    int lane_inst0[MAX_BATCH + 1];
    int order[MAX_BATCH];
    SolveP p[MAX_BATCH];
};

__global__ void __launch_bounds__(NT, 3) k_solve_batch(const __grid_constant__ SolveBatch b) {
    int l = 0;
    while (l + 1 < b.nl && b.lane_blk0[l + 1] <= (int)blockIdx.x) ++l;
    const int bid = (int)blockIdx.x - b.lane_blk0[l], G = b.lane_blk0[l + 1] - b.lane_blk0[l];
    for (int i = b.lane_inst0[l]; i < b.lane_inst0[l + 1]; ++i) {
        solve_body(b.p[b.order[i]], bid, G);
        leave_sync(b.p[b.order[i]], G);
        __syncthreads();   // the block's shared memory is reused by the next instance
    }
}

int g_solve_grid = 0;

}  // namespace

namespace {

SolveP to_params(const SolveArgs& a) {
    SolveP p;
    p.G1 = a.G1; p.G2 = a.G2; p.G3 = a.G3; p.V = a.V; p.Linv = a.Linv; p.M = a.M; p.Z = a.Z;
    p.U = a.U; p.lam = a.lam; p.G = a.G;
    p.sync = a.sync; p.nclamp = a.nclamp; p.err = a.err; p.R = a.R; p.dim = a.dim;
    p.withhold = a.withhold;
    p.wait_ns = a.wait_ns > 0 ? a.wait_ns : BAR_NS;
    return p;
}

int sm_total() {
    if (g_solve_grid == 0) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) return -1;
        g_solve_grid = sms;   // one block per SM: the look-ahead block keeps its SM's FP64 pipe
    }
    return g_solve_grid;
}

// blocks one instance can use: enough for the first block step's tiles and panel
// rows, at least 8, at most one per SM
int solve_want(int dim, int R, int sms) {
    const int t0 = (R > NB) ? (R - NB + NB - 1) / NB : 0;
    const int d = (dim + NB - 1) / NB;
    int want = t0 * (t0 + 1) / 2 + d * t0;
    const int ptask = (R + dim + 7) / 8;
    if (ptask > want) want = ptask;
    if (want < 8) want = 8;
    return want < sms ? want : sms;
}

int g_batch_per_sm = 0;

// blocks of each of n instances (at least 2, at most want[k], cap together) such that all
// of them take the same modelled time, the shortest possible one, which is returned; 0
// when there is none
double own_lanes(int n, int cap, const int* want, const double* work, const double* steps, double rate_blk, double step_s,
                 int* blocks) {
    auto fits = [&](double T, int* G) {
        int sum = 0;
        for (int k = 0; k < n; ++k) {
            const double left = T - steps[k] * step_s;
            if (left <= 0.0 || work[k] > left * rate_blk * want[k]) return false;
            const int g = (int)ceil(work[k] / (left * rate_blk));
            G[k] = g < 2 ? 2 : g;
            sum += G[k];
        }
        return sum <= cap;
    };
    double lo = 0.0, hi = 1.0;
    if (!fits(hi, blocks)) return 0.0;
    for (int it = 0; it < 40; ++it) {
        int G[MAX_BATCH];
        const double T = 0.5 * (lo + hi);
        if (fits(T, G)) {
            hi = T;
            for (int k = 0; k < n; ++k) blocks[k] = G[k];
        } else {
            lo = T;
        }
    }
    return hi;
}

}  // namespace

int solve_mode_coop(const double* G1, const double* G2, const double* G3, const double* M, int dim, int R,
                    double* V, double* Linv, double* Z, double* U, double* lam, double* G,
                    unsigned int* sync, unsigned long long* nclamp, unsigned int* err,
                    int grid_cap, unsigned long long wait_ns, unsigned int* withhold, cudaStream_t s) {
    const int sms = sm_total();
    if (sms <= 0) return -1;
    // small problems take fewer blocks, so that several instances' solves can share the GPU
    int grid = solve_want(dim, R, sms);
    if (grid_cap > 0 && grid > grid_cap) grid = grid_cap < 8 ? 8 : grid_cap;
    SolveArgs a{G1, G2, G3, M, dim, R, V, Linv, Z, U, lam, G, sync, nclamp, err, wait_ns, withhold};
    const SolveP p = to_params(a);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_solve, p);
    return e == cudaSuccess ? 0 : -(1000 + (int)e);
}

int solve_modes_batched(const SolveArgs* a, int n, cudaStream_t s) {
    const int sms = sm_total();
    if (sms <= 0) return -1;
    if (g_batch_per_sm == 0) {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_solve_batch, NT, 0) != cudaSuccess || per <= 0) {
            cudaGetLastError();
            return -2;
        }
        g_batch_per_sm = per;
    }
    for (int k0 = 0; k0 < n; k0 += MAX_BATCH) {
        const int nb = (n - k0 < MAX_BATCH) ? n - k0 : MAX_BATCH;
        // Two blocks per SM for few instances: a third one's FP64 instructions stretch the
        // factorisations of the others' diagonal blocks by more than it brings (sweeps of 6
        // instances 6.00 ms with three and 5.44 with two, 16 instances 27.97 and 27.69; but
        // 24 instances 38.4 and 43.1, 64 79.1 and 81.9)
        const int per_sm = nb <= 16 && g_batch_per_sm > 2 ? 2 : g_batch_per_sm;
        const int cap = per_sm * sms;   // blocks that are co-resident in one cooperative launch
        if (2 * nb > cap) return -3;
        SolveBatch b;
        b.n = nb;
        int want[MAX_BATCH];
        double work[MAX_BATCH], steps[MAX_BATCH];
        for (int k = 0; k < nb; ++k) {
            const SolveArgs& x = a[k0 + k];
            want[k] = solve_want(x.dim, x.R, sms);
            work[k] = (double)x.R * x.R * x.R / 3.0 + 4.0 * x.dim * (double)x.R * x.R;
            steps[k] = (double)((x.R + NB - 1) / NB);
            b.p[k] = to_params(x);
        }
        // Lanes: L lanes of cap / L blocks; each instance goes to one lane, longest
        // first to the least loaded.  Modelled time of an instance on G blocks: its
        // FP64 work at G blocks' share of the FP64 rate (2 FMA per clock per SM at
        // about 2 GHz, shared by the blocks of an SM) plus a latency per 32-wide
        // block step; L is the one with the shortest modelled makespan.
        const double rate_blk = 8.0e9 / per_sm, step_s = 20e-6;
        auto est = [&](int k, int G) { return work[k] / ((double)(G < want[k] ? G : want[k]) * rate_blk) + steps[k] * step_s; };
        int best_L = 0, best_lane[MAX_BATCH] = {};
        double best_span = 0.0;
        for (int L = 1; L <= nb; ++L) {
            const int W = cap / L;
            if (W < 2) break;
            int idx[MAX_BATCH], lane[MAX_BATCH];
            double t[MAX_BATCH], load[MAX_BATCH];
            for (int k = 0; k < nb; ++k) {
                idx[k] = k;
                t[k] = est(k, W);
            }
            std::sort(idx, idx + nb, [&](int x, int y) { return t[x] > t[y]; });
            for (int l = 0; l < L; ++l) load[l] = 0.0;
            for (int q = 0; q < nb; ++q) {
                int lmin = 0;
                for (int l = 1; l < L; ++l)
                    if (load[l] < load[lmin]) lmin = l;
                lane[idx[q]] = lmin;
                load[lmin] += t[idx[q]];
            }
            double span = 0.0;
            for (int l = 0; l < L; ++l) span = load[l] > span ? load[l] : span;
            if (best_L == 0 || span < best_span) {
                best_L = L;
                best_span = span;
                for (int k = 0; k < nb; ++k) best_lane[k] = lane[k];
            }
        }
        if (best_L == 0) return -3;
        // Or every instance in a lane of its own, with as many blocks as its work needs to
        // finish at the same time T as the others: the shortest such T, by bisection.
        // Equal lanes leave the SMs of the small instances idle while the largest one
        // ends.  Sweeps of uneven batches: 16 instances of v 50 .. 234 29.2 -> 27.7 ms, 24
        // 40.3 -> 38.4, four to eight instances 10 to 20 per cent less.
        int own[MAX_BATCH];
        const double own_span = own_lanes(nb, cap, want, work, steps, rate_blk, step_s, own);
        // (not below 14 blocks each: 40 instances 59.7 ms against 57.5 in equal lanes)
        const bool use_own = own_span > 0.0 && own_span < best_span && cap >= 14 * nb;
        if (use_own) best_L = nb;
        b.nl = best_L;
        int blk = 0, q = 0;
        for (int l = 0; l < best_L; ++l) {
            b.lane_blk0[l] = blk;
            blk += use_own ? own[l] : cap / best_L + (l < cap % best_L ? 1 : 0);
            b.lane_inst0[l] = q;
            for (int k = 0; k < nb; ++k)
                if (use_own ? k == l : best_lane[k] == l) b.order[q++] = k;
        }
        b.lane_blk0[best_L] = blk;
        b.lane_inst0[best_L] = q;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blk);
        cfg.blockDim = dim3(NT);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k_solve_batch, b);
        if (e != cudaSuccess) return -(1000 + (int)e);
    }
    return 0;
}

// ---- self-test of the pivot reciprocal --------------------------------------

namespace {

__global__ void k_recip_check(const double* d, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = recip_nr(d[i]);
}

}  // namespace

extern "C" int ppl_test_reciprocal(const double* d, double* out, int n, void* stream) {
    if (!d || !out || n < 0) return 1;   // PPL_EINVAL
    if (n == 0) return 0;
    k_recip_check<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(d, out, n);
    const cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) return 3;   // PPL_ECUDA
    return 0;
}
