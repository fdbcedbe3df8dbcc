// FP64 contraction on the tensor cores by exact digit products, C = alpha A B^T
// (+ beta C), same operands, maps and results as the CUDA-core kernel k_gemm64.
//
// GB300 executes two FP64 FMAs per clock per SM (1.25 TFLOP/s in all), so every
// FP64 contraction of the library was bound by that pipe.  Here each row of A and
// each row of B (column of the product) is scaled by the power of two above its
// largest entry and written as a 64-bit fixed-point number in eight balanced
// base-256 digits (after Ozaki, Ogita, Oishi & Rump, "Error-free transformations of
// matrix multiplication", Numer. Algorithms 59, 2012; for matrix units, Mukunoki et
// al., ISC 2020).  A digit with its weight, d 256^-i, is exact in bf16, a product of
// two is d d' 256^-(i+j) with |d d'| <= 2^14, and up to 7 x 128 products of one weight
// add up below 2^24 units, so tcgen05.mma with its FP32 accumulator forms those sums
// without rounding.  There are seven accumulators, for the weights 0 .. 6; the last also
// takes the products of weight 7, the least kept (its rounding is below the unit of the
// result's last digit).  Every 128 values of k they are folded into an integer
// accumulator of 88 bits, and the result is rounded to FP64 once.
//
// Error: the fixed-point rounding of the entries, 2^-64 of the row's power of two, and
// the products of weight 8 and above: together about sqrt(n) 2^-64 of the product of the
// two rows' powers of two (n non-zero terms, each worth seven products of two digits;
// at most 7 n 2^-64).  An FMA chain errs by 2^-54 of the sum of the |terms| and more.  So
// an eighth accumulator sums the products of the leading digits' absolute values, in
// units of 2^-14 of that product: where it reaches 32 sqrt(n) (n at most the smaller
// number of non-zero entries of the two rows), the digits add no more than 2^-55 of the
// sum of the |terms| (at most 3.5 / sqrt(n) of n FMA roundings).  An element for which it
// does not is formed by FP64 FMAs, as are those of a row with an Inf, a NaN or only
// entries below 2^-959; one whose terms are all zero (the sum then is exactly zero) is
// not.  Against exact sums, max / rms in units of the sum
// of the |terms|, FMA chain in brackets: K 8 .. 64, half of each row scaled by 1/32 ..
// 1/128 where the other is large, 0.9e-16 / 2.8e-17 (2.9e-16 / 5.2e-17); entries spread
// over 2^16, K 32, 0.9e-16 / 3.4e-17 (7.0e-16 / 1.4e-16); normal entries, K 32, 0.6e-16 /
// 1.3e-17 (2.9e-16 / 5.3e-17).  (Seven digits reached 1.4e-15 .. 2.8e-15 in the first.)
//
// Bound: the digit extraction (integer instructions run at half rate on GB300; each
// tile extracts the rows that it shares with others again), with the MMAs (74 of
// 128 x 64 x 16 per 32 values of k, 64 clocks each) under it, then the rounding and
// writing of the tile.  Measured: an energy at o = 20, v = 200, X = 600, R = 800, two
// contractions of M = 12000, N = 800, K = 200, 0.857 ms in all (the same with seven digits
// and the rows' norms in place of their counts), 21.7 ms with k_gemm64 and 20-row tiles.
#include "ppl_internal.h"
#include "ppl_gemm64.cuh"
#include "ppl_ptx.cuh"

namespace {

constexpr int EM = 128, EN = 64, EK = 32;      // tile and k block
constexpr int EWORK = 512;                     // threads that extract digits and fold: warps 0 .. 15
constexpr int ETHREADS = EWORK + 128;          // and a warpgroup of which warp 16 issues the MMAs
// Registers: 96 per thread at launch; the control warpgroup hands some to the workers
// (88-bit sums of 16 columns each): 128 * 64 + 512 * 104 = 640 * 96 (checked on the host
// when a handle is made: a split above the launch's allocation would wait forever).
// Sixteen working warps, not eight with twice the sums: the digit extraction is a
// stream of dependent integer instructions.
constexpr int EREG_LAUNCH = 96, EREG_CTRL = 64, EREG_WORK = 104;
static_assert((ETHREADS - EWORK) * EREG_CTRL + EWORK * EREG_WORK == ETHREADS * EREG_LAUNCH, "register split");
constexpr int NDIG = 8;                        // digits; plane 8 holds |leading digit|
constexpr int NSUM = 7;                        // accumulators of their products
constexpr int FOLD = 4;                        // k blocks per exact FP32 accumulation
// A pair of digit planes shares one 128-byte row: plane p at bytes 64 (p & 1) .. + 63 of
// the rows of pair p / 2, the 128 rows of A and then the 64 of B.  Plane 8 follows, A's
// at bytes 0 .. 63 and B's at bytes 64 .. 127 of the same rows.
constexpr uint32_t BOFF = EM * 128, PAIR = (EM + EN) * 128, GOFF = 4 * PAIR;
constexpr uint32_t ESTAGE = GOFF + EM * 128;
constexpr int CPITCH = EN + 1;
// Two stages and the static arrays, rounded up to the stages' alignment, are exactly the
// 227 KB a block can have.
constexpr size_t ESMEM = 2 * ESTAGE;
// After the products, over the stages: the sums, the guard's limits, the offsets in C, the
// elements below their limit, and which entries are not zero, KBITS of every row at a time
constexpr int KBITS = 1024;
constexpr uint32_t LIMOFF = EM * CPITCH * 12, OFFOFF = LIMOFF + (EM + EN) * 4, BADOFF = OFFOFF + (EM + EN) * 8;
// Up to this many of a tile's 8192 elements a warp forms each by FP64 FMAs (some 240 clocks
// per element at K = 250), beyond it the block computes the whole tile (2 FMAs per clock).
// Reconstruction at o 16, v 150, R 500, with the whole tile for any such element before:
// rows with a tenth of their entries 4.74 -> 2.37 ms, of two symmetry blocks 2.38 -> 0.73,
// all four factors with a tenth 6.44 -> 1.06, entries spread over 2^40 6.44 -> 6.08, full
// rows 0.63 (k_gemm64: 5.72, whatever the entries).
constexpr int MAXBAD = 2048;
constexpr uint32_t BITOFF = BADOFF + MAXBAD * 2, BITPITCH = KBITS / 32 + 1;
constexpr unsigned int LBAD = 0xffffffffu;     // in place of a low sum word: element below its limit
constexpr float GUARD2 = 1024.0f;              // 32 squared, per non-zero entry (see above)
constexpr unsigned long long EWAIT_NS = 500ull * 1000ull * 1000ull;
static_assert(BITOFF + (EM + EN) * BITPITCH * 4 <= ESMEM && BITOFF % 4 == 0 && EM * EN <= 65536 && OFFOFF % 8 == 0, "the output tile is staged over the operand stages");
static_assert(FOLD * EK * (NSUM * (1 << 14) + NDIG * (1 << 6)) < (1 << 24), "exact FP32 sums");

// k -> offset of km, for k0 and the k after it
struct KOff {
    int q, r;
};
__device__ __forceinline__ KOff koff(const Idx2& km, int k) {
    KOff o;
    o.q = km.div >= (1 << 30) ? 0 : k / km.div;
    o.r = k - o.q * km.div;
    return o;
}
__device__ __forceinline__ long long knext(const Idx2& km, KOff& o) {
    const long long at = (long long)o.q * km.hi + (long long)o.r * km.lo;
    if (++o.r == km.div) {
        o.r = 0;
        ++o.q;
    }
    return at;
}

// k range of one split-K slice
__host__ __device__ __forceinline__ int slice_len(int K, int ksplit) { return ((K + ksplit - 1) / ksplit + EK - 1) / EK * EK; }

// ---- the rows' largest entries and counts -----------------------------------------

// A row's largest entry (the high word of its magnitude, 0 only for a row of zeros)
// and its number of non-zero entries.
struct RowStat {
    unsigned int hi, n;
};
__device__ __forceinline__ void stat_add(RowStat& s, double x) {
    const unsigned int h = (unsigned int)__double2hiint(x) & 0x7fffffffu;
    const bool nz = (h | (unsigned int)__double2loint(x)) != 0u;
    s.hi = max(s.hi, h | (nz ? 1u : 0u));        // (the lowest bit is not used)
    s.n += nz ? 1u : 0u;
}
__device__ __forceinline__ void stat_merge(RowStat& s, unsigned int hi, unsigned int n) {
    s.hi = max(s.hi, hi);
    s.n += n;
}

// One operand: `rows` rows (map rm) of K entries (map km) for nb batch entries bs
// apart, in ksplit slices of `per` entries; entry (batch * ksplit + slice) * rows + row
// of the output.
struct RowArgs {
    const double* p;
    Idx2 rm, km;
    long long bs;
    int rows, K, ksplit, per, nb, nblk;
    RowStat* out;
};
constexpr int RM_WARP_K = 512;     // a warp per row up to this K, then a block per row

// Bound: memory (each operand is read once; the products read it once per tile of
// the other).  Lanes run along whichever index is contiguous.
__global__ void __launch_bounds__(256) k_rowstat(const __grid_constant__ RowArgs a, const __grid_constant__ RowArgs b) {
    __shared__ RowStat red[8][33];
    const bool second = (int)blockIdx.x >= a.nblk;
    const RowArgs& x = second ? b : a;
    const int blk = second ? (int)blockIdx.x - a.nblk : (int)blockIdx.x;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    RowStat m{0u, 0u};
    if (x.km.lo == 1) {
        const bool wr = x.per <= RM_WARP_K;
        const long long e = wr ? (long long)blk * 8 + warp : blk;          // (batch, slice, row)
        const bool ok = e < (long long)x.rows * x.nb * x.ksplit;
        if (ok) {
            const int bt = (int)(e / x.rows);
            const double* p = x.p + (long long)(bt / x.ksplit) * x.bs + ixd(x.rm, (int)(e % x.rows));
            const int kbeg = bt % x.ksplit * x.per, kend = min(x.K, kbeg + x.per);
            const int st = wr ? 32 : 256;
#pragma unroll 4
            for (int k = kbeg + (wr ? lane : threadIdx.x); k < kend; k += st) stat_add(m, __ldg(p + ixd(x.km, k)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            stat_merge(m, __shfl_xor_sync(0xffffffffu, m.hi, o), __shfl_xor_sync(0xffffffffu, m.n, o));
        if (wr) {
            if (ok && lane == 0) x.out[e] = m;
            return;
        }
        if (lane == 0) red[0][warp] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) stat_merge(m, red[0][w].hi, red[0][w].n);
            x.out[e] = m;
        }
        return;
    }
    const int per = (x.rows + 31) / 32;
    const int bt = blk / per, row = (blk % per) * 32 + lane;
    if (row < x.rows) {
        const double* p = x.p + (long long)(bt / x.ksplit) * x.bs + ixd(x.rm, row);
        const int kbeg = bt % x.ksplit * x.per, kend = min(x.K, kbeg + x.per);
#pragma unroll 4
        for (int k = kbeg + warp; k < kend; k += 8) stat_add(m, __ldg(p + ixd(x.km, k)));
    }
    red[warp][lane] = m;
    __syncthreads();
    if (warp == 0 && row < x.rows) {
        for (int w = 1; w < 8; ++w) stat_merge(m, red[w][lane].hi, red[w][lane].n);
        x.out[(long long)bt * x.rows + row] = m;
    }
}

// barrier 3 over the working threads
__device__ __forceinline__ void work_sync() { asm volatile("bar.sync 3, 512;" ::: "memory"); }

// a >> d, 0 from d = 64 on
__device__ __forceinline__ unsigned long long shr_clamp(unsigned long long a, unsigned int d) {
    unsigned long long r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(d));
    return r;
}

// the nine planes of four entries as pairs of consecutive k, w[plane][pair].
// emax: the exponent field of the largest entry of the pair's row, in place (bits
// 20 .. 30), at least 64 << 20 (rows below that are left to the FP64 tile, whatever is
// written here).
__device__ __forceinline__ void digits4(const double (&v)[4], const int (&emx)[2], uint32_t (&w)[NDIG + 1][2]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float f[2][NDIG];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int hi = __double2hiint(v[2 * j + u]), lo = __double2loint(v[2 * j + u]);
            // |x| = m 2^(ex - 1075), m < 2^53; X = round(x 2^(63 - e)), 2^e the power of two
            // above the row's maximum, is m 2^(10 - d), d = emax - ex; one bit more is kept
            // for the rounding (a zero has d >= 64 and shifts out)
            const unsigned int d = (unsigned int)((emx[j] - (hi & 0x7ff00000)) >> 20);
            const unsigned long long m = shr_clamp(
                ((unsigned long long)(__funnelshift_l((unsigned int)lo, (unsigned int)hi, 11) | 0x80000000u) << 32) |
                    ((unsigned int)lo << 11), d);
            // balanced digits: the lower seven with 128 added are the bytes of
            // t = X + 128 (256^0 + .. + 256^6), the leading one, -128 .. 128, is what carries on
            const unsigned int sg = (unsigned int)(hi >> 31);
            const unsigned long long q = (m >> 1) + (m & 1u);
            uint32_t tl, th, tc;
            asm("add.cc.u32 %0, %3, %5;\n\taddc.cc.u32 %1, %4, 0x00808080;\n\taddc.u32 %2, %6, 0;"
                : "=r"(tl), "=r"(th), "=r"(tc)
                : "r"((uint32_t)q ^ sg), "r"((uint32_t)(q >> 32) ^ sg), "r"(0x80808080u - sg), "r"(sg));
            // a byte in the mantissa of 2^23 (the second one: 256 times it) less its offset, times
            // the digit's weight 256^-i: one exact FMA
            f[u][0] = __int_as_float(0x4B400000 + (int)__funnelshift_r(th, tc, 24)) - 12582912.0f;
            f[u][1] = fmaf(__uint_as_float(__byte_perm(th, 0x4B000000u, 0x7442)), 0x1p-8f, -8388736.0f * 0x1p-8f);
            f[u][2] = fmaf(__uint_as_float((th & 0xff00u) | 0x4B000000u), 0x1p-24f, -32896.0f * 0x1p-16f);
            f[u][3] = fmaf(__uint_as_float((th & 0xffu) | 0x4B000000u), 0x1p-24f, -8388736.0f * 0x1p-24f);
            f[u][4] = fmaf(__uint_as_float(__byte_perm(tl, 0x4B000000u, 0x7443)), 0x1p-32f, -8388736.0f * 0x1p-32f);
            f[u][5] = fmaf(__uint_as_float(__byte_perm(tl, 0x4B000000u, 0x7442)), 0x1p-40f, -8388736.0f * 0x1p-40f);
            f[u][6] = fmaf(__uint_as_float((tl & 0xff00u) | 0x4B000000u), 0x1p-56f, -32896.0f * 0x1p-48f);
            f[u][7] = fmaf(__uint_as_float((tl & 0xffu) | 0x4B000000u), 0x1p-56f, -8388736.0f * 0x1p-56f);
        }
        // the upper halves are the bf16 values (eight significant bits)
#pragma unroll
        for (int p = 0; p < NDIG; ++p)
            w[p][j] = __byte_perm(__float_as_uint(f[0][p]), __float_as_uint(f[1][p]), 0x7632);
        w[NDIG][j] = w[0][j] & 0x7fff7fffu;
    }
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, unsigned long long ad, unsigned long long bd, uint32_t idesc,
                                         uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}

// four columns of the seven digit-sum accumulators (EN columns apart); the wait is part
// of the statement, so that nothing reads the registers before it
__device__ __forceinline__ void tmem_ld_sums(uint32_t taddr, uint32_t (&s)[NSUM][4]) {
    static_assert(NSUM == 7 && EN == 64, "spelled out below");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%28];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4, %5, %6, %7}, [%29];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8, %9, %10, %11}, [%30];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12, %13, %14, %15}, [%31];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16, %17, %18, %19}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20, %21, %22, %23}, [%33];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24, %25, %26, %27}, [%34];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(s[0][0]), "=r"(s[0][1]), "=r"(s[0][2]), "=r"(s[0][3]), "=r"(s[1][0]), "=r"(s[1][1]),
          "=r"(s[1][2]), "=r"(s[1][3]), "=r"(s[2][0]), "=r"(s[2][1]), "=r"(s[2][2]), "=r"(s[2][3]),
          "=r"(s[3][0]), "=r"(s[3][1]), "=r"(s[3][2]), "=r"(s[3][3]), "=r"(s[4][0]), "=r"(s[4][1]),
          "=r"(s[4][2]), "=r"(s[4][3]), "=r"(s[5][0]), "=r"(s[5][1]), "=r"(s[5][2]), "=r"(s[5][3]),
          "=r"(s[6][0]), "=r"(s[6][1]), "=r"(s[6][2]), "=r"(s[6][3])
        : "r"(taddr + 0u), "r"(taddr + 64u), "r"(taddr + 128u), "r"(taddr + 192u), "r"(taddr + 256u),
          "r"(taddr + 320u), "r"(taddr + 384u)
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr)
                 : "memory");
}

// m 2^e outside the normal range of the fast path below
__device__ __noinline__ double scale_slow(unsigned long long m, int e) { return ldexp((double)m, e); }

// (H 2^24 + L) 2^e rounded to nearest (ties up), 0 <= L < 2^24.  Integer instructions
// only (FP64 conversions and multiplies would cost 64 clocks per warp each).
__device__ __forceinline__ double fixed_to_double(long long H, unsigned int L, int e) {
    const unsigned int sgn = (unsigned int)(H >> 63);
    // magnitude
    unsigned int l = sgn ? (0x1000000u - L) & 0xffffffu : L;
    unsigned long long h = sgn ? ~(unsigned long long)H + (L == 0u ? 1ull : 0ull) : (unsigned long long)H;
    if (h < (1ull << 40)) {       // bring the leading bit into h
        h = (h << 24) | l;
        l = 0u;
        e -= 24;
    }
    if (h == 0ull) return 0.0;
    const int lz = __clzll((long long)h);
    const unsigned long long lw = (unsigned long long)l << 40;
    const unsigned long long w = (h << lz) | ((lw >> 1) >> (63 - lz));    // leading 64 bits, weight 2^(e + 24 - lz)
    const unsigned long long m = (w >> 11) + ((unsigned int)(w >> 10) & 1u);       // a carry to 2^53 is right below
    const int ex = e + 24 - lz + 63 + 1023;       // exponent field of the leading bit
    double r = __longlong_as_double((long long)(m + ((unsigned long long)(unsigned int)(ex - 1) << 52)));
    if (ex < 1 || ex > 2045) r = scale_slow(m, e + 24 - lz + 11);
    return __hiloint2double(__double2hiint(r) | (int)(sgn & 0x80000000u), __double2loint(r));
}

__device__ __noinline__ void write_scaled(const G64& g, double* p, double x) {
    x *= g.alpha;
    if (g.atomic)
        atomicAdd(p, x);
    else
        *p = g.beta != 0.0 ? fma(g.beta, *p, x) : x;
}

struct SplitArgs {
    G64 g;
    const RowStat *ha, *hb;          // k_rowstat of A and B
    int ba, bb;                      // 1: per batch entry, 0: one operand for all
};

__global__ void __launch_bounds__(ETHREADS, 1) k_gemm64_split(const __grid_constant__ SplitArgs sa_) {
    const G64& g = sa_.g;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ int s_ex[EM + EN];              // the rows' exponent fields, in place
    __shared__ long long s_row[EM + EN];       // the rows' offsets in A and B
    __shared__ unsigned long long s_bar[5];    // full[2], empty[2], folded
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail, s_bad, s_zeros, s_empty;

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int ntm = (g.M + EM - 1) / EM, ntn = (g.N + EN - 1) / EN;
    // the operand with fewer tiles varies fastest, so that concurrent blocks share the
    // larger one's rows in L2
    const int t = blockIdx.x;
    const int mt = ntm <= ntn ? t % ntm : t / ntn, nt = ntm <= ntn ? t / ntm : t % ntn;
    const int m0 = mt * EM, n0 = nt * EN;
    const int b = blockIdx.z / g.ksplit, ks = blockIdx.z % g.ksplit;
    const int per = slice_len(g.K, g.ksplit);
    const int kbeg = ks * per, kend = min(g.K, kbeg + per);
    if (kbeg >= kend) return;          // a split slice past the end (atomic outputs only)
    const int nkb = (kend - kbeg + EK - 1) / EK;

    const uint32_t base = smem_u32(sm);
    if (base & 1023u) {                // (the swizzled tiles need the alignment asked for above)
        if (tid == 0) atomicOr(g.err, 256u);
        return;
    }
    const uint32_t full0 = smem_u32(&s_bar[0]), bar0 = smem_u32(&s_bar[2]), folded = smem_u32(&s_bar[4]);
    if (tid == 0) {
        s_fail = 0;
        s_bad = 0;
        s_zeros = 0;
        s_empty = 0;
        // the test of the bounded waits: one arrival more than there are warps, so that the
        // first stage never fills and every wait behind it runs out
        const bool starve = blockIdx.x == 0 && blockIdx.z == 0 && g.withhold && *(volatile unsigned int*)g.withhold != 0u &&
                            atomicExch(g.withhold, 0u) != 0u;
        mbar_init(full0, EWORK / 32 + (starve ? 1 : 0));
        mbar_init(full0 + 8, EWORK / 32);
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        mbar_init(folded, EWORK / 32);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    float lim = 0.0f;                  // the limit of row `tid`
    if (tid < EM + EN) {
        const int i = tid;
        const bool isb = i >= EM;
        const int r = isb ? n0 + i - EM : m0 + i;
        const bool ok = r < (isb ? g.N : g.M);
        // (a row past the end stands for row 0: its sums are never written)
        const RowStat st = !ok ? RowStat{0u, 0u}
                           : isb ? sa_.hb[(long long)(b * sa_.bb * g.ksplit + ks) * g.N + r]
                                 : sa_.ha[(long long)(b * sa_.ba * g.ksplit + ks) * g.M + r];
        s_ex[i] = (int)max(st.hi & 0x7ff00000u, 64u << 20);        // a zero row has zero digits
        // no limit for a zero row; a row with an Inf, a NaN or nothing above 2^-959 never passes
        lim = (st.hi >= 0x7ff00000u || (st.hi >> 20) < 64u) && st.hi != 0u ? -1.0f : GUARD2 * (float)st.n;
        if (st.n > 0u && st.n < (unsigned int)(kend - kbeg)) s_zeros = 1;
        s_row[i] = !ok ? 0 : ixd(isb ? g.bn : g.am, r);
    }
    if (warp == EWORK / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    volatile int* vfail = &s_fail;
    // wait for the MMAs of k block kb
    auto done = [&](int kb) { return mbar_wait(bar0 + 8u * (kb & 1), (uint32_t)(kb >> 1) & 1u, g.wait_ns); };
    if (warp >= EWORK / 32) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(EREG_CTRL) : "memory");
        if (warp != EWORK / 32) return;
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)EN >> 3 << 17) | ((uint32_t)(EM >> 4) << 24);
            int kb = 0;
            for (; kb < nkb && !*vfail; ++kb) {
                if ((kb > 0 && kb % FOLD == 0 && !mbar_wait(folded, (uint32_t)(kb / FOLD - 1) & 1u, g.wait_ns)) ||
                    !mbar_wait(full0 + 8u * (kb & 1), (uint32_t)(kb >> 1) & 1u, g.wait_ns)) {
                    *vfail = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t sa = base + (uint32_t)(kb & 1) * ESTAGE, sb = sa + BOFF;
#pragma unroll
                for (int kk = 0; kk < EK / 16; ++kk) {
#pragma unroll
                    for (int i = 0; i < NDIG; ++i) {
                        const unsigned long long da = make_desc(sa + (uint32_t)(i >> 1) * PAIR) + (unsigned long long)(((i & 1) * 64 + kk * 32) >> 4);
#pragma unroll
                        for (int j = 0; i + j < NDIG; ++j) {
                            const unsigned long long db = make_desc(sb + (uint32_t)(j >> 1) * PAIR) + (unsigned long long)(((j & 1) * 64 + kk * 32) >> 4);
                            // weight i + j, weight 7 with weight 6; the first product of an
                            // accumulator is that of i = 0
                            mma_bf16(tmem + (uint32_t)(min(i + j, NSUM - 1) * EN), da, db, idesc,
                                     (kb % FOLD > 0 || kk > 0 || i > 0 || j >= NSUM) ? 1u : 0u);
                        }
                    }
                    const unsigned long long gd = make_desc(sa + GOFF) + (unsigned long long)((kk * 32) >> 4);
                    mma_bf16(tmem + (uint32_t)(NSUM * EN), gd, gd + (64 >> 4), idesc, (kb > 0 || kk > 0) ? 1u : 0u);
                }
                mma_commit(bar0 + 8u * (kb & 1));
            }
            // what was issued finishes before TMEM is given back
            if (kb > 0 && !done(kb - 1)) *vfail = 1;
        }
        __syncwarp();
        // the workers have read what they need of TMEM
        asm volatile("bar.sync 2, 544;" ::: "memory");
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(EREG_WORK) : "memory");
    const double* A = g.A + (long long)b * g.ab;
    const double* B = g.B + (long long)b * g.bb;

    // A k block is three steps of 64 rows x 32 k (A, A, B), four entries per thread.
    // Along a contiguous k a warp covers 4 rows, half a warp a row (pairs of k, 256
    // contiguous bytes per row); otherwise a warp covers 32 rows at one k.
    const bool akf = g.ak.lo == 1, bkf = g.bk.lo == 1;
    auto step_row = [&](int u, bool kf, int i) { return u * 64 + (kf ? warp * 4 + i * 2 + (lane >> 4) : tid & 63); };
    auto load = [&](int u, int kb, double (&v)[4]) {
        const bool isb = u == 2, kf = isb ? bkf : akf;
        const Idx2& km = isb ? g.bk : g.ak;
        const double* p = isb ? B : A;
        const int k0 = kbeg + kb * EK + (kf ? (lane & 15) * 2 : (tid >> 6) * 4);
        if (kf) {
            long long o0 = k0, o1 = k0 + 1;
            if (km.div < (1 << 30)) {
                KOff ko = koff(km, k0);
                o0 = knext(km, ko);
                o1 = knext(km, ko);
            }
            const bool k0ok = k0 < kend, k1ok = k0 + 1 < kend;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const double* r = p + s_row[step_row(u, true, i)];
                v[2 * i] = k0ok ? __ldg(r + o0) : 0.0;
                v[2 * i + 1] = k1ok ? __ldg(r + o1) : 0.0;
            }
        } else {
            const double* r = p + s_row[step_row(u, false, 0)];
            if (km.div >= (1 << 30) && kbeg + (kb + 1) * EK <= kend) {
                r += (long long)k0 * km.lo;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[j] = __ldg(r);
                    r += km.lo;
                }
            } else {
                KOff ko = koff(km, k0);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const long long o = knext(km, ko);
                    v[j] = k0 + j < kend ? __ldg(r + o) : 0.0;
                }
            }
        }
    };

    constexpr int NC = 16;             // columns per thread
    const int q = warp & 3, c0 = (warp >> 2) * NC;
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
    long long H[NC];
    unsigned int L[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        H[j] = 0;
        L[j] = 0u;
    }
    double v[4];
    load(0, 0, v);
    // digits of block kb into stage kb % 2 while the MMAs of block kb - 1 run; every FOLD
    // blocks (and after the last) the FP32 sums go into the integer sums.  The loops
    // stay rolled: unrolled, the kernel ran at the rate of instruction misses.
#pragma unroll 1
    for (int kb = 0; kb <= nkb && !*vfail; ++kb) {
        if (kb < nkb) {
            if (kb >= 2 && !done(kb - 2)) {
                *vfail = 1;
                break;
            }
#pragma unroll 1
            for (int u = 0; u < 3; ++u) {
                const bool isb = u == 2, kf = isb ? bkf : akf;
                double cur[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) cur[j] = v[j];
                if (u < 2)
                    load(u + 1, kb, v);
                else if (kb + 1 < nkb)
                    load(0, kb + 1, v);
                int emx[2];
                uint32_t w[NDIG + 1][2];
                unsigned char* op = sm + (uint32_t)(kb & 1) * ESTAGE;
                if (kf) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) emx[i] = s_ex[step_row(u, true, i)];
                    digits4(cur, emx, w);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        // the rows of B follow those of A in every pair's rows
                        const uint32_t r = (uint32_t)step_row(u, true, i);
                        unsigned char* q0 = op + r * 128u + (((uint32_t)(lane & 15) * 4u) ^ ((r & 7u) << 4));
                        unsigned char* q1 = op + r * 128u + ((64u + (uint32_t)(lane & 15) * 4u) ^ ((r & 7u) << 4));
#pragma unroll
                        for (int p = 0; p < NDIG; ++p) *(uint32_t*)(((p & 1) ? q1 : q0) + (p >> 1) * PAIR) = w[p][i];
                        *(uint32_t*)((isb ? q1 - BOFF : q0) + GOFF) = w[NDIG][i];
                    }
                } else {
                    const uint32_t r = (uint32_t)step_row(u, false, 0);
                    emx[0] = emx[1] = s_ex[r];
                    digits4(cur, emx, w);
                    unsigned char* q0 = op + r * 128u + (((uint32_t)(tid >> 6) * 8u) ^ ((r & 7u) << 4));
                    unsigned char* q1 = op + r * 128u + ((64u + (uint32_t)(tid >> 6) * 8u) ^ ((r & 7u) << 4));
#pragma unroll
                    for (int p = 0; p < NDIG; ++p) *(uint2*)(((p & 1) ? q1 : q0) + (p >> 1) * PAIR) = make_uint2(w[p][0], w[p][1]);
                    *(uint2*)((isb ? q1 - BOFF : q0) + GOFF) = make_uint2(w[NDIG][0], w[NDIG][1]);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(full0 + 8u * (kb & 1));
        }
        if (kb == nkb || (kb > 0 && kb % FOLD == 0)) {
            if (!done(kb - 1)) {
                *vfail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr float unit[NSUM] = {1.0f, 0x1p8f, 0x1p16f, 0x1p24f, 0x1p32f, 0x1p40f, 0x1p48f};
#pragma unroll
            for (int j0 = 0; j0 < NC; j0 += 4) {
                uint32_t s[NSUM][4];
                tmem_ld_sums(tq + (uint32_t)j0, s);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    int d[NSUM];
#pragma unroll
                    for (int w = 0; w < NSUM; ++w) d[w] = __float2int_rn(__uint_as_float(s[w][j]) * unit[w]);
                    const long long lo = (long long)d[4] * 65536 + (long long)d[5] * 256 + d[6] + (long long)L[j0 + j];
                    H[j0 + j] += (long long)(d[0] * 256 + d[1]) * 65536 + (d[2] * 256 + d[3]) + (lo >> 24);
                    L[j0 + j] = (unsigned int)lo & 0xffffffu;
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (kb < nkb && lane == 0) mbar_arrive(folded);
        }
    }
    // the MMAs have read the operands
    float* s_lim = (float*)(sm + LIMOFF);
    long long* s_off = (long long*)(sm + OFFOFF);
    if (tid < EM + EN) {
        s_lim[tid] = lim;
        s_off[tid] = tid < EM ? ixd(g.cm, m0 + tid) : ixd(g.cn, n0 + tid - EM);
    }
    work_sync();
    const bool failed = *vfail != 0;
    unsigned int bad = 0u, empty = 0u;      // of this thread's columns: below the limit, a sum of zero
    if (!failed) {
        const float la = s_lim[q * 32 + lane];
#pragma unroll 1
        for (int j0 = 0; j0 < NC; j0 += 8) {
            uint32_t s[8];
            tmem_ld8(tq + (uint32_t)(NSUM * EN + j0), s);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float t = fminf(la, s_lim[EM + c0 + j0 + j]), sum = __uint_as_float(s[j]);
                if ((t < 0.0f || sum * sum < t) && n0 + c0 + j0 + j < g.N) bad |= 1u << (j0 + j);
                if (t > 0.0f && sum == 0.0f) empty |= 1u << (j0 + j);
            }
        }
        if (m0 + q * 32 + lane >= g.M) bad = 0u;
        empty &= bad;
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    asm volatile("bar.arrive 2, 544;" ::: "memory");
    if (s_zeros) {
        // Sums whose terms are all exactly zero (rows of disjoint support) are zero as they
        // stand: where rows have zeros, the guard's zero sums are looked through entry by entry.
        if (empty) s_empty = 1;
        work_sync();
        uint32_t* s_bits = (uint32_t*)(sm + BITOFF);
        for (int k0 = kbeg; k0 < kend && s_empty; k0 += KBITS) {
            for (int i = warp; i < EM + EN; i += EWORK / 32) {
                const double* p = i < EM ? A + s_row[i] : B + s_row[i];
                const Idx2& km = i < EM ? g.ak : g.bk;
                for (int k = k0; k < min(kend, k0 + KBITS); k += 32) {
                    const bool nz = k + lane < kend && __double_as_longlong(__ldg(p + ixd(km, k + lane))) << 1 != 0;
                    const unsigned int w = __ballot_sync(0xffffffffu, nz);
                    if (lane == 0) s_bits[i * BITPITCH + (k - k0) / 32] = w;
                }
            }
            work_sync();
            for (unsigned int x = empty; x != 0u; x &= x - 1u) {
                const int j = __ffs(x) - 1;
                unsigned int any = 0u;
                for (int w = 0; w < (min(kend - k0, KBITS) + 31) / 32; ++w)
                    any |= s_bits[(q * 32 + lane) * BITPITCH + w] & s_bits[(EM + c0 + j) * BITPITCH + w];
                if (any) empty &= ~(1u << j);
            }
            work_sync();
        }
        bad &= ~empty;
    }
    unsigned short* s_list = (unsigned short*)(sm + BADOFF);
    if (bad) {
        int at = atomicAdd(&s_bad, __popc(bad));
        for (unsigned int x = bad; x != 0u && at < MAXBAD; x &= x - 1u, ++at)
            s_list[at] = (unsigned short)((q * 32 + lane) * EN + c0 + __ffs(x) - 1);
    }
    // stage the sums in shared memory
    long long* sH = (long long*)sm;
    unsigned int* sL = (unsigned int*)(sH + EM * CPITCH);
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        sH[(q * 32 + lane) * CPITCH + c0 + j] = H[j];
        sL[(q * 32 + lane) * CPITCH + c0 + j] = (bad >> j) & 1u ? LBAD : L[j];
    }
    work_sync();
    if (failed) {
        if (tid == 0) atomicOr(g.err, 128u);
        return;
    }
    const int nbad = s_bad;
    if (nbad > MAXBAD) {
        // FP64 FMAs for this tile, 256 threads per 64 rows
        const int h = tid / 256;
        if (m0 + h * 64 < g.M)
            gemm64_tile(g, b, m0 + h * 64, n0, kbeg, kend, (double*)sm + h * GBK * (GBM + GBN), tid % 256, h == 0 ? 1 : 4);
        return;
    }
    // round and write along the output's contiguous index
    double* C = g.C + (long long)b * g.cb;
    const bool nfast = g.cn.lo == 1;
    const bool plain = g.alpha == 1.0 && g.beta == 0.0 && !g.atomic;      // (no FP64 instruction per element)
    constexpr int NE = 2;              // elements in flight: each is a chain of some sixty integer instructions
#pragma unroll 1
    for (int e0 = tid; e0 < EM * EN; e0 += NE * EWORK) {
        double x[NE];
        double* p[NE];
#pragma unroll
        for (int y = 0; y < NE; ++y) {
            const int e = e0 + y * EWORK;
            const int ml = nfast ? e / EN : e % EM, nl = nfast ? e % EN : e / EM;
            const int ex = (s_ex[ml] >> 20) + (s_ex[EM + nl] >> 20) - (2 * 1022 + 62);
            const unsigned int l = sL[ml * CPITCH + nl];
            x[y] = fixed_to_double(sH[ml * CPITCH + nl], l, ex);
            p[y] = m0 + ml < g.M && n0 + nl < g.N && l != LBAD ? C + s_off[ml] + s_off[EM + nl] : nullptr;
        }
        if (plain) {
#pragma unroll
            for (int y = 0; y < NE; ++y)
                if (p[y]) *p[y] = x[y];
        } else {
#pragma unroll
            for (int y = 0; y < NE; ++y)
                if (p[y]) write_scaled(g, p[y], x[y]);
        }
    }
    // elements below their limit: a warp each, lanes along k
    for (int i = warp; i < nbad; i += EWORK / 32) {
        const int ml = s_list[i] / EN, nl = s_list[i] % EN;
        const double *a = A + s_row[ml], *bp = B + s_row[EM + nl];
        double x = 0.0;
#pragma unroll 4
        for (int k = kbeg + lane; k < kend; k += 32) x = fma(__ldg(a + ixd(g.ak, k)), __ldg(bp + ixd(g.bk, k)), x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) write_scaled(g, C + s_off[ml] + s_off[EM + nl], x);
    }
}

RowArgs row_args(const double* p, const Idx2& rm, const Idx2& km, long long bs, int rows, int K, int ksplit, int nb,
                 RowStat* out) {
    RowArgs a{p, rm, km, bs, rows, K, ksplit, slice_len(K, ksplit), nb, 0, out};
    const long long n = (long long)rows * nb * ksplit;
    a.nblk = km.lo == 1 ? (int)(a.per <= RM_WARP_K ? (n + 7) / 8 : n) : (rows + 31) / 32 * nb * ksplit;
    return a;
}

}  // namespace

int gemm64_split_init() {
    cudaFuncAttributes fa;
    if (cudaFuncSetAttribute(k_gemm64_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ESMEM) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, k_gemm64_split) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return fa.numRegs == EREG_LAUNCH && fa.maxThreadsPerBlock >= ETHREADS ? 0 : -2;
}

int gemm64_split(const G64& g, cudaStream_t s) {
    if (g.lower) return -5;        // (Gram matrices of the CUDA-core form only)
    const long long tiles = (long long)((g.M + EM - 1) / EM) * ((g.N + EN - 1) / EN);
    const long long z = (long long)g.batch * g.ksplit;
    // grid limits, and K 2^38 of the integer sums below 2^63
    if (tiles > 0x7fffffffll || z > 65535 || g.K / g.ksplit >= (1 << 24)) return -2;
    SplitArgs a;
    a.g = g;
    if (a.g.wait_ns == 0) a.g.wait_ns = EWAIT_NS;
    a.ba = g.ab != 0;
    a.bb = g.bb != 0;
    const long long na = (long long)g.M * (a.ba ? g.batch : 1) * g.ksplit, nb = (long long)g.N * (a.bb ? g.batch : 1) * g.ksplit;
    // a Gram matrix has one operand
    const bool same = g.A == g.B && g.ab == g.bb && g.M == g.N && g.am.hi == g.bn.hi && g.am.lo == g.bn.lo &&
                      g.am.div == g.bn.div && g.ak.hi == g.bk.hi && g.ak.lo == g.bk.lo && g.ak.div == g.bk.div;
    if (!g.scratch || na + (same ? 0 : nb) > g.nscratch || na > 0x7fffffffll || nb > 0x7fffffffll) return -4;
    RowStat* st = (RowStat*)g.scratch;
    a.ha = st;
    a.hb = same ? st : st + na;
    const RowArgs ra = row_args(g.A, g.am, g.ak, g.ab, g.M, g.K, g.ksplit, a.ba ? g.batch : 1, st);
    RowArgs rb = row_args(g.B, g.bn, g.bk, g.bb, g.N, g.K, g.ksplit, a.bb ? g.batch : 1, st + na);
    if (same) rb.nblk = 0;
    k_rowstat<<<ra.nblk + rb.nblk, 256, 0, s>>>(ra, rb);
    k_gemm64_split<<<dim3((unsigned)tiles, 1, (unsigned)z), ETHREADS, ESMEM, s>>>(a);
    return 0;
}
