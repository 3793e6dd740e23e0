// FP64 contractions on the sm_103a tensor cores by exact digit products.
//
// GB300 runs FP64 at 1/64 of its FP32 rate (1.2 TFLOP/s), so the FP64 form's
// contractions were bound by the FP64 pipe at a few per cent of the memory
// rate.  Here every operand is written as an integer of 54 bits relative to a
// power of two (of its row of A, of its column of X), cut into six balanced
// base-512 digits d in [-256, 256] (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59, 2012).  Digits are exact in fp16, a
// product of two is at most 2^16, and the FP32 accumulator of tcgen05.mma
// holds the sum of a group (the pairs i + j = s) exactly up to 2^24: over 256
// reals of K for s = 10 (one pair), 128 for s = 9, 64 for s = 8 and 7, the lengths
// after which these are read out.  s = 6 (5 pairs) is read out every 128 reals, s = 5
// and 4 (6 and 5 pairs) every 512: their sums can reach 2^25.3, 2^27.6 and 2^27.3
// and are rounded past 2^24, as constant operands often do for s = 5 and 4.  Were every
// product of the largest size and one sign, with the accumulator's last bit lost at
// each, that were 2^-51.6 of K times the row's and the column's largest entries for s
// = 6 and 2^-58 for the others; the cut of the operands is 2^-53 of it at most.
// (Read out every 64 reals, s = 6 still passes 2^24, for a seventh more read-outs,
// which bound the large products.)  The groups s = 4 .. 10 are kept (26 of 36 pairs;
// the dropped ones are below the 2^-54 of the cut itself), read out and added up as
// 64-bit integers: what order the K slices meet in changes nothing, how many there are
// only what s = 4 to 6 round.  The accuracy is relative to the largest entries of a row
// and a column: a column that decays over six decades comes out of the direct sum
// with 1.4 to 1.8 times FP64's error in the norm, a flat one with about half of it.
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "dg.h"
#include "rtd.h"
#include "rttddft.h"
#include "tcgen05.cuh"

namespace cg = cooperative_groups;

#define DG_P 6              // digits of an operand: 54 bits
// in the Chebyshev series, 63 bits: 34 of 49 pairs, s = 5 .. 12, of which s = 9 and above are
// exact, s = 8 and 7 read out every 64 reals and rounded past 2^24
#define DG_PS 7
#define DG_KS 32            // reals per stage: 64 bytes of fp16, one row of the 64-byte swizzle
#define DG_BM 128           // rows per tile
// smallest i + j kept with P digits, and the groups kept, s = dg_s0(P) + g, of NT columns of tensor memory each
__host__ __device__ constexpr int dg_s0(int P) { return P - 2; }
__host__ __device__ constexpr int dg_ng(int P) { return 2 * (P - 1) - dg_s0(P) + 1; }
#define DG_THREADS 320      // 8 read-out warps, one product warp, one copy warp
// and 256 (16 columns) or 128 threads that generate the left operand (GEN): with more columns the
// read-out's integers need the registers
__host__ __device__ constexpr int dg_gen(int NT) { return NT == 16 ? 256 : 128; }
#define DG_A_PL (DG_BM * 64)

// slices of 64 reals that a group collects before it is read out; g counted from the largest s (of
// 1, 2, 3, ... pairs), the two smallest ones last
__host__ __device__ constexpr int dg_run(int P, int g) {
    const int t = dg_ng(P) - 1 - g;
    return t == 0 ? 4 : (t == 1 ? 2 : (g < 2 ? 8 : (P == 6 && t == 4 ? 2 : 1)));
}

typedef long long i64;

// ------------------------------------------------------------ digits
// q = sum_i d_i 512^i with |q| <= 2^(9 P - 1), returned as the P biased values
// d_i + 256 (0 .. 512)
template <int P>
__device__ __forceinline__ void dg_cut(i64 q, uint32_t* d) {
    unsigned long long bias = 0ull;
#pragma unroll
    for (int i = 0; i < P; ++i) bias += 256ull << (9 * i);
    const unsigned long long u = (unsigned long long)q + bias;
#pragma unroll
    for (int i = 0; i < P - 1; ++i) d[i] = (uint32_t)(u >> (9 * i)) & 511u;
    d[P - 1] = (uint32_t)(u >> (9 * (P - 1)));
}
// fp16 pair (x - 256, y - 256) of biased digits: 1024 + x is exact in fp16
__device__ __forceinline__ uint32_t dg_pair(uint32_t x, uint32_t y) {
    const uint32_t b = (x | (y << 16)) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&b), __floats2half2_rn(1280.f, 1280.f));
    return *reinterpret_cast<const uint32_t*>(&h);
}
#define DG_NEG 0x8000u
// exponent e with |x| < 2^e from the high word of the largest |x|; 2048 marks Inf and NaN
__device__ __forceinline__ int dg_exp(int hw) {
    const int f = hw >> 20;
    return f == 2047 ? 2048 : f - 1022;
}
__device__ __forceinline__ int dg_hw(double x) { return __double2hiint(x) & 0x7fffffff; }
// x 2^(53 - e) as an integer; the power of two is applied in two halves so that neither overflows
struct DgScale {
    double p1, p2;
};
__device__ __forceinline__ double dg_pow2(int n) { return __hiloint2double((n + 1023) << 20, 0); }
__device__ __forceinline__ DgScale dg_scale(int e) {
    const int s = 53 - e, h = s / 2;
    return DgScale{dg_pow2(h), dg_pow2(s - h)};
}
__device__ __forceinline__ i64 dg_int(double x, DgScale s) { return __double2ll_rn((x * s.p1) * s.p2); }

// (hi 2^SH + lo) 2^e as a double with integer arithmetic (the conversions of
// the FP64 pipe would cost more than the products of a short K)
template <int SH>
__device__ __forceinline__ double dg_double(i64 hi, i64 lo, int e) {
    i64 m = hi + (lo >> SH);
    unsigned long long r = (unsigned long long)lo & ((1ull << SH) - 1ull);
    const bool neg = m < 0;
    if (neg) {
        const bool b = r != 0ull;
        m = -m - (b ? 1 : 0);
        r = b ? (1ull << SH) - r : 0ull;
    }
    // keep the leading 63 bits of m 2^SH + r
    const int lz = __clzll(m);
    const int k = lz > SH ? SH : lz - 1;
    const unsigned long long x = ((unsigned long long)m << k) | (r >> (SH - k));
    if (x == 0ull) return 0.0;
    const int z = __clzll(x);
    const unsigned long long t = ((x << z) + (1ull << 10));  // the carry out of a value of all ones:
    const bool cy = t < (1ull << 10);
    const int ex = e + (SH - k) + 63 - z + (cy ? 1 : 0) + 1023;
    const unsigned long long man = cy ? 0ull : (t >> 11) & ((1ull << 52) - 1ull);
    double v;
    if (ex >= 1 && ex <= 2046) {
        v = __longlong_as_double((i64)(((unsigned long long)ex << 52) | man));
    } else if (ex > 2046) {
        v = __longlong_as_double(0x7ff0000000000000ll);
    } else {
        v = scalbn(__longlong_as_double((i64)((1023ull << 52) | man)), ex - 1023);
    }
    return neg ? -v : v;
}

// Operands lie tile by tile as a block of k_dg takes them: per tile of RT rows
// and stage of 16 complex k, P planes of RT rows of 64 bytes, the 16-byte
// chunks of a row permuted as the 64-byte swizzle wants them.  A stage is one
// contiguous copy (as boxes of a row-major array, 64 bytes a row, the copies
// gave 4.9 TB/s over the chip).  Word (two fp16) of row r, complex k, plane 0;
// the planes are RT 16 words apart.
template <int P>
__host__ __device__ __forceinline__ size_t dg_word(int r, int k, int RT, int nst) {
    const int rr = r % RT;
    return (((size_t)(r / RT) * nst + (k >> 4)) * P * RT + rr) * 16 + ((((k >> 2) & 3) ^ ((rr >> 1) & 3)) << 2) + (k & 3);
}
// rows 2n: [Re, -Im] and 2n + 1: [Im, Re] of a right operand, entry k of complex column n
template <int P>
__device__ __forceinline__ void dg_put_col(uint32_t* b, int NT, int nst, int n, int k, i64 qr, i64 qi) {
    uint32_t dr[P], di[P];
    dg_cut<P>(qr, dr);
    dg_cut<P>(qi, di);
    b += dg_word<P>(2 * n, k, NT, nst);
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const uint32_t p = dg_pair(dr[i], di[i]);
        b[(size_t)i * NT * 16] = p ^ (DG_NEG << 16);
        b[(size_t)i * NT * 16 + 16] = (p >> 16) | (p << 16);
    }
}

// ------------------------------------------------------------ the product kernel
struct DgOut {
    const unsigned char *A, *B;  // operands of the product
    int M, nst, nsta, ldc;       // rows, K stages of X and of A (at least as many), leading dimension of C
    const int* er;      // row exponents of A
    const int* ec;      // column exponents of X
    zd* C;
    const double* scale;  // factor on the product, or null
    const int* glin;    // GEN: table offsets of the G set
    int tile0;          // first tile in the split buffers
};
struct DgCheb {
    int n;              // N_aux
    zd *y0, *y1;        // y of even and of odd terms: [ns][n]
    zd* acc;            // sum_n c_n y_n
    const double* diag; // of H~
    uint32_t* Bn[2];    // digit operands of even and odd terms
    int nst;
    const zd* coef;     // c_n
};
struct DgArgs {
    const DgOut* out;
    const DgCheb* ch;
    int kofs, ncol, ntn, cs, gs, beta, term, last;  // cs K slices per cluster, gs clusters per tile
    i64* part;
    unsigned* cnt;
    int* flag;
    const uint4* tab4;   // GEN: digits 0 .. 3 of every table entry, (re, im) pairs,
    const uint2* tab2;   // digits 4 and 5,
    const int* tabe;     // and the exponent of the table
    int center;
};

__device__ __forceinline__ uint64_t dg_desc(uint32_t saddr) {  // K-major, 64-byte swizzle, 8-row atoms of 512 B
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}
__device__ __forceinline__ void dg_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
template <int W>
__device__ __forceinline__ void dg_ld(uint32_t taddr, uint32_t* r) {
    static_assert(W == 8 || W == 16, "columns per load");
    if constexpr (W == 8) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(taddr));
    } else {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr));
    }
}
// digits of a mode's operands, and stages of shared memory
__host__ __device__ constexpr int dg_p(int mode) { return mode == 1 ? DG_PS : DG_P; }
__host__ __device__ constexpr int dg_stages(int NT, int mode) { return mode == 1 ? (NT == 64 ? 2 : 3) : (NT == 16 ? 4 : 3); }

// One 128-row x NT-column tile of D = A^ B^^T over this split's K stages (NT
// real columns: Re and Im of NT / 2 complex ones).  The copy warp brings the
// P digit planes of both operands of a stage with one bulk copy each.  A group has
// its own NT columns of tensor memory in the order of s, and X's digit planes
// lie one after another in shared memory, so digit i of A meets a run of X's
// digits in one product of up to N = 256 (9 instructions per 16 reals for
// NT = 64 instead of 26, 6 for fewer columns: a product reads A's 128 rows once
// whatever its N).  The read-out warps add a finished group (64 reals of K) to
// their integers while the products of the others run; a group is handed back
// and forth by a pair of mbarriers.  The K slices of a tile meet in the
// distributed shared memory of a cluster, further clusters of the tile in
// global memory, where the last one finishes it.
// MODE 0: C (+)= the product, scaled back.  MODE 1: a Chebyshev term.  GEN: the left
// operand is V~_(G - G') of the table (Eq. v_interstitial): eight more warps write
// a stage's planes from the table's digits, 24 bytes an entry through L1, loaded
// before the wait for the stage's slot.
template <int NT, int MODE, bool GEN>
__global__ void __launch_bounds__(DG_THREADS + (GEN ? dg_gen(NT) : 0), 1) k_dg(const DgArgs g) {
    extern __shared__ unsigned char dgsm[];
    constexpr int P = dg_p(MODE), T = P - 1, S0 = dg_s0(P), G = dg_ng(P);  // digits, the largest one, groups
    constexpr int STAGES = dg_stages(NT, MODE);
    constexpr int B_PL = NT * 64;
    constexpr int STAGE = P * (DG_A_PL + B_PL);
    constexpr int CP = NT / 2;  // columns per read-out thread
    constexpr uint32_t NCOLS = G * NT <= 128 ? 128 : (G * NT <= 256 ? 256 : 512);
    constexpr int GH = G - 4, SH = 9 * GH;  // groups GH .. go to hi, in units of 2^SH of lo's
    unsigned char* smem = dgsm + ((1024u - (smem_u32(dgsm) & 1023u)) & 1023u);
    constexpr int THREADS = DG_THREADS + (GEN ? dg_gen(NT) : 0);
    __shared__ __align__(8) uint64_t full[STAGES], fullA[STAGES], empty[STAGES], gfull[G], gfree[G], done;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int is_last;
    const int z = blockIdx.z + g.kofs;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = blockIdx.x % g.cs, nt_i = (blockIdx.x / g.cs) % g.ntn;
    const int sp = blockIdx.x / (g.cs * g.ntn) * g.cs + rank, splits = g.cs * g.gs;
    const int m_i = blockIdx.y;
    const DgOut& o = g.out[z];
    const int m0 = m_i * DG_BM, n0 = nt_i * NT;
    if (m0 >= o.M) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int st0 = (int)((i64)o.nst * sp / splits), nk = (int)((i64)o.nst * (sp + 1) / splits) - st0;
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&fullA[s], dg_gen(NT) / 32);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < G; ++s) {
            mbar_init(&gfull[s], 1);
            mbar_init(&gfree[s], 8);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(NCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    i64 hi[CP], lo[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) hi[c] = lo[c] = 0;
    if (warp == 9) {
        if (lane == 0) {
            int issued = 0;
            const unsigned char* ga = o.A + ((size_t)m_i * o.nsta + st0) * (P * DG_A_PL);
            const unsigned char* gb = (MODE == 0 ? o.B : (const unsigned char*)g.ch[z].Bn[(g.term - 1) & 1]) +
                                      ((size_t)nt_i * o.nst + st0) * (P * B_PL);
            for (int t = 0; t < nk; ++t) {
                const int s = t % STAGES;
                if (t >= STAGES && !mbar_wait(&empty[s], (uint32_t)((t / STAGES - 1) & 1))) {
                    abort_flag = 1;
                    atomicOr(g.flag, 8);
                    break;
                }
                if (abort_flag) break;
                unsigned char* sa = smem + s * STAGE;
                mbar_expect_tx(&full[s], GEN ? P * B_PL : STAGE);
                if (!GEN) dg_copy(sa, ga + (size_t)t * (P * DG_A_PL), P * DG_A_PL, &full[s]);
                dg_copy(sa + P * DG_A_PL, gb + (size_t)t * (P * B_PL), P * B_PL, &full[s]);
                issued = t + 1;
            }
            // nothing may still be on its way into shared memory when the block ends
            for (int t = issued > STAGES ? issued - STAGES : 0; t < issued; ++t)
                mbar_wait(&full[t % STAGES], (uint32_t)((t / STAGES) & 1));
        }
    } else if (warp == 8) {
        if (lane == 0) {
            // kind::f16, fp16 operands, FP32 accumulator, both K-major
            const uint32_t idesc0 = (1u << 4) | ((uint32_t)(DG_BM >> 4) << 24);
            constexpr int WMAX = 256 / NT < P ? 256 / NT : P;  // digits of X per product
            bool ok = true;
            for (int t = 0; t < nk && ok; ++t) {
                const int s = t % STAGES;
                if (!mbar_wait(&full[s], (uint32_t)((t / STAGES) & 1)) ||
                    (GEN && !mbar_wait(&fullA[s], (uint32_t)((t / STAGES) & 1)))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const bool first = (t & 1) == 0, lastp = !first || t == nk - 1;
                const int sl = t >> 1;
                const uint64_t da = dg_desc(smem_u32(smem + s * STAGE));
                const uint64_t db = dg_desc(smem_u32(smem + s * STAGE + P * DG_A_PL));
                // digit i of A times the digits j .. j + w - 1 of X in one product of N = w NT
                auto mma = [&](int kk, int i, int j, int w, uint32_t acc) {
                    umma_bf16(tmem + (uint32_t)((i + j - S0) * NT), da + (uint64_t)((i * DG_A_PL + kk * 32) >> 4),
                              db + (uint64_t)((j * B_PL + kk * 32) >> 4),
                              idesc0 | ((uint32_t)((w * NT) >> 3) << 17), acc);
                };
                if (first) {
                    // the slice's first products, a group at a time: a group that starts anew waits
                    // for its read-out and overwrites its columns
#pragma unroll
                    for (int q = G - 1; q >= 0; --q) {
                        const bool anew = (sl & (dg_run(P, q) - 1)) == 0;
                        if (anew && sl > 0) {
                            if (!mbar_wait(&gfree[q], (uint32_t)((sl / dg_run(P, q) - 1) & 1))) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                        }
                        if (q > 0) mma(0, T, q + S0 - T, 1, anew ? 0u : 1u);
                        else mma(0, T - 1, 0, 1, anew ? 0u : 1u);
                    }
                    if (!ok) break;
                }
#pragma unroll
                for (int i = T; i >= 0; --i) {
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk) {
                        int j = i < S0 ? S0 - i : 0;
                        if (first && kk == 0) {
                            if (i == T) continue;
                            if (i == T - 1) j = 1;
                        }
#pragma unroll
                        for (; j < P; j += WMAX) mma(kk, i, j, P - j < WMAX ? P - j : WMAX, 1u);
                    }
                    // the largest group that digit i reaches is complete (the smallest two with digit 0)
                    if (lastp) {
                        const int q = i + T - S0;
                        if (t == nk - 1 || (sl & (dg_run(P, q) - 1)) == dg_run(P, q) - 1) umma_commit(&gfull[q]);
                        if (i == 0 && (t == nk - 1 || (sl & (dg_run(P, 0) - 1)) == dg_run(P, 0) - 1)) umma_commit(&gfull[0]);
                    }
                }
                umma_commit(&empty[s]);
            }
            umma_commit(&done);
            if (!ok) {
                abort_flag = 1;
                atomicOr(g.flag, 8);
            }
        }
    } else if (GEN && warp >= 10) {
        // row r, PER of a stage's 16 k in batches of QB; for 16 columns the next batch's entries are on
        // their way while one is written (203 us at N_G 5900, 2 columns, 212 without; 512 threads with
        // fewer registers: 361.  Loads and stores of a stage take 1700 cycles of the L1 pipe, the products
        // 600; the FP64 pipe took 697 us)
        constexpr int PER = 16 * DG_BM / dg_gen(NT), QB = 4, NB = PER / QB;
        constexpr bool AHEAD = NT == 16;
        const int r = (tid - DG_THREADS) & (DG_BM - 1), h = (tid - DG_THREADS) / DG_BM;
        const int row = m0 + r;
        const bool act = row < o.M;
        const int lrow = act ? o.glin[row] + g.center : 0;
        uint4 a4[QB], b4[QB];
        uint2 a2[QB], b2[QB];
        auto load = [&](int t, int b) {
            const int k0 = (st0 + t) * 16 + h * PER + b * QB;
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                b4[q] = make_uint4(0u, 0u, 0u, 0u);
                b2[q] = make_uint2(0u, 0u);
                if (act && k0 + q < o.M) {
                    const int d = lrow - __ldg(o.glin + k0 + q);
                    b4[q] = __ldg(g.tab4 + d);
                    b2[q] = __ldg(g.tab2 + d);
                }
            }
        };
        if (AHEAD && nk > 0) load(0, 0);
        bool ok = true;
        for (int t = 0; t < nk; ++t) {
            const int s = t % STAGES;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                if (!AHEAD) load(t, b);
#pragma unroll
                for (int q = 0; q < QB; ++q) {
                    a4[q] = b4[q];
                    a2[q] = b2[q];
                }
                if (AHEAD) {
                    if (b + 1 < NB) load(t, b + 1);
                    else if (t + 1 < nk) load(t + 1, 0);
                }
                // after a wait that ran out no lane waits again, and none leaves the warp: what is
                // written then is not used
                if (b == 0 && t >= STAGES && ok && (!mbar_wait(&empty[s], (uint32_t)((t / STAGES - 1) & 1)) || abort_flag)) {
                    ok = false;
                    abort_flag = 1;
                    atomicOr(g.flag, 8);
                }
                unsigned char* d = smem + s * STAGE + r * 64;
#pragma unroll
                for (int c = 0; c < QB / 4; ++c) {
                    const int ch = (h * PER + b * QB) / 4 + c;  // the row's 16-byte chunk
                    unsigned char* p = d + ((ch ^ ((r >> 1) & 3)) << 4);
                    const uint4* w = a4 + 4 * c;
                    const uint2* v = a2 + 4 * c;
                    *(uint4*)(p + 0 * DG_A_PL) = make_uint4(w[0].x, w[1].x, w[2].x, w[3].x);
                    *(uint4*)(p + 1 * DG_A_PL) = make_uint4(w[0].y, w[1].y, w[2].y, w[3].y);
                    *(uint4*)(p + 2 * DG_A_PL) = make_uint4(w[0].z, w[1].z, w[2].z, w[3].z);
                    *(uint4*)(p + 3 * DG_A_PL) = make_uint4(w[0].w, w[1].w, w[2].w, w[3].w);
                    *(uint4*)(p + 4 * DG_A_PL) = make_uint4(v[0].x, v[1].x, v[2].x, v[3].x);
                    *(uint4*)(p + 5 * DG_A_PL) = make_uint4(v[0].y, v[1].y, v[2].y, v[3].y);
                }
            }
            // the planes are read by the products' proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&fullA[s])) : "memory");
        }
    } else {
        const int nsl = (nk + 1) >> 1;
        const uint32_t tb = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * CP);
        bool ok = true;
        for (int sl = 0; sl < nsl; ++sl) {
#pragma unroll
            for (int gi = G - 1; gi >= 0; --gi) {
                if (sl != nsl - 1 && (sl & (dg_run(P, gi) - 1)) != dg_run(P, gi) - 1) continue;
                // after a wait that ran out no lane waits again, and none leaves the warp, whose loads
                // below take all of them (a vote, or the block's flag, at each read-out took 2 to 6%
                // of the large products' time)
                if (ok && !mbar_wait(&gfull[gi], (uint32_t)((sl / dg_run(P, gi)) & 1))) ok = false;
                tc_fence_after();
                constexpr int W = CP >= 16 ? 16 : 8;
#pragma unroll
                for (int c0 = 0; c0 < CP; c0 += W) {
                    uint32_t r[W];
                    dg_ld<W>(tb + (uint32_t)(gi * NT + c0), r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (c0 + W >= CP) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0)
                            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&gfree[gi])) : "memory");
                    }
#pragma unroll
                    for (int c = 0; c < W; ++c) {
                        const i64 v = (i64)__float2int_rn(__uint_as_float(r[c]));
                        if (gi >= GH) hi[c0 + c] += v << (9 * (gi - GH));  // units of s = S0 + GH
                        else lo[c0 + c] += v << (9 * gi);                  // units of s = S0
                    }
                }
            }
        }
        if (!ok) {
            abort_flag = 1;
            atomicOr(g.flag, 8);
        }
    }
    __syncthreads();
    // every product has written its accumulator before tensor memory goes back
    // (a block that gave up, with its flag raised, still takes part below: the split
    // buffers and counters are left ready for the next launch)
    if (!mbar_wait(&done, 0) && tid == 0) atomicOr(g.flag, 8);
    tc_fence_after();
    // the stages are free now: the tile's integers go to shared memory, column by
    // column, and the blocks of the cluster (K slices of one tile) each add up and
    // finish their share of the columns
    i64* S = (i64*)smem;  // [NT][hi, lo][128]
    if (warp < 8) {
        const int rl = (warp & 3) * 32 + lane, cb = (warp >> 2) * CP;
#pragma unroll
        for (int c = 0; c < CP; ++c) {
            S[(size_t)(2 * (cb + c)) * DG_BM + rl] = hi[c];
            S[(size_t)(2 * (cb + c) + 1) * DG_BM + rl] = lo[c];
        }
    }
    if (g.cs > 1) cl.sync();
    else __syncthreads();
    const int share = NT / g.cs, c0 = rank * share;  // real columns of this block, an even number
    const int items = DG_BM * share;
    bool mine = true;
    // the sum over the clusters (beside S, which the cluster's other blocks may still read)
    i64* T0 = g.cs > 1 ? S + (size_t)2 * NT * DG_BM : S;
    if (g.gs > 1) {
        const int tile = (o.tile0 + m_i * g.ntn + nt_i) * g.cs + rank;
        unsigned long long* P = (unsigned long long*)g.part + (size_t)tile * share * 2 * DG_BM;
        for (int it = tid; it < 2 * items; it += THREADS) {
            i64 v = 0;
            for (int q = 0; q < g.cs; ++q) v += (g.cs > 1 ? cl.map_shared_rank(S, q) : S)[(size_t)2 * c0 * DG_BM + it];
            atomicAdd(P + it, (unsigned long long)v);
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            is_last = atomicAdd(g.cnt + tile, 1u) == (unsigned)(g.gs - 1);
            if (is_last) g.cnt[tile] = 0u;
        }
        __syncthreads();
        mine = is_last != 0;
        if (mine) {
            __threadfence();
            for (int it = tid; it < 2 * items; it += THREADS) {
                T0[it] = (i64)__ldcg(P + it);
                __stcg(P + it, 0ull);  // ready for the next launch
            }
            __syncthreads();
        }
    }
    constexpr int E0 = 2 * (9 * P - 1) - 9 * S0;  // lo's unit is 2^(er + ec - E0)
    if (mine) {
        for (int it = tid; it < items / 2; it += THREADS) {
            const int rl = it & (DG_BM - 1), row = m0 + rl, c = (it / DG_BM) * 2, n = (n0 + c0 + c) >> 1;
            if (row >= o.M || n >= g.ncol) continue;
            i64 hv[2], lv[2];
            if (g.gs > 1) {
                const i64* T = T0 + (size_t)2 * c * DG_BM + rl;
                hv[0] = T[0];
                lv[0] = T[DG_BM];
                hv[1] = T[2 * DG_BM];
                lv[1] = T[3 * DG_BM];
            } else {
                hv[0] = hv[1] = lv[0] = lv[1] = 0;
                for (int q = 0; q < g.cs; ++q) {
                    const i64* T = (g.cs > 1 ? cl.map_shared_rank(S, q) : S) + (size_t)2 * (c0 + c) * DG_BM + rl;
                    hv[0] += T[0];
                    lv[0] += T[DG_BM];
                    hv[1] += T[2 * DG_BM];
                    lv[1] += T[3 * DG_BM];
                }
            }
            if constexpr (MODE == 0) {
                const int er = GEN ? *g.tabe : o.er[row], ec = o.ec[n];
                zd v;
                if (ec >= 2048 || er >= 2048) {
                    v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
                } else {
                    v.x = dg_double<SH>(hv[0], lv[0], er + ec - E0);
                    v.y = dg_double<SH>(hv[1], lv[1], er + ec - E0);
                }
                if (o.scale) v = zscale(v, *o.scale);
                zd* p = o.C + row + (size_t)n * o.ldc;
                if (g.beta) v = zadd(*p, v);
                *p = v;
            } else {
                // H~ y: its diagonal in FP64, the rest as digits; the recurrence and the sum in FP64
                const DgCheb& ch = g.ch[z];
                zd* yb = (g.term & 1) ? ch.y1 : ch.y0;
                const size_t e = (size_t)n * ch.n + row;
                const int er = o.er[row], ec = o.ec[n];
                const zd yp = ((g.term & 1) ? ch.y0 : ch.y1)[e];
                const double d = ch.diag[row];
                zd y = zmk(fma(d, yp.x, dg_double<SH>(hv[0], lv[0], er + ec - E0)), fma(d, yp.y, dg_double<SH>(hv[1], lv[1], er + ec - E0)));
                if (g.term > 1) {
                    const zd y2 = yb[e];
                    y = zmk(fma(2.0, y.x, -y2.x), fma(2.0, y.y, -y2.y));
                }
                zd sm = ch.acc[e];
                zfma(sm, ch.coef[g.term], y);
                ch.acc[e] = sm;
                if (!g.last) {
                    yb[e] = y;
                    dg_put_col<P>(ch.Bn[g.term & 1], NT, ch.nst, n, row, fix64(y.x, ec, 9 * P - 1), fix64(y.y, ec, 9 * P - 1));
                }
            }
        }
    }
    if (g.cs > 1) cl.sync();  // a block's integers are read before the block may end
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(NCOLS) : "memory");
}

// ------------------------------------------------------------ packing
// element (r, k) of op(A): src[r rs + k cs], conjugated when conj
struct DgSrc {
    const zd* src;
    size_t rs, cs;
    int conj, M, K, nst;
    uint32_t* dst;  // tiles of 128 rows
    int* er;
};
// row exponents: a warp per row
__global__ void k_dg_rowmax(const DgSrc* d) {
    const DgSrc& s = d[blockIdx.z];
    int mx = 0;
    if (s.rs == 1) {  // rows contiguous: 32 rows per block, 8 threads stride K
        const int r = blockIdx.x * 32 + (threadIdx.x & 31);
        if (r < s.M)
            for (int k = threadIdx.x >> 5; k < s.K; k += 8) {
                const zd v = s.src[r + (size_t)k * s.cs];
                mx = max(mx, max(dg_hw(v.x), dg_hw(v.y)));
            }
        __shared__ int sh[8][32];
        sh[threadIdx.x >> 5][threadIdx.x & 31] = mx;
        __syncthreads();
        if (threadIdx.x < 32 && r < s.M) {
            for (int q = 0; q < 8; ++q) mx = max(mx, sh[q][threadIdx.x]);
            s.er[r] = dg_exp(mx);
        }
        return;
    }
    for (int u = 0; u < 4; ++u) {
        const int r = blockIdx.x * 32 + (threadIdx.x >> 5) * 4 + u;
        if (r >= s.M) return;
        mx = 0;
        for (int k = threadIdx.x & 31; k < s.K; k += 32) {
            const zd v = s.src[r * s.rs + (size_t)k * s.cs];
            mx = max(mx, max(dg_hw(v.x), dg_hw(v.y)));
        }
        for (int w = 16; w > 0; w >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, w));
        if ((threadIdx.x & 31) == 0) s.er[r] = dg_exp(mx);
    }
}
// digits of a 32 x 32 tile, read along the source's contiguous axis, written along K
__global__ void k_dg_pack_a(const DgSrc* d) {
    __shared__ zd t[32][33];
    const DgSrc& s = d[blockIdx.z];
    const int k0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    if (r0 >= s.M || k0 >= s.K) return;
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    for (int q = y; q < 32; q += 8) {
        const int r = s.rs == 1 ? r0 + x : r0 + q, k = s.rs == 1 ? k0 + q : k0 + x;
        zd v = zmk(0.0, 0.0);
        if (r < s.M && k < s.K) v = s.src[r * s.rs + (size_t)k * s.cs];
        if (s.conj) v.y = -v.y;
        if (s.rs == 1) t[x][q] = v;
        else t[q][x] = v;
    }
    __syncthreads();
    const int k = k0 + x;
    for (int q = y; q < 32; q += 8) {
        const int r = r0 + q;
        if (r >= s.M || k >= s.K) continue;
        const zd v = t[q][x];
        const int e = s.er[r];
        const DgScale sc = dg_scale(e >= 2048 ? 0 : e);
        uint32_t dr[DG_P], di[DG_P];
        dg_cut<DG_P>(e >= 2048 ? 0 : dg_int(v.x, sc), dr);
        dg_cut<DG_P>(e >= 2048 ? 0 : dg_int(v.y, sc), di);
        for (int i = 0; i < DG_P; ++i)
            s.dst[dg_word<DG_P>(r, k, DG_BM, s.nst) + (size_t)i * DG_BM * 16] = dg_pair(dr[i], di[i]);
    }
}

// right operand: per complex column n of X (K x N) the rows 2n: [Re, -Im] and
// 2n + 1: [Im, Re] of every k, and the column's exponent.  A cluster of eight
// blocks shares a column: the largest entry goes around through distributed
// shared memory, the entries stay in registers meanwhile.
struct DgPackB {
    const zd *X, *X2;  // rows 0 .. K1 - 1 from X, the others from X2
    int ldx, ldx2, K1, K, NT, nst;
    uint32_t* dst;  // tiles of NT rows
    int* ec;
};
#define DG_PB_T 256
#define DG_PB_E 4  // entries per thread held in registers
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(DG_PB_T) k_dg_pack_b(const DgPackB* d, int kofs) {
    __shared__ int sh[8];
    __shared__ int cmax;
    cg::cluster_group cl = cg::this_cluster();
    const DgPackB& s = d[blockIdx.z + kofs];
    const int rank = blockIdx.x & 7, n = blockIdx.x >> 3;
    const int tid = threadIdx.x;
    const zd* __restrict__ x = s.X + (size_t)n * s.ldx;
    const zd* __restrict__ x2 = s.X2 + (size_t)n * s.ldx2 - s.K1;
    auto get = [&](int k) { return k < s.K1 ? x[k] : x2[k]; };
    zd v[DG_PB_E];
    int mx = 0;
#pragma unroll
    for (int u = 0; u < DG_PB_E; ++u) {
        const int k = (u * 8 + rank) * DG_PB_T + tid;
        v[u] = k < s.K ? get(k) : zmk(0.0, 0.0);
        mx = max(mx, max(dg_hw(v[u].x), dg_hw(v[u].y)));
    }
    for (int k = (DG_PB_E * 8 + rank) * DG_PB_T + tid; k < s.K; k += 8 * DG_PB_T) {
        const zd w = get(k);
        mx = max(mx, max(dg_hw(w.x), dg_hw(w.y)));
    }
    for (int w = 16; w > 0; w >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, w));
    if ((tid & 31) == 0) sh[tid >> 5] = mx;
    __syncthreads();
    if (tid == 0) {
        for (int w = 0; w < DG_PB_T / 32; ++w) mx = max(mx, sh[w]);
        cmax = mx;
    }
    cl.sync();
    mx = 0;
    for (int w = 0; w < 8; ++w) mx = max(mx, *cl.map_shared_rank(&cmax, w));
    cl.sync();  // a block's value is read before the block may end
    const int e = dg_exp(mx);
    if (rank == 0 && tid == 0) s.ec[n] = e;
    const bool bad = e >= 2048;
    const DgScale sc = dg_scale(bad ? 0 : e);
    auto put = [&](int k, zd w) {
        dg_put_col<DG_P>(s.dst, s.NT, s.nst, n, k, bad ? 0 : dg_int(w.x, sc), bad ? 0 : dg_int(w.y, sc));
    };
#pragma unroll
    for (int u = 0; u < DG_PB_E; ++u) {
        const int k = (u * 8 + rank) * DG_PB_T + tid;
        if (k < s.K) put(k, v[u]);
    }
    for (int k = (DG_PB_E * 8 + rank) * DG_PB_T + tid; k < s.K; k += 8 * DG_PB_T) put(k, get(k));
}

// ------------------------------------------------------------ host side
struct DgPool {  // device memory of a plan
    std::vector<void*> p;
    bool ok = true;
    void* get(size_t bytes, bool zero) {
        void* q = nullptr;
        if (!ok || cudaMalloc(&q, std::max<size_t>(bytes, 16)) != cudaSuccess) {
            cudaGetLastError();
            ok = false;
            return nullptr;
        }
        p.push_back(q);
        if (zero && cudaMemset(q, 0, std::max<size_t>(bytes, 16)) != cudaSuccess) ok = false;
        return q;
    }
    template <typename T>
    T* up(const std::vector<T>& v) {
        T* q = (T*)get(v.size() * sizeof(T), false);
        if (q && cudaMemcpy(q, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess) ok = false;
        return q;
    }
    void drop() {
        for (void* q : p) cudaFree(q);
        p.clear();
    }
};
static int dg_up(int n, int m) { return (n + m - 1) / m * m; }
static int dg_nt(int ncol) { return 2 * ncol <= 16 ? 16 : (2 * ncol <= 32 ? 32 : 64); }
static int dg_nst(int K) { return (2 * K + DG_KS - 1) / DG_KS; }
static size_t dg_bytes(int rows, int K, int P = DG_P) { return (size_t)P * rows * dg_nst(K) * 64; }

// the stages, or a block's integers and its share of a cluster's sum of them
template <int NT, int MODE>
static constexpr int dg_smem() {
    const int st = dg_stages(NT, MODE) * dg_p(MODE) * (DG_A_PL + NT * 64), ep = 3 * NT * DG_BM * 8;
    return (st > ep ? st : ep) + 1024;
}
template <int MODE, bool GEN>
static const void* dg_fn(int NT, int* smem) {
    *smem = NT == 16 ? dg_smem<16, MODE>() : (NT == 32 ? dg_smem<32, MODE>() : dg_smem<64, MODE>());
    if constexpr (GEN) return NT == 16 ? (const void*)k_dg<16, MODE, true> : (const void*)k_dg<32, MODE, true>;
    else
        return NT == 16 ? (const void*)k_dg<16, MODE, false>
                        : (NT == 32 ? (const void*)k_dg<32, MODE, false> : (const void*)k_dg<64, MODE, false>);
}
template <int MODE, bool GEN>
static cudaError_t dg_attr(int NT) {
    int sm;
    const void* f = dg_fn<MODE, GEN>(NT, &sm);
    return raise_smem(f, sm);
}
template <int MODE, bool GEN>
static void dg_launch(int NT, int mt, int nk, DgArgs a, cudaStream_t s) {
    int sm;
    const void* f = dg_fn<MODE, GEN>(NT, &sm);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.cs * a.ntn * a.gs, mt, nk);
    cfg.blockDim = dim3(DG_THREADS + (GEN ? dg_gen(NT) : 0));
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = a.cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void* args[1] = {&a};
    cudaLaunchKernelExC(&cfg, f, args);
}
// K slices so that the waves of blocks are short.  In units of one stage's
// products (about 0.9 us) a block costs its stages, a start and a read-out worth
// about four, one more for the cluster's exchange and three where clusters
// meet in global memory.  Clusters of eight leave a few of the 152 SMs idle.
static void dg_splits(int tiles, int nst, int* cs, int* gs) {
    double tb = 1e30;
    *cs = *gs = 1;
    for (int c = 1; c <= 8; c *= 2)
        for (int q = 1; q <= 32 && c * q <= std::max(1, nst); ++q) {
            const int room = c == 8 ? 136 : 152;
            const double t = (double)((tiles * c * q + room - 1) / room) *
                             ((nst + c * q - 1) / (c * q) + 4.0 + (c > 1 ? 1.0 : 0.0) + (q > 1 ? 3.0 : 0.0));
            if (t < tb * 0.97) {
                tb = t;
                *cs = c;
                *gs = q;
            }
        }
}

struct DgLeft {
    DgPool pool;
    std::vector<DgSrc> src;
    DgSrc* d_src = nullptr;
    int mm = 1, mk = 1;
};
struct DgGemm {
    DgPool pool;
    int nk = 0, ncol = 0, NT = 0, ntn = 0, mt = 0, cs = 1, gs = 1;
    DgOut* out = nullptr;
    DgPackB* pb = nullptr;
    std::vector<DgPackB> host;
    i64* part = nullptr;
    unsigned* cnt = nullptr;
    int* flag = nullptr;
};

void dg_left_destroy(DgLeft* l) {
    if (!l) return;
    l->pool.drop();
    delete l;
}
void dg_gemm_destroy(DgGemm* g) {
    if (!g) return;
    g->pool.drop();
    delete g;
}

// cut the source's present values
int launch_dg_left(const DgLeft* l, cudaStream_t s) {
    const int nk = (int)l->src.size();
    k_dg_rowmax<<<dim3((l->mm + 31) / 32, 1, nk), 256, 0, s>>>(l->d_src);
    k_dg_pack_a<<<dim3((l->mk + 31) / 32, (l->mm + 31) / 32, nk), 256, 0, s>>>(l->d_src);
    return 2;
}

DgLeft* dg_left_create(int nk, const DgMat* m, cudaStream_t s) {
    DgLeft* l = new DgLeft();
    l->src.resize(nk);
    for (int k = 0; k < nk; ++k) {
        DgSrc& d = l->src[k];
        d.src = m[k].src;
        d.rs = m[k].rs;
        d.cs = m[k].cs;
        d.conj = m[k].conj;
        d.M = m[k].M;
        d.K = m[k].K;
        d.nst = dg_nst(m[k].K);
        const int mp = dg_up(m[k].M, DG_BM);
        d.dst = (uint32_t*)l->pool.get(dg_bytes(mp, m[k].K), true);
        d.er = (int*)l->pool.get(mp * sizeof(int), true);
        l->mm = std::max(l->mm, m[k].M);
        l->mk = std::max(l->mk, m[k].K);
    }
    if (l->pool.ok) l->d_src = l->pool.up(l->src);
    if (l->pool.ok) {
        launch_dg_left(l, s);
        if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) l->pool.ok = false;
    }
    if (!l->pool.ok) {
        dg_left_destroy(l);
        return nullptr;
    }
    return l;
}

// device bytes of dg_left_create
size_t dg_left_bytes(int M, int K) { return dg_bytes(dg_up(M, DG_BM), K); }

// x: a product whose right operands (the same ones) are taken; glin: the left operand is generated
static DgGemm* dg_gemm_build(const DgLeft* l, int nk, const DgRight* r, int ncol, int* flag, int lmod, const DgGemm* x,
                             const int* const* glin) {
    DgGemm* g = new DgGemm();
    g->nk = nk;
    g->ncol = ncol;
    g->NT = glin ? std::min(32, dg_nt(ncol)) : dg_nt(ncol);
    g->ntn = (2 * ncol + g->NT - 1) / g->NT;
    g->flag = flag;
    const int np = g->ntn * g->NT;
    std::vector<DgOut> out(nk);
    g->host.resize(nk);
    std::vector<DgPackB>& pb = g->host;
    int tiles = 0, nst = 1;
    for (int k = 0; k < nk; ++k) {
        const DgSrc& d = l->src[lmod > 0 ? k % lmod : k];
        pb[k].X = r[k].X;
        pb[k].ldx = r[k].ldx;
        pb[k].X2 = r[k].X2 ? r[k].X2 : r[k].X;
        pb[k].ldx2 = r[k].X2 ? r[k].ldx2 : r[k].ldx;
        pb[k].K1 = r[k].X2 ? r[k].K1 : r[k].K;
        pb[k].K = r[k].K;
        pb[k].NT = g->NT;
        pb[k].nst = dg_nst(r[k].K);
        pb[k].dst = x ? x->host[k].dst : (uint32_t*)g->pool.get(dg_bytes(np, r[k].K), true);
        pb[k].ec = x ? x->host[k].ec : (int*)g->pool.get(ncol * sizeof(int), true);
        out[k].A = (const unsigned char*)d.dst;
        out[k].B = (const unsigned char*)pb[k].dst;
        out[k].M = d.M;
        out[k].nst = pb[k].nst;
        out[k].nsta = d.nst;
        out[k].ldc = r[k].ldc;
        out[k].er = d.er;
        out[k].ec = pb[k].ec;
        out[k].C = r[k].C;
        out[k].scale = r[k].scale;
        out[k].glin = glin ? glin[k] : nullptr;
        out[k].tile0 = tiles;
        const int mt = (d.M + DG_BM - 1) / DG_BM;
        g->mt = std::max(g->mt, mt);
        tiles += mt * g->ntn;
        nst = std::max(nst, out[k].nst);
    }
    dg_splits(std::max(tiles, 1), nst, &g->cs, &g->gs);
    if (g->gs > 1) {
        g->part = (i64*)g->pool.get((size_t)tiles * g->NT * 2 * DG_BM * sizeof(i64), true);
        g->cnt = (unsigned*)g->pool.get((size_t)tiles * g->cs * sizeof(unsigned), true);
    }
    if (g->pool.ok) {
        g->out = g->pool.up(out);
        g->pb = g->pool.up(pb);
    }
    if (!g->pool.ok || dg_attr<0, false>(g->NT) != cudaSuccess) {
        dg_gemm_destroy(g);
        return nullptr;
    }
    return g;
}

DgGemm* dg_gemm_create(const DgLeft* l, int nk, const DgRight* r, int ncol, int* flag, int lmod) {
    return dg_gemm_build(l, nk, r, ncol, flag, lmod, nullptr, nullptr);
}

static DgArgs dg_args(const DgGemm* g, int kofs, int beta) {
    DgArgs a{};
    a.out = g->out;
    a.kofs = kofs;
    a.ncol = g->ncol;
    a.ntn = g->ntn;
    a.cs = g->cs;
    a.gs = g->gs;
    a.beta = beta;
    a.part = g->part;
    a.cnt = g->cnt;
    a.flag = g->flag;
    return a;
}

// C (+)= A X for entries kofs .. kofs + nk - 1; packed: X's digits are those of the last call
int launch_dg_gemm(const DgGemm* g, int kofs, int nk, int beta, cudaStream_t s, bool packed) {
    if (!packed) k_dg_pack_b<<<dim3(8 * g->ncol, 1, nk), DG_PB_T, 0, s>>>(g->pb, kofs);
    dg_launch<0, false>(g->NT, g->mt, nk, dg_args(g, kofs, beta), s);
    return packed ? 1 : 2;
}

// ------------------------------------------------------------ interstitial sum
struct DgToep {
    DgPool pool;
    DgGemm* g = nullptr;  // shapes, right operand and split buffers
    bool own = false;     // it packs the right operand itself
    // of V~ (0) and of the step's V~ + s dV~ (1):
    uint4* tab4[2] = {nullptr, nullptr};
    uint2* tab2[2] = {nullptr, nullptr};
    int* hw = nullptr;    // high words of the tables' largest entries
    int* e = nullptr;     // their exponents
    int nvt = 0, center = 0;
};
__global__ void __launch_bounds__(256) k_dg_tab_max(const zd* __restrict__ tab, int n, int* hw) {
    int m = 0;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) m = max(m, max(dg_hw(tab[i].x), dg_hw(tab[i].y)));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(hw, m);
}
__global__ void __launch_bounds__(256) k_dg_tab_cut(const zd* __restrict__ tab, int n, const int* hw, int* eo, uint4* t4, uint2* t2) {
    const int i = blockIdx.x * 256 + threadIdx.x, e = dg_exp(*hw);
    if (i == 0) *eo = e;
    if (i >= n) return;
    const DgScale sc = dg_scale(e >= 2048 ? 0 : e);
    uint32_t dr[DG_P], di[DG_P], p[DG_P];
    dg_cut<DG_P>(e >= 2048 ? 0 : dg_int(tab[i].x, sc), dr);
    dg_cut<DG_P>(e >= 2048 ? 0 : dg_int(tab[i].y, sc), di);
#pragma unroll
    for (int q = 0; q < DG_P; ++q) p[q] = dg_pair(dr[q], di[q]);
    t4[i] = make_uint4(p[0], p[1], p[2], p[3]);
    t2[i] = make_uint2(p[4], p[5]);
}

void dg_toep_destroy(DgToep* t) {
    if (!t) return;
    dg_gemm_destroy(t->g);
    t->pool.drop();
    delete t;
}

// T = V~ * C_G per k-point (r: C_G and T).  x: a product with the same right
// operands, whose digits are then taken, or null.
DgToep* dg_toep_create(int nk, const DgRight* r, const int* const* glin, int ncol, const DgGemm* x, int nvt, int center, int* flag) {
    DgToep* t = new DgToep();
    if (x && x->NT > 32) x = nullptr;
    t->nvt = nvt;
    t->center = center;
    t->own = !x;
    for (int q = 0; q < 2; ++q) {
        t->tab4[q] = (uint4*)t->pool.get((size_t)nvt * sizeof(uint4), false);
        t->tab2[q] = (uint2*)t->pool.get((size_t)nvt * sizeof(uint2), false);
    }
    t->hw = (int*)t->pool.get(2 * sizeof(int), true);
    t->e = (int*)t->pool.get(2 * sizeof(int), true);
    DgLeft l;  // shapes only
    l.src.resize(nk);
    for (int k = 0; k < nk; ++k) {
        l.src[k] = DgSrc{};
        l.src[k].M = l.src[k].K = r[k].K;
        l.src[k].nst = dg_nst(r[k].K);
    }
    if (t->pool.ok) t->g = dg_gemm_build(&l, nk, r, ncol, flag, 0, x, glin);
    if (!t->g || dg_attr<0, true>(t->g->NT) != cudaSuccess) {
        dg_toep_destroy(t);
        return nullptr;
    }
    return t;
}

// cut a table; which: 0 V~, 1 the step's
int launch_dg_table(const DgToep* t, int which, const zd* tab, cudaStream_t s) {
    cudaMemsetAsync(t->hw + which, 0, sizeof(int), s);
    k_dg_tab_max<<<std::min(304, (t->nvt + 255) / 256), 256, 0, s>>>(tab, t->nvt, t->hw + which);
    k_dg_tab_cut<<<(t->nvt + 255) / 256, 256, 0, s>>>(tab, t->nvt, t->hw + which, t->e + which, t->tab4[which], t->tab2[which]);
    return 2;
}
int launch_dg_toep(const DgToep* t, int which, int kofs, int nk, cudaStream_t s) {
    const DgGemm* g = t->g;
    if (t->own) k_dg_pack_b<<<dim3(8 * g->ncol, 1, nk), DG_PB_T, 0, s>>>(g->pb, kofs);
    DgArgs a = dg_args(g, kofs, 0);
    a.tab4 = t->tab4[which];
    a.tab2 = t->tab2[which];
    a.tabe = t->e + which;
    a.center = t->center;
    dg_launch<0, true>(g->NT, g->mt, nk, a, s);
    return t->own ? 2 : 1;
}

// ------------------------------------------------------------ Chebyshev series
// The series with H~ y_{n-1} as digit products, one launch per term, for more
// states or rows than k_cheb_coop takes.  In FP64 its rate was the FP64 pipe's (16
// k-points of N_aux 300, N_s 60: 9.0 GFLOP in 8.3 ms; 2 k-points 1.91 ms); here the
// 2 k-points take 0.28 ms, bound by the 14 launches of a few stages each.
// H~ = (HH - lam_c) / lam_h is its diagonal, which multiplies y in FP64, and the
// rest as digits, a power of two above the largest entry for each row; a column of
// y takes the power of two above theta's 2-norm, which bounds every y_n (H~ has
// norm <= 1).  The recurrence and the sum are FP64.  Seven digits, 63 bits: the cut
// is 2^-63 of what couples an amplitude to the others, and an amplitude that a weak
// field feeds keeps FP64's relative accuracy, also where a state couples to others a
// hundred times more strongly than to the occupied ones (with the diagonal among the
// digits and y_n in integers it kept 2^-54 of the column's norm, 1e-8 of the excited
// amplitudes at A = 1e-4; with six digits 2.5e-15 where FP64 has 0.8e-15).
struct DgSeriesK {
    uint32_t* A;     // digits of H~ off its diagonal, tiles of 128 rows
    int nst, NT;
    int* er;         // their row exponents
    double* diag;
    int* bad;        // per row: HH not finite
    int* ec;         // column exponents of y; 2048: theta not finite
};
struct DgSeries {
    DgPool pool;
    int nk = 0, n = 0, ns = 0, NT = 0, ntn = 0, mt = 0, cs = 1, gs = 1;
    DgOut* out = nullptr;
    DgCheb* ch = nullptr;
    DgSeriesK* sk = nullptr;
    i64* part = nullptr;
    unsigned* cnt = nullptr;
};

// digits of row i of H~ off its diagonal (HH as in k_hsub; HH is Hermitian, so
// row i is read as the conjugate of the contiguous column i).  A thread holds
// its first DG_HS_E entries from the search for the largest one to the cut.
#define DG_HS_E 4
__global__ void __launch_bounds__(128) k_dg_hsub(StepArgs a, const DgSeriesK* sk) {
    __shared__ int smx[4];
    const DgSeriesK& S = sk[blockIdx.z];
    const KDev& K = a.kd[blockIdx.z];
    const int n = a.naux, i = blockIdx.x;
    DevState* st = a.st;
    const double* av = a.a + 3 * (size_t)st->cstep;
    const double ax = av[0], ay = av[1], az = av[2];
    const double aa = (ax * ax + ay * ay + az * az) * a.half_inv_c2;
    if (i == 0 && blockIdx.z == 0 && threadIdx.x == 0) {
        if (!a.dv_on) {
            st->cur_a[0] = ax;
            st->cur_a[1] = ay;
            st->cur_a[2] = az;
            st->cur_s = 0.0;
            st->cur_aa = aa;
        }
    }
    const double lc = K.lam[0], ilh = K.lam[2];
    const double al[3] = {ax * a.inv_c, ay * a.inv_c, az * a.inv_c};
    const size_t nn = (size_t)n * n;
    auto entry = [&](int j) {
        const size_t e = (size_t)i * n + j;
        zd v = zmk(0.0, 0.0);
#pragma unroll
        for (int l = 0; l < 3; ++l)
            if (al[l] != 0.0) v = zadd(v, zscale(K.psub[l * nn + e], al[l]));
        if (i == j) v.x += K.eps[i] + aa;
        if (a.dv_on) v = zadd(v, K.dvsub[e]);
        if (i == j) v.x -= lc;
        return zscale(v, ilh);
    };
    int bad = 0, hm = 0;
    auto look = [&](int j, zd& v) {  // the diagonal entry's real part goes to S.diag
        const int hx = dg_hw(v.x), hy = dg_hw(v.y);
        if (hx >= 0x7ff00000 || hy >= 0x7ff00000) bad = 1;
        if (j == i) {
            S.diag[i] = v.x;
            v.x = 0.0;
            hm = max(hm, hy);
        } else {
            hm = max(hm, max(hx, hy));
        }
    };
    zd h[DG_HS_E];
#pragma unroll
    for (int u = 0; u < DG_HS_E; ++u) {
        const int j = threadIdx.x + u * 128;
        if (j >= n) continue;
        h[u] = entry(j);
        look(j, h[u]);
    }
    for (int j = threadIdx.x + DG_HS_E * 128; j < n; j += 128) {
        zd v = entry(j);
        look(j, v);
    }
    hm = __reduce_max_sync(0xffffffffu, hm);
    if ((threadIdx.x & 31) == 0) smx[threadIdx.x >> 5] = hm;
    bad = __syncthreads_or(bad);
    const int e = bad ? 0 : dg_exp(max(max(smx[0], smx[1]), max(smx[2], smx[3])));
    if (threadIdx.x == 0) {
        S.bad[i] = bad;
        S.er[i] = e;
    }
    auto put = [&](int j, zd v) {
        uint32_t dr[DG_PS], di[DG_PS];
        dg_cut<DG_PS>(fix64(v.x, e, 9 * DG_PS - 1), dr);
        dg_cut<DG_PS>(-fix64(v.y, e, 9 * DG_PS - 1), di);
#pragma unroll
        for (int q = 0; q < DG_PS; ++q)
            S.A[dg_word<DG_PS>(i, j, DG_BM, S.nst) + (size_t)q * DG_BM * 16] = dg_pair(dr[q], di[q]);
    };
#pragma unroll
    for (int u = 0; u < DG_HS_E; ++u) {
        const int j = threadIdx.x + u * 128;
        if (j < n) put(j, h[u]);
    }
    for (int j = threadIdx.x + DG_HS_E * 128; j < n; j += 128) {
        zd v = entry(j);
        if (j == i) v.x = 0.0;
        put(j, v);
    }
}

// y_0 = theta, its digits, and c_0 y_0
__global__ void __launch_bounds__(128) k_dg_y0(StepArgs a, const DgSeriesK* sk, const DgCheb* chs) {
    __shared__ double sh[4];
    const DgSeriesK& S = sk[blockIdx.z];
    const DgCheb& ch = chs[blockIdx.z];
    const KDev& K = a.kd[blockIdx.z];
    const int n = a.naux, c = blockIdx.x, tid = threadIdx.x;
    const zd* th = K.theta + (size_t)c * n;
    // the norm of theta / 2^e with e from its largest entry: no overflow in the squares
    int mx = 0;
    for (int i = tid; i < n; i += 128) mx = max(mx, max(dg_hw(th[i].x), dg_hw(th[i].y)));
    mx = __reduce_max_sync(0xffffffffu, mx);
    __shared__ int smx[4];
    if ((tid & 31) == 0) smx[tid >> 5] = mx;
    __syncthreads();
    mx = max(max(smx[0], smx[1]), max(smx[2], smx[3]));
    int e = dg_exp(mx);
    const bool bad = e >= 2048;
    if (bad) e = 0;
    const DgScale s0 = dg_scale(e);
    double q = 0.0;
    for (int i = tid; i < n; i += 128) {
        const double x = (th[i].x * s0.p1) * s0.p2, y = (th[i].y * s0.p1) * s0.p2;  // 2^53 at most
        q += x * x + y * y;
    }
    q = warp_sum(q);
    if ((tid & 31) == 0) sh[tid >> 5] = q;
    __syncthreads();
    q = sqrt(sh[0] + sh[1] + sh[2] + sh[3]);
    // the power of two above the norm, with room for the rounding of the terms
    const int en = q > 0.0 ? dg_exp(dg_hw(q * (1.0 + 1e-9))) : 53;
    e += en - 53;
    if (tid == 0) S.ec[c] = bad ? 2048 : e;
    const zd c0 = K.coef[0];
    for (int i = tid; i < n; i += 128) {
        const zd y = bad ? zmk(0.0, 0.0) : th[i];
        const size_t x = (size_t)c * n + i;
        ch.y0[x] = y;
        ch.acc[x] = zmul(c0, y);
        dg_put_col<DG_PS>(ch.Bn[0], S.NT, ch.nst, c, i, fix64(y.x, e, 9 * DG_PS - 1), fix64(y.y, e, 9 * DG_PS - 1));
    }
}

// theta = phase x sum; a k-point whose HH is not finite gives NaN
__global__ void __launch_bounds__(128) k_dg_theta(StepArgs a, const DgSeriesK* sk, const DgCheb* chs) {
    const DgSeriesK& S = sk[blockIdx.z];
    const DgCheb& ch = chs[blockIdx.z];
    const KDev& K = a.kd[blockIdx.z];
    const int n = a.naux, c = blockIdx.x, tid = threadIdx.x;
    int bad = S.ec[c] >= 2048;
    for (int i = tid; i < n; i += 128) bad |= S.bad[i];
    bad = __syncthreads_or(bad);
    const zd ph = (a.prop == 0) ? zmk(K.lam[3], K.lam[4]) : zmk(1.0, 0.0);
    for (int i = tid; i < n; i += 128) {
        zd v = zmul(ph, ch.acc[(size_t)c * n + i]);
        if (bad) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
        K.theta[i + (size_t)c * n] = v;
    }
}

void dg_series_destroy(DgSeries* g) {
    if (!g) return;
    g->pool.drop();
    delete g;
}

DgSeries* dg_series_create(int nk, int n, int ns, const zd* const* coef) {
    DgSeries* g = new DgSeries();
    g->nk = nk;
    g->n = n;
    g->ns = ns;
    g->NT = dg_nt(ns);
    g->ntn = (2 * ns + g->NT - 1) / g->NT;
    g->mt = (n + DG_BM - 1) / DG_BM;
    const int np = g->ntn * g->NT, nst = dg_nst(n);
    std::vector<DgOut> out(nk);
    std::vector<DgCheb> ch(nk);
    std::vector<DgSeriesK> sk(nk);
    for (int k = 0; k < nk; ++k) {
        sk[k].A = (uint32_t*)g->pool.get(dg_bytes(g->mt * DG_BM, n, DG_PS), true);
        sk[k].nst = nst;
        sk[k].NT = g->NT;
        sk[k].bad = (int*)g->pool.get(n * sizeof(int), true);
        sk[k].ec = (int*)g->pool.get(ns * sizeof(int), true);
        DgCheb& c = ch[k];
        c.n = n;
        sk[k].er = (int*)g->pool.get(n * sizeof(int), true);
        sk[k].diag = (double*)g->pool.get(n * sizeof(double), true);
        c.y0 = (zd*)g->pool.get((size_t)ns * n * sizeof(zd), true);
        c.y1 = (zd*)g->pool.get((size_t)ns * n * sizeof(zd), true);
        c.acc = (zd*)g->pool.get((size_t)ns * n * sizeof(zd), true);
        c.diag = sk[k].diag;
        for (int q = 0; q < 2; ++q) c.Bn[q] = (uint32_t*)g->pool.get(dg_bytes(np, n, DG_PS), true);
        c.nst = nst;
        c.coef = coef[k];
        out[k] = DgOut{};
        out[k].A = (const unsigned char*)sk[k].A;
        out[k].er = sk[k].er;
        out[k].ec = sk[k].ec;
        out[k].M = n;
        out[k].nst = out[k].nsta = nst;
        out[k].tile0 = k * g->mt * g->ntn;
    }
    const int tiles = nk * g->mt * g->ntn;
    dg_splits(tiles, nst, &g->cs, &g->gs);
    if (g->gs > 1) {
        g->part = (i64*)g->pool.get((size_t)tiles * g->NT * 2 * DG_BM * sizeof(i64), true);
        g->cnt = (unsigned*)g->pool.get((size_t)tiles * g->cs * sizeof(unsigned), true);
    }
    if (g->pool.ok) {
        g->out = g->pool.up(out);
        g->ch = g->pool.up(ch);
        g->sk = g->pool.up(sk);
    }
    if (!g->pool.ok || dg_attr<1, false>(g->NT) != cudaSuccess) {
        dg_series_destroy(g);
        return nullptr;
    }
    return g;
}

int launch_dg_series(const DgSeries* g, const StepArgs& a, cudaStream_t s) {
    k_dg_hsub<<<dim3(g->n, 1, g->nk), 128, 0, s>>>(a, g->sk);
    k_dg_y0<<<dim3(g->ns, 1, g->nk), 128, 0, s>>>(a, g->sk, g->ch);
    DgArgs d{};
    d.out = g->out;
    d.ch = g->ch;
    d.ncol = g->ns;
    d.ntn = g->ntn;
    d.cs = g->cs;
    d.gs = g->gs;
    d.part = g->part;
    d.cnt = g->cnt;
    d.flag = a.flag;
    for (int t = 1; t < a.nterms; ++t) {
        d.term = t;
        d.last = t == a.nterms - 1;
        dg_launch<1, false>(g->NT, g->mt, g->nk, d, s);
    }
    k_dg_theta<<<dim3(g->ns, 1, g->nk), 128, 0, s>>>(a, g->sk, g->ch);
    return a.nterms + 2;
}
