// Interstitial convolution of Eq. v_interstitial by fast Fourier transforms:
// the route that the paper recommends for large plane-wave cut-offs (Sec. 3,
// the cost of the interstitial term, and the FFT against matrix-product
// comparison).
//
//   Y_G = sum_G' V~_{G-G'} C_G'     for G in the plane-wave set of a k-point
//
// The G - G' differences of one k-point lie in the table box |d_i| <= e_i,
// so on a periodic grid of F_i >= 2 e_i + 1 points per axis every difference
// has its own residue (d_i mod F_i).  With V~ placed on the grid by residue,
// v(r_j) = F^-3 sum_d V~_d e^{+2 pi i d.j/F} (set-up), the circular
// convolution equals the sum above:
//   c(r_j) = sum_G' C_G' e^{+2 pi i G'.j/F}                (inverse transform)
//   Y_G    = sum_j e^{-2 pi i G.j/F} v(r_j) c(r_j)          (forward transform)
// Both transforms are pruned to the G set: C is non-zero on the lines
// (n1, n2) and planes n1 that hold a G vector, and Y is needed only there.
// Five passes per product, each a batch of 1-D transforms in shared memory
// (Stockham autosort, radices 2, 3, 4, 5):
//   A  inverse along axis 3, lines holding a G        (scatter C_G)
//   B  inverse along axis 2, planes holding a G
//   C  along axis 1 on every (r2, r3): inverse, times v(r), forward
//   D  forward along axis 2, kept on the lines holding a G
//   E  forward along axis 3                           (gather Y_G)
// All k-points and columns of a product run in the same five launches.
#include "rtd.h"
#include "rttddft.h"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <string>
#include <vector>

#define FFT_LPB 16        // lines per block at most
#define FFT_BLK_PTS 2048  // points of a line block at most: lines per block = min(16, 2048 / L)
#define FFT_THREADS 128
#define FFT_PV (FFT_BLK_PTS / FFT_THREADS)  // points of a block per thread
#define FFT_PTHREADS 256  // plane kernels
#define FFT_MAX_N 512     // longest axis
#define FFT_MAX_ST 8

// lines of length L per block of a line pass
static inline int fft_lpb(int L) { return std::min(FFT_LPB, FFT_BLK_PTS / std::max(L, 1)); }

struct FftK {
    int nline, nplane;
    const int* lg0;       // [nline + 1] first entry of each line in line order
    const int* gperm;     // [ng] G index of each entry in line order
    const int* lpos;      // [ng] line * F3 + residue of n3, per entry
    const int* plane_of;  // [F1] plane of a residue of n1, or -1
    const int* line_of;   // [nplane][F2] line of (plane, residue of n2), or -1
    const int* pl0;       // [nplane + 1] first line of each plane
    const int* lr2;       // [nline] residue of n2 of each line
};

struct FftArgs {
    int F1, F2, F3;
    int nst[3];
    int rad[3][FFT_MAX_ST];
    unsigned mg[3][2 * FFT_MAX_ST];  // per stage: multipliers that divide by its butterflies per line and its stride
    int lpb[3];             // lines per block of the passes along each axis
    const void* w[3];       // twiddles e^{-2 pi i m / F_a}, m < F_a (FP64 or FP32 complex)
    const FftK* fk;         // per k-point of the launch
    const ToepDesc* td;     // per k-point: source X (ld ldx) and destination Y (ld ldy)
    void* b3;               // [k][col][max_lines][F3]
    void* b2;               // [k][col][max_planes][F2][F3]
    size_t b3_col, b2_col;  // elements per column
    int ncol;
    int vmode;              // 0: v (+ s vd when use_vd), 1: s vd alone
    int use_vd;
    const void* v;          // potential on the grid (complex, FP64 or FP32)
    const void* vd;
    const double* s;        // scale of vd (device)
    // fixed-point form: the potential's image and its exponents per (r2, chunk
    // of axis 1's blocks); exponents of the stored values per (line, chunk),
    // (plane, chunk) and (r2, chunk) of each column
    const struct tq* vq;
    const int* vqe;
    int2 *ma, *mb, *mc;
    int lines_max, planes_max;
    int qb[3];              // bits that an axis' transform may start with
    int tune;               // 1: transform zeros like values (the set-up's timing runs on zeros)
};

struct FftPlan {
    int F[3];
    int nst[3];
    int rad[3][FFT_MAX_ST];
    int prec;  // 0 FP64, 1 FP32
    int nk;
    int max_lines, max_planes;
    int ncol;
    int fused = 0;  // 1: axes 3 and 2 of a plane in one launch (three launches per product)
    float ms_split = 0.f, ms_fused = 0.f;  // set-up timings of both launch sets
    zd* w64[3] = {nullptr, nullptr, nullptr};
    zf* w32[3] = {nullptr, nullptr, nullptr};
    zd* v64 = nullptr;
    zf* v32 = nullptr;
    zd* vd64 = nullptr;
    zf* vd32 = nullptr;
    FftK* d_fk = nullptr;
    void* b3 = nullptr;
    void* b2 = nullptr;
    // fixed-point form (FP64 plans, axes of at most FX_MAX_N points): twiddles,
    // images of v and of a call's v + s vd with their exponents, exponents of b3 and b2
    int fx = 0;
    struct tq* wq[3] = {nullptr, nullptr, nullptr};
    struct tq* vq[2] = {nullptr, nullptr};
    int* vqe[2] = {nullptr, nullptr};
    int2 *ma = nullptr, *mb = nullptr, *mc = nullptr;
    std::vector<void*> tables;  // per-k index arrays
    // Hartree feedback: density grid (forward transformed), its value at the
    // start, the box extents, the reciprocal vectors, the l1 accumulator
    // (the density and its potential are FP64 in every form: the change n(t) - n(0)
    // is a small difference of two densities, which FP32 rounding would swamp)
    zd* rho = nullptr;
    zd* rho0 = nullptr;
    zd* b3d = nullptr;  // FP64 transform buffers of the density (FP32 plans only)
    zd* b2d = nullptr;
    int fused_d = 0;    // the density's plane pass fused (FP64 plane in shared memory)
    double* l1 = nullptr;
    int hartree = 0;
    int e[3] = {0, 0, 0};
    double recip[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    double omega = 1.0, bound = 0.0;
};

// ---------------------------------------------------------------- complex ops
template <typename C> struct Rt;
template <> struct Rt<zd> { typedef double R; };
template <> struct Rt<zf> { typedef float R; };
template <typename C> __device__ __forceinline__ C cmk(typename Rt<C>::R x, typename Rt<C>::R y) {
    C r;
    r.x = x;
    r.y = y;
    return r;
}
template <typename C> __device__ __forceinline__ C cad(C a, C b) { return cmk<C>(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csb(C a, C b) { return cmk<C>(a.x - b.x, a.y - b.y); }
template <typename C> __device__ __forceinline__ C cml(C a, C b) {
    return cmk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// i * z * sgn
template <typename C> __device__ __forceinline__ C cis(C z, typename Rt<C>::R sg) { return cmk<C>(-sg * z.y, sg * z.x); }
template <typename C> __device__ __forceinline__ C cwt(const C* W, int i, bool inv) {
    C w = W[i];
    if (inv) w.y = -w.y;
    return w;
}
// a +- i b by the direction's sign; a + w b, i w z, i (w1 d1 + w2 d2) for real w
template <typename C> __device__ __forceinline__ C cisg(C z, bool inv) {
    return inv ? cmk<C>(-z.y, z.x) : cmk<C>(z.y, -z.x);
}
template <typename C> __device__ __forceinline__ C cma(C a, typename Rt<C>::R w, C b) {
    return cmk<C>(a.x + w * b.x, a.y + w * b.y);
}
template <typename C> __device__ __forceinline__ C cma2(C a, typename Rt<C>::R w, C b, typename Rt<C>::R v, C d) {
    return cma(cma(a, w, b), v, d);
}
template <typename C> __device__ __forceinline__ C ci2(typename Rt<C>::R w1, C d1, typename Rt<C>::R w2, C d2) {
    return cmk<C>(-(w1 * d1.y + w2 * d2.y), w1 * d1.x + w2 * d2.x);
}

// Fixed point: 64-bit integers, complex values below 2^62 in modulus (so the middle
// sums of a product stay below 2 sqrt(2) 2^61), a power-of-two scale per block,
// factors (twiddles, potential) with 62 binary places.  A product keeps the three
// largest of its four 32-bit partial products; the low words are signed
// (balanced), so what is dropped averages to zero and stays below one unit.
// Factors are stored split; their low word is never -2^31, so that it can change
// its sign.
struct __align__(16) zq {
    long long x, y;
};
struct rq {
    int h, l;
};
struct __align__(16) tq {
    rq x, y;
};
template <> struct Rt<zq> { typedef long long R; };
__host__ __device__ __forceinline__ rq qsplit(long long w) {
    rq r;
    r.l = (int)w;
    if (r.l == (int)0x80000000) r.l += 1, w += 1;
    r.h = (int)((w - r.l) >> 32);
    return r;
}
__device__ __forceinline__ rq qneg(rq w) {
    w.h = -w.h;
    w.l = -w.l;
    return w;
}
__device__ __forceinline__ int qhi(long long a) { return (int)((a + 0x80000000LL) >> 32); }
// a w and a w + b v
__device__ __forceinline__ long long qml(long long a, rq w) {
    const int ah = qhi(a), al = (int)a;
    return (((long long)ah * w.h) << 2) + ((((long long)ah * w.l + (1LL << 29)) + (long long)al * w.h) >> 30);
}
__device__ __forceinline__ long long qml2(long long a, rq w, long long b, rq v) {
    const int ah = qhi(a), al = (int)a, bh = qhi(b), bl = (int)b;
    const long long h = (long long)ah * w.h + (long long)bh * v.h;
    const long long m =
        ((((long long)ah * w.l + (1LL << 29)) + (long long)al * w.h) + (long long)bh * v.l) + (long long)bl * v.h;
    return (h << 2) + (m >> 30);
}
__device__ __forceinline__ zq cml(zq a, tq w) {
    return cmk<zq>(qml2(a.x, w.x, a.y, qneg(w.y)), qml2(a.x, w.y, a.y, w.x));
}
__device__ __forceinline__ zq cis(zq z, rq w) { return cmk<zq>(qml(z.y, qneg(w)), qml(z.x, w)); }
__device__ __forceinline__ zq cma(zq a, rq w, zq b) { return cmk<zq>(a.x + qml(b.x, w), a.y + qml(b.y, w)); }
__device__ __forceinline__ zq cma2(zq a, rq w, zq b, rq v, zq d) {
    return cmk<zq>(a.x + qml2(b.x, w, d.x, v), a.y + qml2(b.y, w, d.y, v));
}
__device__ __forceinline__ zq ci2(rq w1, zq d1, rq w2, zq d2) {
    return cmk<zq>(qml2(d1.y, qneg(w1), d2.y, qneg(w2)), qml2(d1.x, w1, d2.x, w2));
}
// the table's entries and their parts
template <typename C> struct Tw { typedef C T; };
template <> struct Tw<zq> { typedef tq T; };
__device__ __forceinline__ tq cwt(const tq* W, int i, bool inv) {
    tq w = W[i];
    if (inv) w.y = qneg(w.y);
    return w;
}
__device__ __forceinline__ double rneg(double w) { return -w; }
__device__ __forceinline__ float rneg(float w) { return -w; }
__device__ __forceinline__ rq rneg(rq w) { return qneg(w); }
__device__ __forceinline__ zd cvt(zd a, zd) { return a; }
__device__ __forceinline__ zf cvt(zd a, zf) { return tof(a); }
__device__ __forceinline__ zd todz(zd a) { return a; }
__device__ __forceinline__ zd todz(zf a) { return tod(a); }

// floor(n / d) for n d < 2^32 by the multiplier ceil(2^32 / d) (0: d = 1)
__host__ __device__ __forceinline__ unsigned fft_magic(int d) { return d == 1 ? 0u : 0xffffffffu / (unsigned)d + 1u; }
__device__ __forceinline__ int fft_div(int n, unsigned mg) { return mg ? (int)__umulhi((unsigned)n, mg) : n; }

// Stockham autosort, decimation in frequency: nl lines of length L stored
// line by line in x (y is scratch of the same size).  A stage of radix R on
// sub-transforms of length n = L/s (s interleaved sequences) maps
//   x[q + s(p + r m)]  ->  y[q + s(R p + t)] = w_n^{p t} sum_r x[q + s(p + r m)] w_R^{r t},
// m = n/R, p < m, q < s; after the last stage the transform is in natural
// order.  inv selects e^{+}.  Element j of line l sits at l ls + j es (in x and
// y alike).  Returns the buffer holding the result.
// LF: neighbouring threads take the same butterfly of neighbouring lines (lines
// stored side by side, ls = 1: no bank conflicts); otherwise neighbouring
// butterflies of a line.  Indices are divided by multiplication (mg, fft_div) and
// the last stage, whose twiddles are all 1, multiplies by none: an integer
// division costs as much as a radix-4 butterfly in FP32, a twiddle four of the
// slow FP64 instructions.
// A transform of R values in registers, in natural order; W is the table of L
// entries.  (Radices 6, 8, 9 and 10 as two steps in registers measured slower,
// 2225 against 1367 us at 200 columns on 48^3 points in fixed point, 737 against
// 676 us at 240 columns in FP32: a block has half the butterflies, fewer than it
// has threads, and the registers halve the blocks per SM.)
template <int R, typename C>
__device__ __forceinline__ void fft_bfly(C* a, const typename Tw<C>::T* W, int L, bool inv) {
    if constexpr (R == 2) {
        const C t = a[0];
        a[0] = cad(t, a[1]);
        a[1] = csb(t, a[1]);
    } else if constexpr (R == 4) {
        const C s02 = cad(a[0], a[2]), d02 = csb(a[0], a[2]), s13 = cad(a[1], a[3]), d13 = csb(a[1], a[3]);
        // w_4 = -i (forward): b1 = d02 - i d13, b3 = d02 + i d13
        const C id13 = cisg(d13, inv);
        a[0] = cad(s02, s13);
        a[1] = cad(d02, id13);
        a[2] = csb(s02, s13);
        a[3] = csb(d02, id13);
    } else if constexpr (R == 3) {
        const auto w = cwt(W, L / 3, inv);  // w_3
        const C sm = cad(a[1], a[2]), df = csb(a[1], a[2]);
        const C t = cma(a[0], w.x, sm);
        const C u = cis(df, w.y);  // i Im(w_3) (a1 - a2)
        a[0] = cad(a[0], sm);
        a[1] = cad(t, u);
        a[2] = csb(t, u);
    } else {
        const auto w1 = cwt(W, L / 5, inv), w2 = cwt(W, 2 * (L / 5), inv);  // w_5, w_5^2
        const C s1 = cad(a[1], a[4]), d1 = csb(a[1], a[4]), s2 = cad(a[2], a[3]), d2 = csb(a[2], a[3]);
        const C ta = cma2(a[0], w1.x, s1, w2.x, s2);
        const C tb = cma2(a[0], w2.x, s1, w1.x, s2);
        // i (Im w1 d1 + Im w2 d2) and i (Im w2 d1 - Im w1 d2)
        const C ua = ci2(w1.y, d1, w2.y, d2);
        const C ub = ci2(w2.y, d1, rneg(w1.y), d2);
        a[0] = cad(a[0], cad(s1, s2));
        a[1] = cad(ta, ua);
        a[2] = cad(tb, ub);
        a[3] = csb(tb, ub);
        a[4] = csb(ta, ua);
    }
}

template <int R, bool LF, bool LAST, typename C>
__device__ __forceinline__ void fft_stage_r(const C* x, C* y, int m, int s0, unsigned mgl, unsigned mgs, int nl, int L,
                                            int ls, int es, const typename Tw<C>::T* W, bool inv) {
    const int nb = m * s0;  // butterflies per line
    const int tot = nl * nb;
    const int ms = nb * es, os = s0 * es;  // strides between the points of a butterfly: input, output
    for (int b = threadIdx.x; b < tot; b += blockDim.x) {
        const int o = fft_div(b, mgl);  // LF: the butterfly, else the line
        const int l = LF ? b - o * nl : o;
        const int bb = LF ? o : b - o * nb;
        const int p = fft_div(bb, mgs);
        const int q = bb - p * s0;
        const C* xi = x + l * ls + bb * es;
        C* yo = y + l * ls + (q + s0 * R * p) * es;
        C a[R];
#pragma unroll
        for (int t = 0; t < R; ++t) a[t] = xi[t * ms];
        fft_bfly<R>(a, W, L, inv);
        yo[0] = a[0];
        const int ps = p * s0;
#pragma unroll
        for (int t = 1; t < R; ++t) {
            if constexpr (LAST) yo[t * os] = a[t];
            else yo[t * os] = cml(a[t], cwt(W, t * ps, inv));
        }
    }
}

template <bool LF, bool LAST, typename C>
__device__ __forceinline__ void fft_stage(const C* x, C* y, int R, int m, int s0, unsigned mgl, unsigned mgs, int nl, int L,
                                          int ls, int es, const typename Tw<C>::T* W, bool inv) {
    switch (R) {
#define FFT_R(r) \
    case r: fft_stage_r<r, LF, LAST>(x, y, m, s0, mgl, mgs, nl, L, ls, es, W, inv); break;
        FFT_R(2) FFT_R(3) FFT_R(4) FFT_R(5)
#undef FFT_R
    }
}
template <bool LF, typename C>
__device__ C* fft_lines_s(C* x, C* y, int nl, int L, int ls, int es, const int* rad, const unsigned* mg, int nst,
                          const typename Tw<C>::T* W, bool inv) {
    int s0 = 1;
    const unsigned mnl = LF ? fft_magic(nl) : 0u;
    for (int st = 0; st < nst; ++st) {
        const int R = rad[st];
        const int m = L / (s0 * R);
        const unsigned mgl = LF ? mnl : mg[2 * st], mgs = mg[2 * st + 1];
        if (st + 1 < nst) fft_stage<LF, false>(x, y, R, m, s0, mgl, mgs, nl, L, ls, es, W, inv);
        else fft_stage<LF, true>(x, y, R, m, s0, mgl, mgs, nl, L, ls, es, W, inv);
        __syncthreads();
        C* t = x;
        x = y;
        y = t;
        s0 *= R;
    }
    return x;
}

template <typename C>
__device__ __forceinline__ C* fft_lines(C* x, C* y, int nl, int L, const FftArgs& f, int ax,
                                       const typename Tw<C>::T* W, bool inv) {
    return fft_lines_s<false>(x, y, nl, L, L, 1, f.rad[ax], f.mg[ax], f.nst[ax], W, inv);
}
// lines side by side: element j of line l at j nl + l
template <typename C>
__device__ __forceinline__ C* fft_cols(C* x, C* y, int nl, int L, const FftArgs& f, int ax,
                                       const typename Tw<C>::T* W, bool inv) {
    return fft_lines_s<true>(x, y, nl, L, 1, nl, f.rad[ax], f.mg[ax], f.nst[ax], W, inv);
}

template <typename C>
__device__ __forceinline__ void load_tw(C* W, const void* src, int L) {
    const C* w = (const C*)src;
    for (int i = threadIdx.x; i < L; i += blockDim.x) W[i] = w[i];
}

// A: scatter C_G onto the lines of axis 3 and transform them (inverse)
template <typename C>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_a(FftArgs f) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int F3 = f.F3, LPB = f.lpb[2];
    C* W = (C*)fsm;
    C* x = W + F3;
    C* y = x + LPB * F3;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int l0 = blockIdx.x * LPB;
    if (l0 >= K.nline) return;
    const int nl = min(LPB, K.nline - l0);
    load_tw(W, f.w[2], F3);
    for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) x[i] = cmk<C>(0, 0);
    __syncthreads();
    const ToepDesc td = f.td[k];
    const int j0 = K.lg0[l0], j1 = K.lg0[l0 + nl];
    const int base = l0 * F3;
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x)
        x[K.lpos[j] - base] = cvt(td.X[K.gperm[j] + (size_t)c * td.ldx], C());
    __syncthreads();
    const C* r = fft_lines(x, y, nl, F3, f, 2, W, true);
    C* out = (C*)f.b3 + ((size_t)k * f.ncol + c) * f.b3_col + (size_t)base;
    for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) out[i] = r[i];
}

// B (fwd = 0) and D (fwd = 1): axis 2 on the planes holding a G; a block
// takes lpb[1] consecutive r3 of one plane
template <typename C>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_bd(FftArgs f, int fwd) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int F2 = f.F2, F3 = f.F3, LPB = f.lpb[1];
    C* W = (C*)fsm;
    C* x = W + F2;
    C* y = x + LPB * F2;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int nch = (F3 + LPB - 1) / LPB;
    const int p = blockIdx.x / nch, i30 = (blockIdx.x - p * nch) * LPB;
    if (p >= K.nplane) return;
    const int nl = min(LPB, F3 - i30);
    load_tw(W, f.w[1], F2);
    C* b3 = (C*)f.b3 + ((size_t)k * f.ncol + c) * f.b3_col;
    C* b2 = (C*)f.b2 + ((size_t)k * f.ncol + c) * f.b2_col + (size_t)p * F2 * F3;
    const int* lo = K.line_of + (size_t)p * F2;
    const unsigned mnl = fft_magic(nl);
    for (int i = threadIdx.x; i < F2 * nl; i += blockDim.x) {
        const int r2 = fft_div(i, mnl), l = i - r2 * nl;
        C v = cmk<C>(0, 0);
        if (fwd) {
            v = b2[(size_t)r2 * F3 + i30 + l];
        } else {
            const int id = lo[r2];
            if (id >= 0) v = b3[(size_t)id * F3 + i30 + l];
        }
        x[i] = v;
    }
    __syncthreads();
    const C* r = fft_cols(x, y, nl, F2, f, 1, W, !fwd);
    for (int i = threadIdx.x; i < F2 * nl; i += blockDim.x) {
        const int r2 = fft_div(i, mnl), l = i - r2 * nl;
        if (fwd) {
            const int id = lo[r2];
            if (id >= 0) b3[(size_t)id * F3 + i30 + l] = r[i];
        } else {
            b2[(size_t)r2 * F3 + i30 + l] = r[i];
        }
    }
}

// C: axis 1 on every (r2, r3): inverse, times the potential, forward; the
// result is kept on the planes holding a G
template <typename C>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_c(FftArgs f) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int F1 = f.F1, F2 = f.F2, F3 = f.F3, LPB = f.lpb[0];
    C* W = (C*)fsm;
    C* x = W + F1;
    C* y = x + LPB * F1;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int nch = (F3 + LPB - 1) / LPB;
    const int r2 = blockIdx.x / nch, i30 = (blockIdx.x - r2 * nch) * LPB;
    const int nl = min(LPB, F3 - i30);
    load_tw(W, f.w[0], F1);
    C* b2 = (C*)f.b2 + ((size_t)k * f.ncol + c) * f.b2_col;
    const size_t pst = (size_t)F2 * F3;
    const unsigned mnl = fft_magic(nl);
    const size_t off = (size_t)r2 * F3 + i30;
    for (int i = threadIdx.x; i < F1 * nl; i += blockDim.x) {
        const int r1 = fft_div(i, mnl), l = i - r1 * nl;
        const int p = K.plane_of[r1];
        x[i] = (p >= 0) ? b2[(size_t)p * pst + off + l] : cmk<C>(0, 0);
    }
    // the potential of this block's points, loaded (coalesced along r3) before
    // the inverse transform so that the loads overlap it
    constexpr int PV = FFT_PV;  // F1 nl <= FFT_BLK_PTS
    C pv[PV];
    {
        const C* v = (const C*)f.v;
        const C* vd = (const C*)f.vd;
        typedef typename Rt<C>::R R_;
        const R_ sc = f.use_vd ? (R_)(*f.s) : R_(0);
#pragma unroll
        for (int u = 0; u < PV; ++u) {
            const int i = threadIdx.x + u * FFT_THREADS;
            pv[u] = cmk<C>(0, 0);
            if (i < F1 * nl) {
                const int r1 = fft_div(i, mnl), l = i - r1 * nl;
                const size_t gi = (size_t)r1 * pst + off + l;
                if (f.vmode == 0) {
                    pv[u] = v[gi];
                    if (f.use_vd) {
                        const C d = vd[gi];
                        pv[u] = cmk<C>(pv[u].x + sc * d.x, pv[u].y + sc * d.y);
                    }
                } else {
                    const C d = vd[gi];
                    pv[u] = cmk<C>(sc * d.x, sc * d.y);
                }
            }
        }
    }
    __syncthreads();
    C* r = fft_cols(x, y, nl, F1, f, 0, W, true);
#pragma unroll
    for (int u = 0; u < PV; ++u) {
        const int i = threadIdx.x + u * FFT_THREADS;
        if (i < F1 * nl) {
            r[i] = cml(r[i], pv[u]);
        }
    }
    __syncthreads();
    const C* o = fft_cols(r, r == x ? y : x, nl, F1, f, 0, W, false);
    for (int i = threadIdx.x; i < F1 * nl; i += blockDim.x) {
        const int r1 = fft_div(i, mnl), l = i - r1 * nl;
        const int p = K.plane_of[r1];
        if (p >= 0) b2[(size_t)p * pst + off + l] = o[i];
    }
}

// E: transform the lines of axis 3 (forward) and gather Y_G
template <typename C>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_e(FftArgs f) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int F3 = f.F3, LPB = f.lpb[2];
    C* W = (C*)fsm;
    C* x = W + F3;
    C* y = x + LPB * F3;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int l0 = blockIdx.x * LPB;
    if (l0 >= K.nline) return;
    const int nl = min(LPB, K.nline - l0);
    load_tw(W, f.w[2], F3);
    const int base = l0 * F3;
    const C* in = (const C*)f.b3 + ((size_t)k * f.ncol + c) * f.b3_col + (size_t)base;
    for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) x[i] = in[i];
    __syncthreads();
    const C* r = fft_lines(x, y, nl, F3, f, 2, W, false);
    const ToepDesc td = f.td[k];
    const int j0 = K.lg0[l0], j1 = K.lg0[l0 + nl];
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x)
        td.Y[K.gperm[j] + (size_t)c * td.ldy] = todz(r[K.lpos[j] - base]);
}

// A+B (fwd = 0) and D+E (fwd = 1) for one plane holding a G: the plane's
// lines (compacted) along axis 3 and its F3 columns along axis 2, with the
// whole plane in shared memory
template <typename C>
__global__ void __launch_bounds__(FFT_PTHREADS) k_fft_plane(FftArgs f, int fwd) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int F2 = f.F2, F3 = f.F3, n2 = F2 * F3;
    C* W2 = (C*)fsm;
    C* W3 = W2 + F2;
    C* A = W3 + F3;
    C* B = A + n2;
    const int k = blockIdx.z, c = blockIdx.y, p = blockIdx.x;
    const FftK K = f.fk[k];
    if (p >= K.nplane) return;
    load_tw(W2, f.w[1], F2);
    load_tw(W3, f.w[2], F3);
    const unsigned m3 = fft_magic(F3);
    const int l0 = K.pl0[p], nl = K.pl0[p + 1] - l0;
    const int base = l0 * F3;
    C* b2 = (C*)f.b2 + ((size_t)k * f.ncol + c) * f.b2_col + (size_t)p * n2;
    const ToepDesc td = f.td[k];
    const int j0 = K.lg0[l0], j1 = K.lg0[l0 + nl];
    if (!fwd) {
        for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) A[i] = cmk<C>(0, 0);
        __syncthreads();
        for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x)
            A[K.lpos[j] - base] = cvt(td.X[K.gperm[j] + (size_t)c * td.ldx], C());
        __syncthreads();
        C* r = fft_lines(A, B, nl, F3, f, 2, W3, true);
        C* P = (r == A) ? B : A;
        for (int i = threadIdx.x; i < n2; i += blockDim.x) P[i] = cmk<C>(0, 0);
        __syncthreads();
        for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) {
            const int l = fft_div(i, m3), r3 = i - l * F3;
            P[K.lr2[l0 + l] * F3 + r3] = r[i];
        }
        __syncthreads();
        const C* q = fft_cols(P, r, F3, F2, f, 1, W2, true);
        for (int i = threadIdx.x; i < n2; i += blockDim.x) b2[i] = q[i];
    } else {
        for (int i = threadIdx.x; i < n2; i += blockDim.x) A[i] = b2[i];
        __syncthreads();
        C* q = fft_cols(A, B, F3, F2, f, 1, W2, false);
        C* o = (q == A) ? B : A;
        for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) {
            const int l = fft_div(i, m3), r3 = i - l * F3;
            o[i] = q[K.lr2[l0 + l] * F3 + r3];
        }
        __syncthreads();
        const C* r = fft_lines(o, q, nl, F3, f, 2, W3, false);
        for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x)
            td.Y[K.gperm[j] + (size_t)c * td.ldy] = todz(r[K.lpos[j] - base]);
    }
}

// ---------------------------------------------------------------- fixed point
// The FP64 form's convolution on the integer pipe.  FP64 instructions (2 lanes
// per clock and SM) bound its transforms: a radix-4 butterfly has 28 of them,
// 14 clocks a lane; in 64-bit integers its 16 additions are 2 instructions each
// at 64 or more lanes per clock and a twiddle 12 wide products at about 16.
// Values are q 2^e with one exponent per block of a pass: a block takes the
// largest magnitude of the blocks that it reads, aligned so that its transform
// of L points cannot pass 2^62 (the terms of any partial sum are at most
// sqrt(2) L times the largest part), and stores the bit length of its results.
// So 54 bits or more lie below the largest value of a block at each pass (the
// reason for FX_MAX_N), and what a pass rounds is below what FP64 rounds in it.
// A block that reads an infinity or a NaN makes the column NaN, as the sums did.
// 200 columns on 48^3 points 3273 -> 1367 us, 60 columns of the interface 1414 ->
// 613 us, 7 columns of 25527 plane waves 524 -> 245 us (FP64 transforms before).
// Exponent entries: x = e, y = top, the values are below 2^top.
#define FX_MAX_N 181              // 61.5 - log2(181) = 54 bits
#define FX_ZERO (-(1 << 28))      // top of a block of zeros (its values are not stored)
#define FX_NAN (1 << 28)          // top of a block that met a non-finite value (nor are these)

// bits that the values of a transform of L points may start with: floor(61.5 - log2 L)
static int fx_bits(int L) {
    int b = 61;
    while ((double)L * (double)(1LL << b) > 3260954456333195553.0) --b;
    return b;
}
__device__ __forceinline__ long long fx_sh1(long long v, int s) {
    if (s >= 0) return v << s;
    const int n = -s;
    return n > 62 ? 0 : (v + (1LL << (n - 1))) >> n;
}
__device__ __forceinline__ zq fx_sh(zq v, int s) { return cmk<zq>(fx_sh1(v.x, s), fx_sh1(v.y, s)); }
__device__ __forceinline__ unsigned long long fx_mag(zq v) {
    return (unsigned long long)((v.x ^ (v.x >> 63)) | (v.y ^ (v.y >> 63)));
}
// largest m of the block (two barriers)
__device__ __forceinline__ int fx_bmax(int m, int* red) {
    m = __reduce_max_sync(0xffffffffu, m);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, red[w]);
    return m;
}
// bit length of the block's largest magnitude (0: all zero)
__device__ __forceinline__ int fx_bbits(unsigned long long o, int* red) {
    const unsigned h = __reduce_or_sync(0xffffffffu, (unsigned)(o >> 32));
    const unsigned l = __reduce_or_sync(0xffffffffu, (unsigned)o);
    return fx_bmax(h ? 64 - __clz(h) : 32 - __clz(l), red);
}
// exponent field of the larger part (subnormals as 1, zero 0, non-finite 2047)
__device__ __forceinline__ int fx_ex1(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
    return u == 0 ? 0 : max((int)(u >> 52), 1);
}
__device__ __forceinline__ int fx_ex(zd v) { return max(fx_ex1(v.x), fx_ex1(v.y)); }
// v 2^-e for a finite v, rounded to an integer (below 2^62)
__device__ __forceinline__ long long fx_from1(double v, int e) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const int ex = (int)(u >> 52) & 2047;
    const long long m = (long long)(u & 0xfffffffffffffULL) | (ex ? 1LL << 52 : 0LL);
    const long long q = fx_sh1(m, max(ex, 1) - 1075 - e);
    return v < 0.0 ? -q : q;
}
__device__ __forceinline__ zq fx_from(zd v, int e) { return cmk<zq>(fx_from1(v.x, e), fx_from1(v.y, e)); }
// the exponent entry of results below 2^bits with exponent e
__device__ __forceinline__ int2 fx_entry(int e, int bits) { return make_int2(e, bits ? e + bits : FX_ZERO); }
// the value of an entry's block aligned to exponent e
__device__ __forceinline__ zq fx_get(const zq* p, int2 m, int e) {
    return m.y == FX_ZERO ? cmk<zq>(0, 0) : fx_sh(*p, m.x - e);
}

// The potential of a call, v + s vd, v or s vd, in fixed point: values below
// 2^61 of 2^62, an exponent per block of pass C (its (r2, chunk))
__global__ void __launch_bounds__(FFT_THREADS) k_fx_v(FftArgs f, tq* __restrict__ vq, int* __restrict__ vqe) {
    __shared__ int red[8];
    const int F1 = f.F1, F3 = f.F3, LPB = f.lpb[0];
    const int nch = (F3 + LPB - 1) / LPB;
    const int r2 = blockIdx.x / nch, i30 = (blockIdx.x - r2 * nch) * LPB;
    const int nl = min(LPB, F3 - i30);
    const unsigned mnl = fft_magic(nl);
    const size_t pst = (size_t)f.F2 * F3, off = (size_t)r2 * F3 + i30;
    const zd* v = (const zd*)f.v;
    const zd* vd = (const zd*)f.vd;
    const double sc = f.vmode != 0 || f.use_vd ? *f.s : 0.0;
    zd pv[FFT_PV];  // F1 nl <= FFT_BLK_PTS
    int m = 0;
#pragma unroll
    for (int u = 0; u < FFT_PV; ++u) {
        const int i = threadIdx.x + u * FFT_THREADS;
        pv[u] = zmk(0.0, 0.0);
        if (i < F1 * nl) {
            const int r1 = fft_div(i, mnl), l = i - r1 * nl;
            const size_t gi = (size_t)r1 * pst + off + l;
            if (f.vmode == 0) pv[u] = v[gi];
            if (f.vmode != 0 || f.use_vd) {
                const zd d = vd[gi];
                pv[u] = f.vmode == 0 ? zmk(pv[u].x + sc * d.x, pv[u].y + sc * d.y) : zmk(sc * d.x, sc * d.y);
            }
        }
        m = max(m, fx_ex(pv[u]));
    }
    m = fx_bmax(m, red);
    // below 2^(m - 1022): e = that - 61 leaves |v| < 2^61
    const int e = m - 1022 - 61;
    if (threadIdx.x == 0) vqe[blockIdx.x] = m == 0 ? FX_ZERO : m == 2047 ? FX_NAN : e + 62;
    if (m == 0 || m == 2047) return;
#pragma unroll
    for (int u = 0; u < FFT_PV; ++u) {
        const int i = threadIdx.x + u * FFT_THREADS;
        if (i < F1 * nl) {
            const int r1 = fft_div(i, mnl), l = i - r1 * nl;
            const zq q = fx_from(pv[u], e);
            vq[(size_t)r1 * pst + off + l] = tq{qsplit(q.x), qsplit(q.y)};
        }
    }
}

// Passes A to E as above
__global__ void __launch_bounds__(FFT_THREADS) k_fx_a(FftArgs f) {
    extern __shared__ __align__(16) unsigned char fsm[];
    __shared__ int red[8];
    const int F3 = f.F3, LPB = f.lpb[2];
    tq* W = (tq*)fsm;
    zq* x = (zq*)W + F3;
    zq* y = x + LPB * F3;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int l0 = blockIdx.x * LPB;
    if (l0 >= K.nline) return;
    const int nl = min(LPB, K.nline - l0);
    load_tw(W, f.w[2], F3);
    for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) x[i] = cmk<zq>(0, 0);
    const ToepDesc td = f.td[k];
    const zd* X = td.X + (size_t)c * td.ldx;
    const int j0 = K.lg0[l0], j1 = K.lg0[l0 + nl];
    const int base = l0 * F3;
    int m = f.tune;
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) m = max(m, fx_ex(X[K.gperm[j]]));
    m = fx_bmax(m, red);
    const size_t kc = (size_t)k * f.ncol + c;
    const int ch1 = (F3 + f.lpb[1] - 1) / f.lpb[1];
    int2 mt = make_int2(0, m == 0 ? FX_ZERO : FX_NAN);
    if (m != 0 && m != 2047) {
        const int e = m - 1022 - f.qb[2];
        for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) x[K.lpos[j] - base] = fx_from(X[K.gperm[j]], e);
        __syncthreads();
        const zq* r = fft_lines(x, y, nl, F3, f, 2, W, true);
        zq* out = (zq*)f.b3 + kc * f.b3_col + (size_t)base;
        unsigned long long o = f.tune;
        for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) {
            out[i] = r[i];
            o |= fx_mag(r[i]);
        }
        mt = fx_entry(e, fx_bbits(o, red));
    }
    int2* ma = f.ma + (kc * f.lines_max + l0) * ch1;
    for (int i = threadIdx.x; i < nl * ch1; i += blockDim.x) ma[i] = mt;
}

__global__ void __launch_bounds__(FFT_THREADS) k_fx_bd(FftArgs f, int fwd) {
    extern __shared__ __align__(16) unsigned char fsm[];
    __shared__ int red[8];
    const int F2 = f.F2, F3 = f.F3, LPB = f.lpb[1];
    tq* W = (tq*)fsm;
    zq* x = (zq*)W + F2;
    zq* y = x + LPB * F2;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int ch1 = (F3 + LPB - 1) / LPB, ch0 = (F3 + f.lpb[0] - 1) / f.lpb[0];
    const int p = blockIdx.x / ch1, ch = blockIdx.x - p * ch1, i30 = ch * LPB;
    if (p >= K.nplane) return;
    const int nl = min(LPB, F3 - i30);
    load_tw(W, f.w[1], F2);
    const size_t kc = (size_t)k * f.ncol + c;
    zq* b3 = (zq*)f.b3 + kc * f.b3_col;
    zq* b2 = (zq*)f.b2 + kc * f.b2_col + (size_t)p * F2 * F3;
    int2* ma = f.ma + kc * f.lines_max * ch1;
    int2* mb = f.mb + (kc * f.planes_max + p) * ch1;
    const int2* mc = f.mc + kc * F2 * ch0;
    const int* lo = K.line_of + (size_t)p * F2;
    const unsigned mnl = fft_magic(nl), m0 = fft_magic(f.lpb[0]);
    int t = FX_ZERO;
    if (fwd) {
        const int c0 = fft_div(i30, m0), nc = fft_div(i30 + nl - 1, m0) - c0 + 1;
        for (int i = threadIdx.x; i < F2 * nc; i += blockDim.x) t = max(t, mc[(i / nc) * ch0 + c0 + i % nc].y);
    } else {
        for (int r2 = threadIdx.x; r2 < F2; r2 += blockDim.x)
            if (lo[r2] >= 0) t = max(t, ma[lo[r2] * ch1 + ch].y);
    }
    t = fx_bmax(t, red);
    int2 mt = make_int2(0, t);
    if (t != FX_ZERO && t != FX_NAN) {
        const int e = t - f.qb[1];
        for (int i = threadIdx.x; i < F2 * nl; i += blockDim.x) {
            const int r2 = fft_div(i, mnl), l = i - r2 * nl;
            zq v = cmk<zq>(0, 0);
            if (fwd) {
                v = fx_get(b2 + (size_t)r2 * F3 + i30 + l, mc[r2 * ch0 + fft_div(i30 + l, m0)], e);
            } else {
                const int id = lo[r2];
                if (id >= 0) v = fx_get(b3 + (size_t)id * F3 + i30 + l, ma[id * ch1 + ch], e);
            }
            x[i] = v;
        }
        __syncthreads();
        const zq* r = fft_cols(x, y, nl, F2, f, 1, W, !fwd);
        unsigned long long o = f.tune;
        for (int i = threadIdx.x; i < F2 * nl; i += blockDim.x) {
            const int r2 = fft_div(i, mnl), l = i - r2 * nl;
            if (fwd) {
                const int id = lo[r2];
                if (id >= 0) {
                    b3[(size_t)id * F3 + i30 + l] = r[i];
                    o |= fx_mag(r[i]);
                }
            } else {
                b2[(size_t)r2 * F3 + i30 + l] = r[i];
                o |= fx_mag(r[i]);
            }
        }
        mt = fx_entry(e, fx_bbits(o, red));
    }
    if (fwd) {
        for (int l = K.pl0[p] + threadIdx.x; l < K.pl0[p + 1]; l += blockDim.x) ma[l * ch1 + ch] = mt;
    } else if (threadIdx.x == 0) {
        mb[ch] = mt;
    }
}

__global__ void __launch_bounds__(FFT_THREADS) k_fx_c(FftArgs f) {
    extern __shared__ __align__(16) unsigned char fsm[];
    __shared__ int red[8];
    const int F1 = f.F1, F2 = f.F2, F3 = f.F3, LPB = f.lpb[0];
    tq* W = (tq*)fsm;
    zq* x = (zq*)W + F1;
    zq* y = x + LPB * F1;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int ch0 = (F3 + LPB - 1) / LPB, ch1 = (F3 + f.lpb[1] - 1) / f.lpb[1];
    const int r2 = blockIdx.x / ch0, i30 = (blockIdx.x - r2 * ch0) * LPB;
    const int nl = min(LPB, F3 - i30);
    load_tw(W, f.w[0], F1);
    const size_t kc = (size_t)k * f.ncol + c;
    zq* b2 = (zq*)f.b2 + kc * f.b2_col;
    const int2* mb = f.mb + kc * f.planes_max * ch1;
    const size_t pst = (size_t)F2 * F3, off = (size_t)r2 * F3 + i30;
    const unsigned mnl = fft_magic(nl), m1 = fft_magic(f.lpb[1]);
    int t = FX_ZERO;
    {
        const int c1 = fft_div(i30, m1), nc = fft_div(i30 + nl - 1, m1) - c1 + 1;
        for (int i = threadIdx.x; i < K.nplane * nc; i += blockDim.x) t = max(t, mb[(i / nc) * ch1 + c1 + i % nc].y);
    }
    const int ve = f.vqe[blockIdx.x];
    t = fx_bmax(t, red);
    int2 mt = make_int2(0, t == FX_NAN || ve == FX_NAN ? FX_NAN : FX_ZERO);
    if (t != FX_ZERO && t != FX_NAN && ve != FX_ZERO && ve != FX_NAN) {
        const int b = f.qb[0];
        int e = t - b;
        for (int i = threadIdx.x; i < F1 * nl; i += blockDim.x) {
            const int r1 = fft_div(i, mnl), l = i - r1 * nl;
            const int p = K.plane_of[r1];
            x[i] = p >= 0 ? fx_get(b2 + (size_t)p * pst + off + l, mb[p * ch1 + fft_div(i30 + l, m1)], e) : cmk<zq>(0, 0);
        }
        __syncthreads();
        zq* r = fft_cols(x, y, nl, F1, f, 0, W, true);
        // times v (its own exponent), and aligned again
        unsigned long long o = f.tune;
        for (int i = threadIdx.x; i < F1 * nl; i += blockDim.x) {
            const int r1 = fft_div(i, mnl), l = i - r1 * nl;
            const zq w = cml(r[i], f.vq[(size_t)r1 * pst + off + l]);
            r[i] = w;
            o |= fx_mag(w);
        }
        const int bits = fx_bbits(o, red), sh = b - bits;
        e += ve - sh;
        for (int i = threadIdx.x; i < F1 * nl; i += blockDim.x) r[i] = fx_sh(r[i], sh);
        __syncthreads();
        const zq* q = fft_cols(r, r == x ? y : x, nl, F1, f, 0, W, false);
        o = f.tune;
        for (int i = threadIdx.x; i < F1 * nl; i += blockDim.x) {
            const int r1 = fft_div(i, mnl), l = i - r1 * nl;
            const int p = K.plane_of[r1];
            if (p >= 0) {
                b2[(size_t)p * pst + off + l] = q[i];
                o |= fx_mag(q[i]);
            }
        }
        mt = fx_entry(e, fx_bbits(o, red));
    }
    if (threadIdx.x == 0) f.mc[kc * F2 * ch0 + blockIdx.x] = mt;
}

// q 2^e in FP64: one product by a power of two where that is a normal number
__device__ __forceinline__ zd fx_out(zq v, int e) {
    if (e > -960 && e < 960) {
        const double f = __longlong_as_double((long long)(e + 1023) << 52);
        return zmk((double)v.x * f, (double)v.y * f);
    }
    return zmk(scalbn((double)v.x, e), scalbn((double)v.y, e));
}

__global__ void __launch_bounds__(FFT_THREADS) k_fx_e(FftArgs f) {
    extern __shared__ __align__(16) unsigned char fsm[];
    __shared__ int red[8];
    const int F3 = f.F3, LPB = f.lpb[2];
    tq* W = (tq*)fsm;
    zq* x = (zq*)W + F3;
    zq* y = x + LPB * F3;
    const int k = blockIdx.z, c = blockIdx.y;
    const FftK K = f.fk[k];
    const int l0 = blockIdx.x * LPB;
    if (l0 >= K.nline) return;
    const int nl = min(LPB, K.nline - l0);
    load_tw(W, f.w[2], F3);
    const int base = l0 * F3;
    const size_t kc = (size_t)k * f.ncol + c;
    const int ch1 = (F3 + f.lpb[1] - 1) / f.lpb[1];
    const unsigned m1 = fft_magic(f.lpb[1]), m3 = fft_magic(F3);
    const int2* ma = f.ma + (kc * f.lines_max + l0) * ch1;
    const zq* in = (const zq*)f.b3 + kc * f.b3_col + (size_t)base;
    int t = FX_ZERO;
    for (int i = threadIdx.x; i < nl * ch1; i += blockDim.x) t = max(t, ma[i].y);
    t = fx_bmax(t, red);
    const ToepDesc td = f.td[k];
    zd* Y = td.Y + (size_t)c * td.ldy;
    const int j0 = K.lg0[l0], j1 = K.lg0[l0 + nl];
    if (t == FX_ZERO || t == FX_NAN) {
        const double v = t == FX_NAN ? nan("") : 0.0;
        for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) Y[K.gperm[j]] = zmk(v, v);
        return;
    }
    const int e = t - f.qb[2];
    for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) {
        const int l = fft_div(i, m3);
        x[i] = fx_get(in + i, ma[l * ch1 + fft_div(i - l * F3, m1)], e);
    }
    __syncthreads();
    const zq* r = fft_lines(x, y, nl, F3, f, 2, W, false);
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) Y[K.gperm[j]] = fx_out(r[K.lpos[j] - base], e);
}

// A+B (fwd = 0) and D+E (fwd = 1) of one plane, aligned again between the axes
__global__ void __launch_bounds__(FFT_PTHREADS) k_fx_plane(FftArgs f, int fwd) {
    extern __shared__ __align__(16) unsigned char fsm[];
    __shared__ int red[8];
    const int F2 = f.F2, F3 = f.F3, n2 = F2 * F3;
    tq* W2 = (tq*)fsm;
    tq* W3 = W2 + F2;
    zq* A = (zq*)W3 + F3;
    zq* B = A + n2;
    const int k = blockIdx.z, c = blockIdx.y, p = blockIdx.x;
    const FftK K = f.fk[k];
    if (p >= K.nplane) return;
    load_tw(W2, f.w[1], F2);
    load_tw(W3, f.w[2], F3);
    const unsigned m3 = fft_magic(F3), m0 = fft_magic(f.lpb[0]);
    const int l0 = K.pl0[p], nl = K.pl0[p + 1] - l0;
    const int base = l0 * F3;
    const size_t kc = (size_t)k * f.ncol + c;
    const int ch1 = (F3 + f.lpb[1] - 1) / f.lpb[1], ch0 = (F3 + f.lpb[0] - 1) / f.lpb[0];
    zq* b2 = (zq*)f.b2 + kc * f.b2_col + (size_t)p * n2;
    const ToepDesc td = f.td[k];
    const int j0 = K.lg0[l0], j1 = K.lg0[l0 + nl];
    unsigned long long o = f.tune;
    if (!fwd) {
        const zd* X = td.X + (size_t)c * td.ldx;
        int m = f.tune;
        for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) m = max(m, fx_ex(X[K.gperm[j]]));
        for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) A[i] = cmk<zq>(0, 0);
        m = fx_bmax(m, red);
        int2 mt = make_int2(0, m == 0 ? FX_ZERO : FX_NAN);
        if (m != 0 && m != 2047) {
            int e = m - 1022 - f.qb[2];
            for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) A[K.lpos[j] - base] = fx_from(X[K.gperm[j]], e);
            __syncthreads();
            zq* r = fft_lines(A, B, nl, F3, f, 2, W3, true);
            zq* P = (r == A) ? B : A;
            for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) o |= fx_mag(r[i]);
            for (int i = threadIdx.x; i < n2; i += blockDim.x) P[i] = cmk<zq>(0, 0);
            const int sh = f.qb[1] - fx_bbits(o, red);
            e -= sh;
            for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) {
                const int l = fft_div(i, m3), r3 = i - l * F3;
                P[K.lr2[l0 + l] * F3 + r3] = fx_sh(r[i], sh);
            }
            __syncthreads();
            const zq* q = fft_cols(P, r, F3, F2, f, 1, W2, true);
            o = f.tune;
            for (int i = threadIdx.x; i < n2; i += blockDim.x) {
                b2[i] = q[i];
                o |= fx_mag(q[i]);
            }
            mt = fx_entry(e, fx_bbits(o, red));
        }
        for (int i = threadIdx.x; i < ch1; i += blockDim.x) f.mb[(kc * f.planes_max + p) * ch1 + i] = mt;
    } else {
        const int2* mc = f.mc + kc * F2 * ch0;
        int t = FX_ZERO;
        for (int i = threadIdx.x; i < F2 * ch0; i += blockDim.x) t = max(t, mc[i].y);
        t = fx_bmax(t, red);
        zd* Y = td.Y + (size_t)c * td.ldy;
        if (t == FX_ZERO || t == FX_NAN) {
            const double v = t == FX_NAN ? nan("") : 0.0;
            for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) Y[K.gperm[j]] = zmk(v, v);
            return;
        }
        int e = t - f.qb[1];
        for (int i = threadIdx.x; i < n2; i += blockDim.x) {
            const int r2 = fft_div(i, m3);
            A[i] = fx_get(b2 + i, mc[r2 * ch0 + fft_div(i - r2 * F3, m0)], e);
        }
        __syncthreads();
        zq* q = fft_cols(A, B, F3, F2, f, 1, W2, false);
        zq* u = (q == A) ? B : A;
        for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) {
            const int l = fft_div(i, m3), r3 = i - l * F3;
            u[i] = q[K.lr2[l0 + l] * F3 + r3];
            o |= fx_mag(u[i]);
        }
        const int sh = f.qb[2] - fx_bbits(o, red);
        e -= sh;
        for (int i = threadIdx.x; i < nl * F3; i += blockDim.x) u[i] = fx_sh(u[i], sh);
        __syncthreads();
        const zq* r = fft_lines(u, q, nl, F3, f, 2, W3, false);
        for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) Y[K.gperm[j]] = fx_out(r[K.lpos[j] - base], e);
    }
}

// Interstitial density of the propagated states on the grid: for every
// (r2, r3) line of axis 1 the inverse transform of each (k, state) column
// (planes from the plane pass), |psi|^2 summed with the weights w_k f_j in
// (k, j) order; n(r) = that sum / Omega (psi~ = sqrt(Omega) psi here)
template <typename C>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_density(FftArgs f, int nk, const double* __restrict__ occ,
                                                          const double* __restrict__ wk, double inv_omega, C* rho) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int F1 = f.F1, F2 = f.F2, F3 = f.F3, LPB = f.lpb[0];
    C* W = (C*)fsm;
    C* x = W + F1;
    C* y = x + LPB * F1;
    const int nch = (F3 + LPB - 1) / LPB;
    const int r2 = blockIdx.x / nch, i30 = (blockIdx.x - r2 * nch) * LPB;
    const int nl = min(LPB, F3 - i30);
    load_tw(W, f.w[0], F1);
    const size_t pst = (size_t)F2 * F3;
    const size_t off = (size_t)r2 * F3 + i30;
    constexpr int PV = FFT_PV;
    double acc[PV];
#pragma unroll
    for (int u = 0; u < PV; ++u) acc[u] = 0.0;
    for (int k = 0; k < nk; ++k) {
        const FftK K = f.fk[k];
        for (int c = 0; c < f.ncol; ++c) {
            const C* b2 = (const C*)f.b2 + ((size_t)k * f.ncol + c) * f.b2_col;
            for (int i = threadIdx.x; i < F1 * nl; i += blockDim.x) {
                const int r1 = i / nl, l = i - r1 * nl;
                const int p = K.plane_of[r1];
                x[i] = (p >= 0) ? b2[(size_t)p * pst + off + l] : cmk<C>(0, 0);
            }
            __syncthreads();
            const C* r = fft_cols(x, y, nl, F1, f, 0, W, true);
            const double wf = wk[k] * occ[c];
#pragma unroll
            for (int u = 0; u < PV; ++u) {
                const int i = threadIdx.x + u * FFT_THREADS;
                if (i < F1 * nl) {
                    const C v = r[i];
                    acc[u] += wf * ((double)v.x * v.x + (double)v.y * v.y);
                }
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int u = 0; u < PV; ++u) {
        const int i = threadIdx.x + u * FFT_THREADS;
        if (i < F1 * nl) {
            const int r1 = i / nl, l = i - r1 * nl;
            rho[(size_t)r1 * pst + off + l] = cmk<C>((typename Rt<C>::R)(acc[u] * inv_omega), 0);
        }
    }
}

// A full-grid 1-D pass along `axis` (0, 1, 2) in place, every line
template <typename C>
__global__ void __launch_bounds__(FFT_THREADS) k_fft_full(FftArgs f, C* buf, int axis, int inv) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int F1 = f.F1, F2 = f.F2, F3 = f.F3;
    const int L = axis == 0 ? F1 : (axis == 1 ? F2 : F3);
    const int LPB = f.lpb[axis];
    C* W = (C*)fsm;
    C* x = W + L;
    C* y = x + LPB * L;
    load_tw(W, f.w[axis], L);
    size_t base, es, ls;
    int nl;
    if (axis == 2) {
        const int l0 = blockIdx.x * LPB;
        nl = min(LPB, F1 * F2 - l0);
        base = (size_t)l0 * F3;
        es = 1;
        ls = F3;
    } else {
        const int nch = (F3 + LPB - 1) / LPB;
        const int o = blockIdx.x / nch, i30 = (blockIdx.x - o * nch) * LPB;
        nl = min(LPB, F3 - i30);
        es = axis == 1 ? (size_t)F3 : (size_t)F2 * F3;
        base = (axis == 1 ? (size_t)o * F2 * F3 : (size_t)o * F3) + i30;
        ls = 1;
    }
    // element j of line l at base + l ls + j es; coalesced along l for axes 0, 1
    for (int i = threadIdx.x; i < nl * L; i += blockDim.x) {
        int l, j;
        if (axis == 2) {
            l = i / L;
            j = i - l * L;
        } else {
            j = i / nl;
            l = i - j * nl;
        }
        x[l * L + j] = buf[base + l * ls + j * es];
    }
    __syncthreads();
    const C* r = fft_lines(x, y, nl, L, f, axis, W, inv != 0);
    for (int i = threadIdx.x; i < nl * L; i += blockDim.x) {
        int l, j;
        if (axis == 2) {
            l = i / L;
            j = i - l * L;
        } else {
            j = i / nl;
            l = i - j * nl;
        }
        buf[base + l * ls + j * es] = r[l * L + j];
    }
}

// Poisson equation on the table box: vd(g) = 4 pi (N - N0)(g) / (F^6 |g|^2)
// at the residues of |g_i| <= e_i, g != 0, zero elsewhere (N = F^3 n_g; the
// second F^3 is the normalisation of the potential's grid image), and the sum
// of |dV_g| for the bound check
template <typename C>
__global__ void k_hartree(const C* __restrict__ N, const C* __restrict__ N0, C* vd, int F1, int F2, int F3, int e0,
                          int e1, int e2, double b00, double b01, double b02, double b10, double b11, double b12,
                          double b20, double b21, double b22, double inv_f3, double* l1) {
    __shared__ double part[8];
    const size_t n = (size_t)F1 * F2 * F3;
    double mine = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int r2 = (int)(i % F3), r1 = (int)((i / F3) % F2), r0 = (int)(i / ((size_t)F2 * F3));
        const int d0 = r0 <= e0 ? r0 : (r0 >= F1 - e0 ? r0 - F1 : 1 << 20);
        const int d1 = r1 <= e1 ? r1 : (r1 >= F2 - e1 ? r1 - F2 : 1 << 20);
        const int d2 = r2 <= e2 ? r2 : (r2 >= F3 - e2 ? r2 - F3 : 1 << 20);
        C out = cmk<C>(0, 0);
        if (d0 != (1 << 20) && d1 != (1 << 20) && d2 != (1 << 20) && (d0 | d1 | d2) != 0) {
            const double gx = d0 * b00 + d1 * b10 + d2 * b20;
            const double gy = d0 * b01 + d1 * b11 + d2 * b21;
            const double gz = d0 * b02 + d1 * b12 + d2 * b22;
            const double g2 = gx * gx + gy * gy + gz * gz;
            const double f = 4.0 * 3.14159265358979323846 * inv_f3 / g2;  // 4 pi / (F^3 |g|^2)
            const double dre = ((double)N[i].x - (double)N0[i].x) * inv_f3;
            const double dim = ((double)N[i].y - (double)N0[i].y) * inv_f3;
            out = cmk<C>((typename Rt<C>::R)(f * dre), (typename Rt<C>::R)(f * dim));
            mine += f * sqrt(dre * dre + dim * dim) / inv_f3;
        }
        vd[i] = out;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    mine = warp_sum(mine);
    if (lane == 0) part[warp] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
        atomicAdd(l1, t);  // only compared with the bound: the order does not matter
    }
}

// the device accumulator compared with the bound after every step (other parts of
// the potential change add their own bounds to it before the check)
double* fft_l1(const FftPlan* pl) { return pl ? pl->l1 : nullptr; }

// the l1 norm of dV against the bound of the spectral interval; flag bit 6
__global__ void k_hartree_check(double* l1, double bound, int* flag) {
    if (*l1 > bound) atomicOr(flag, 64);
    *l1 = 0.0;
}

// ---------------------------------------------------------------- set-up kernels
// V~ placed on the grid by residue
__global__ void k_fft_place(const zd* tab, int d0, int d1, int d2, int F1, int F2, int F3, zd* grid) {
    const int n = d0 * d1 * d2;
    const int e0 = (d0 - 1) / 2, e1 = (d1 - 1) / 2, e2 = (d2 - 1) / 2;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int i2 = i % d2, i1 = (i / d2) % d1, i0 = i / (d1 * d2);
        const int r0 = ((i0 - e0) % F1 + F1) % F1;
        const int r1 = ((i1 - e1) % F2 + F2) % F2;
        const int r2 = ((i2 - e2) % F3 + F3) % F3;
        grid[((size_t)r0 * F2 + r1) * F3 + r2] = tab[i];
    }
}

// out = scale * (inverse DFT along axis `ax` of in), directly (set-up only)
__global__ void k_fft_dft_axis(const zd* in, zd* out, int F1, int F2, int F3, int ax, const zd* W, double scale) {
    const int n = F1 * F2 * F3;
    const int L = ax == 0 ? F1 : (ax == 1 ? F2 : F3);
    const int st = ax == 0 ? F2 * F3 : (ax == 1 ? F3 : 1);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int j = (i / st) % L;
        const int b = i - j * st;
        zd acc = zmk(0.0, 0.0);
        for (int m = 0; m < L; ++m) {
            const zd w = W[(int)(((long long)j * m) % L)];
            zfma(acc, in[b + (size_t)m * st], zmk(w.x, -w.y));
        }
        out[i] = zscale(acc, scale);
    }
}

__global__ void k_fft_to32(const zd* in, zf* out, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = make_float2((float)in[i].x, (float)in[i].y);
}

// ---------------------------------------------------------------- host side
static bool factor_axis(int n, int* rad, int* nst) {
    int k = 0;
    while (n % 4 == 0 && k < FFT_MAX_ST) {
        rad[k++] = 4;
        n /= 4;
    }
    const int ps[3] = {2, 3, 5};
    for (int pi = 0; pi < 3; ++pi)
        while (n % ps[pi] == 0 && k < FFT_MAX_ST) {
            rad[k++] = ps[pi];
            n /= ps[pi];
        }
    *nst = k;
    return n == 1;
}

// smallest 2^a 3^b 5^c >= n
static int smooth_at_least(int n) {
    for (int m = std::max(n, 1);; ++m) {
        int r = m;
        for (int p : {2, 3, 5})
            while (r % p == 0) r /= p;
        if (r == 1) return m;
    }
}

static size_t fft_smem(int L, int elt) { return (size_t)(L + 2 * fft_lpb(L) * L) * elt; }
static size_t fft_plane_smem(int F2, int F3, int elt) { return (size_t)(F2 + F3 + 2 * F2 * F3) * elt; }
#define FFT_PLANE_SMEM_MAX (200 * 1024)
// blocks of a line pass over one row of axis 3
static inline int fft_chunks(int F3, int L) { return (F3 + fft_lpb(L) - 1) / fft_lpb(L); }

template <typename T> static T* fdalloc(size_t n, std::string* why, bool* ok) {
    void* p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(n, 1) * sizeof(T)) != cudaSuccess) {
        *ok = false;
        if (why) *why = "FFT route: device allocation failed";
        return nullptr;
    }
    return (T*)p;
}

int fft_grid_for(const int vt_dim[3], int F[3]) {
    for (int i = 0; i < 3; ++i) {
        F[i] = smooth_at_least(vt_dim[i]);
        if (F[i] > FFT_MAX_N) return -1;
    }
    return 0;
}

static bool potential_on_grid(const FftPlan* pl, const zd* tab, const int vt_dim[3], zd* v64, zf* v32,
                              cudaStream_t st) {
    const int F1 = pl->F[0], F2 = pl->F[1], F3 = pl->F[2];
    const size_t n = (size_t)F1 * F2 * F3;
    zd* tmp = nullptr;
    if (cudaMalloc(&tmp, n * sizeof(zd)) != cudaSuccess) return false;
    cudaMemsetAsync(v64, 0, n * sizeof(zd), st);
    k_fft_place<<<256, 256, 0, st>>>(tab, vt_dim[0], vt_dim[1], vt_dim[2], F1, F2, F3, v64);
    const double inv = 1.0 / ((double)F1 * F2 * F3);
    const int nb = (int)std::min<size_t>((n + 255) / 256, 4096);
    k_fft_dft_axis<<<nb, 256, 0, st>>>(v64, tmp, F1, F2, F3, 0, pl->w64[0], 1.0);
    k_fft_dft_axis<<<nb, 256, 0, st>>>(tmp, v64, F1, F2, F3, 1, pl->w64[1], 1.0);
    cudaMemcpyAsync(tmp, v64, n * sizeof(zd), cudaMemcpyDeviceToDevice, st);
    k_fft_dft_axis<<<nb, 256, 0, st>>>(tmp, v64, F1, F2, F3, 2, pl->w64[2], inv);
    if (v32) k_fft_to32<<<nb, 256, 0, st>>>(v64, v32, n);
    const bool ok = cudaStreamSynchronize(st) == cudaSuccess;
    cudaFree(tmp);
    return ok;
}

// device bytes that a potential change over ncol columns asks for: the grids of the
// change and of the density, and the transform buffers
size_t fft_change_bytes(const FftPlan* pl, int ncol) {
    if (!pl) return 0;
    const size_t elt = pl->prec == 0 ? sizeof(zd) : sizeof(zf), L = pl->max_lines, P = pl->max_planes;
    const size_t ch1 = fft_chunks(pl->F[2], pl->F[1]), ch0 = fft_chunks(pl->F[2], pl->F[0]);
    return (size_t)pl->F[0] * pl->F[1] * pl->F[2] * (3 * sizeof(zd) + sizeof(zf)) + (size_t)pl->nk * ncol *
           ((L + P * pl->F[1]) * pl->F[2] * elt + (pl->fx ? ((L + P) * ch1 + pl->F[1] * ch0) * sizeof(int2) : 0));
}
static bool fft_alloc_buffers(FftPlan* pl, int ncol, std::string* why) {
    const size_t elt = pl->prec == 0 ? sizeof(zd) : sizeof(zf);
    const size_t c3 = (size_t)pl->max_lines * pl->F[2];
    const size_t c2 = (size_t)pl->max_planes * pl->F[1] * pl->F[2];
    void* b3 = nullptr;
    void* b2 = nullptr;
    // exponents of the fixed-point form: per (line, chunk), (plane, chunk), (r2, chunk)
    const size_t nm = pl->fx ? (size_t)pl->nk * ncol : 0;
    const size_t ch1 = fft_chunks(pl->F[2], pl->F[1]), ch0 = fft_chunks(pl->F[2], pl->F[0]);
    const size_t na = nm * pl->max_lines * ch1, nb = nm * pl->max_planes * ch1, nc = nm * pl->F[1] * ch0;
    int2* mm = nullptr;
    if (cudaMalloc(&b3, std::max<size_t>((size_t)pl->nk * ncol * c3 * elt, 16)) != cudaSuccess ||
        cudaMalloc(&b2, std::max<size_t>((size_t)pl->nk * ncol * c2 * elt, 16)) != cudaSuccess ||
        (nm && cudaMalloc((void**)&mm, (na + nb + nc) * sizeof(int2)) != cudaSuccess)) {
        if (b3) cudaFree(b3);
        if (b2) cudaFree(b2);
        cudaGetLastError();
        if (why) *why = "FFT route: device allocation of the transform buffers failed";
        return false;
    }
    if (pl->ma) cudaFree(pl->ma);
    pl->ma = mm;
    pl->mb = mm + na;
    pl->mc = mm + na + nb;
    if (pl->b3) cudaFree(pl->b3);
    if (pl->b2) cudaFree(pl->b2);
    pl->b3 = b3;
    pl->b2 = b2;
    pl->ncol = ncol;
    return true;
}

int fft_plan_create(FftPlan** out, int nk, const int* ng, const int* const* gint, const int vt_dim[3],
                    const zd* vtab_dev, int ncol, int prec, cudaStream_t st, std::string* why) {
    *out = nullptr;
    FftPlan* pl = new FftPlan();
    pl->prec = prec;
    pl->nk = nk;
    if (fft_grid_for(vt_dim, pl->F)) {
        if (why) *why = "FFT route: a table extent needs more than 512 grid points";
        delete pl;
        return RTTDDFT_ERR_UNSUPPORTED;
    }
    for (int a = 0; a < 3; ++a) factor_axis(pl->F[a], pl->rad[a], &pl->nst[a]);
    bool ok = true;
    // twiddles from the C library's cos and sin in FP64
    for (int a = 0; a < 3; ++a) {
        const int L = pl->F[a];
        std::vector<zd> w(L);
        std::vector<zf> w32(L);
        for (int m = 0; m < L; ++m) {
            const double ang = 2.0 * M_PI * (double)m / (double)L;
            w[m] = zmk(std::cos(ang), -std::sin(ang));
            w32[m] = make_float2((float)w[m].x, (float)w[m].y);
        }
        pl->w64[a] = fdalloc<zd>(L, why, &ok);
        pl->w32[a] = fdalloc<zf>(L, why, &ok);
        if (!ok) break;
        cudaMemcpy(pl->w64[a], w.data(), L * sizeof(zd), cudaMemcpyHostToDevice);
        cudaMemcpy(pl->w32[a], w32.data(), L * sizeof(zf), cudaMemcpyHostToDevice);
    }
    // per-k line tables: entries sorted by (n1, n2, n3); a line is a run of
    // equal (n1, n2), a plane a run of equal n1
    const int F1 = pl->F[0], F2 = pl->F[1], F3 = pl->F[2];
    std::vector<FftK> hk(nk);
    pl->max_lines = 1;
    pl->max_planes = 1;
    for (int k = 0; k < nk && ok; ++k) {
        const int n = ng[k];
        const int* gi = gint[k];
        std::vector<int> perm(n);
        for (int g = 0; g < n; ++g) perm[g] = g;
        std::sort(perm.begin(), perm.end(), [&](int a, int b) {
            const int* x = gi + 3 * a;
            const int* y = gi + 3 * b;
            if (x[0] != y[0]) return x[0] < y[0];
            if (x[1] != y[1]) return x[1] < y[1];
            return x[2] < y[2];
        });
        auto res = [](int v, int F) { return ((v % F) + F) % F; };
        std::vector<int> lg0, lpos(n), plane_of(F1, -1), line_of, pl0, lr2;
        int nline = 0, nplane = 0;
        for (int j = 0; j < n; ++j) {
            const int* t = gi + 3 * perm[j];
            const bool newplane = (j == 0) || t[0] != gi[3 * perm[j - 1]];
            const bool newline = newplane || t[1] != gi[3 * perm[j - 1] + 1];
            if (newplane) {
                plane_of[res(t[0], F1)] = nplane++;
                line_of.resize((size_t)nplane * F2, -1);
                pl0.push_back(nline);
            }
            if (newline) {
                lg0.push_back(j);
                lr2.push_back(res(t[1], F2));
                line_of[(size_t)(nplane - 1) * F2 + res(t[1], F2)] = nline++;
            }
            lpos[j] = (nline - 1) * F3 + res(t[2], F3);
        }
        lg0.push_back(n);
        pl0.push_back(nline);
        auto up = [&](const std::vector<int>& v) -> const int* {
            int* d = fdalloc<int>(v.size(), why, &ok);
            if (!ok) return nullptr;
            cudaMemcpy(d, v.data(), v.size() * sizeof(int), cudaMemcpyHostToDevice);
            pl->tables.push_back(d);
            return d;
        };
        hk[k].nline = nline;
        hk[k].nplane = nplane;
        hk[k].lg0 = up(lg0);
        hk[k].gperm = up(perm);
        hk[k].lpos = up(lpos);
        hk[k].plane_of = up(plane_of);
        hk[k].line_of = up(line_of);
        hk[k].pl0 = up(pl0);
        hk[k].lr2 = up(lr2);
        pl->max_lines = std::max(pl->max_lines, nline);
        pl->max_planes = std::max(pl->max_planes, nplane);
    }
    if (ok) {
        pl->d_fk = fdalloc<FftK>(nk, why, &ok);
        if (ok) cudaMemcpy(pl->d_fk, hk.data(), nk * sizeof(FftK), cudaMemcpyHostToDevice);
    }
    const size_t n3 = (size_t)F1 * F2 * F3;
    pl->fx = prec == 0 && std::max(F1, std::max(F2, F3)) <= FX_MAX_N;
    const int nvb = F2 * fft_chunks(F3, F1);
    for (int a = 0; a < 3 && pl->fx; ++a) {
        const int L = pl->F[a];
        std::vector<tq> w(L);
        for (int m = 0; m < L; ++m) {
            const long double th = 2.0L * 3.14159265358979323846264338327950288L * m / L;
            w[m].x = qsplit(llroundl(cosl(th) * 4611686018427387904.0L));
            w[m].y = qsplit(-llroundl(sinl(th) * 4611686018427387904.0L));
        }
        pl->wq[a] = fdalloc<tq>(L, why, &ok);
        if (ok) cudaMemcpy(pl->wq[a], w.data(), L * sizeof(tq), cudaMemcpyHostToDevice);
    }
    for (int i = 0; i < 2 && pl->fx; ++i) {
        pl->vq[i] = fdalloc<tq>(n3, why, &ok);
        pl->vqe[i] = fdalloc<int>(nvb, why, &ok);
    }
    if (ok) pl->v64 = fdalloc<zd>(n3, why, &ok);
    if (ok && prec != 0) pl->v32 = fdalloc<zf>(n3, why, &ok);
    if (ok) ok = fft_alloc_buffers(pl, ncol, why);
    if (ok && !potential_on_grid(pl, vtab_dev, vt_dim, pl->v64, pl->v32, st)) {
        ok = false;
        if (why) *why = "FFT route: the potential's grid image failed";
    }
    if (ok) {
        // dynamic shared memory beyond 48 KB for the longest axes
        const int elt = prec == 0 ? (int)sizeof(zd) : (int)sizeof(zf);
        const int mx = (int)fft_smem(std::max(F1, std::max(F2, F3)), elt);
        const size_t psm = fft_plane_smem(F2, F3, elt);
        if (psm <= FFT_PLANE_SMEM_MAX) {
            if (pl->fx) raise_smem((const void*)k_fx_plane, (int)psm);
            if (prec == 0) raise_smem((const void*)k_fft_plane<zd>, (int)psm);
            else raise_smem((const void*)k_fft_plane<zf>, (int)psm);
        }
        if (pl->fx) {
            raise_smem((const void*)k_fx_a, mx);
            raise_smem((const void*)k_fx_bd, mx);
            raise_smem((const void*)k_fx_c, mx);
            raise_smem((const void*)k_fx_e, mx);
            FftArgs f = {};
            f.F1 = F1, f.F2 = F2, f.F3 = F3;
            f.lpb[0] = fft_lpb(F1);
            f.v = pl->v64;
            k_fx_v<<<nvb, FFT_THREADS, 0, st>>>(f, pl->vq[0], pl->vqe[0]);
        }
        if (prec == 0) {
            raise_smem((const void*)k_fft_a<zd>, mx);
            raise_smem((const void*)k_fft_bd<zd>, mx);
            raise_smem((const void*)k_fft_c<zd>, mx);
            raise_smem((const void*)k_fft_e<zd>, mx);
        } else {
            raise_smem((const void*)k_fft_a<zf>, mx);
            raise_smem((const void*)k_fft_bd<zf>, mx);
            raise_smem((const void*)k_fft_c<zf>, mx);
            raise_smem((const void*)k_fft_e<zf>, mx);
        }
        if (cudaGetLastError() != cudaSuccess) {
            ok = false;
            if (why) *why = "FFT route: set-up kernels failed";
        }
    }
    if (!ok) {
        fft_plan_destroy(pl);
        return RTTDDFT_ERR_OOM;
    }
    *out = pl;
    return 0;
}

int fft_set_dv(FftPlan* pl, const zd* dvtab_dev, const int vt_dim[3], int ncol, cudaStream_t st,
               std::string* why) {
    const size_t n3 = (size_t)pl->F[0] * pl->F[1] * pl->F[2];
    bool ok = true;
    if (!pl->vd64) pl->vd64 = fdalloc<zd>(n3, why, &ok);
    if (ok && pl->prec != 0 && !pl->vd32) pl->vd32 = fdalloc<zf>(n3, why, &ok);
    if (!ok) return RTTDDFT_ERR_OOM;
    if (ncol > pl->ncol) {
        cudaStreamSynchronize(st);
        if (!fft_alloc_buffers(pl, ncol, why)) return RTTDDFT_ERR_OOM;
    }
    if (!potential_on_grid(pl, dvtab_dev, vt_dim, pl->vd64, pl->vd32, st) || cudaGetLastError() != cudaSuccess) {
        if (why) *why = "FFT route: potential change set-up failed";
        return RTTDDFT_ERR_CUDA;
    }
    return 0;
}

// transform buffers for at least ncol columns per k-point
int fft_reserve_columns(FftPlan* pl, int ncol, cudaStream_t st, std::string* why) {
    if (ncol <= pl->ncol) return 0;
    cudaStreamSynchronize(st);
    return fft_alloc_buffers(pl, ncol, why) ? 0 : RTTDDFT_ERR_OOM;
}

void fft_plan_destroy(FftPlan* pl) {
    if (!pl) return;
    for (int a = 0; a < 3; ++a) {
        if (pl->w64[a]) cudaFree(pl->w64[a]);
        if (pl->w32[a]) cudaFree(pl->w32[a]);
        if (pl->wq[a]) cudaFree(pl->wq[a]);
    }
    for (int i = 0; i < 2; ++i) {
        if (pl->vq[i]) cudaFree(pl->vq[i]);
        if (pl->vqe[i]) cudaFree(pl->vqe[i]);
    }
    if (pl->ma) cudaFree(pl->ma);
    for (void* p : {(void*)pl->v64, (void*)pl->v32, (void*)pl->vd64, (void*)pl->vd32, (void*)pl->d_fk, pl->b3, pl->b2,
                    (void*)pl->rho, (void*)pl->rho0, (void*)pl->l1, (void*)pl->b3d, (void*)pl->b2d})
        if (p) cudaFree(p);
    for (void* p : pl->tables) cudaFree(p);
    delete pl;
}

void fft_plan_info(const FftPlan* pl, int F[3], int* fused) {
    for (int a = 0; a < 3; ++a) F[a] = pl ? pl->F[a] : 0;
    if (fused) *fused = pl ? pl->fused : 0;
}

static void fft_stages(FftArgs& f, const FftPlan* pl, int a) {
    int s0 = 1;
    for (int i = 0; i < FFT_MAX_ST; ++i) {
        f.rad[a][i] = pl->rad[a][i];
        if (i >= pl->nst[a]) continue;
        f.mg[a][2 * i] = fft_magic(pl->F[a] / pl->rad[a][i]);
        f.mg[a][2 * i + 1] = fft_magic(s0);
        s0 *= pl->rad[a][i];
    }
}

// The convolution for k-points kofs .. kofs + nk - 1 (descriptors td[kofs ..])
// over ncol columns; vmode 0 multiplies by v (+ s vd when
// use_vd), vmode 1 by s vd alone.  Five launches.
static int launch_fft_any(const FftPlan* pl, int fused, const ToepDesc* td, int kofs, int nk, int ncol, int vmode,
                          int use_vd, const double* s, cudaStream_t st, int tune = 0) {
    FftArgs f = {};
    f.tune = tune;
    f.F1 = pl->F[0];
    f.F2 = pl->F[1];
    f.F3 = pl->F[2];
    for (int a = 0; a < 3; ++a) {
        f.nst[a] = pl->nst[a];
        fft_stages(f, pl, a);
        f.lpb[a] = fft_lpb(pl->F[a]);
        f.w[a] = pl->fx ? (const void*)pl->wq[a] : pl->prec == 0 ? (const void*)pl->w64[a] : (const void*)pl->w32[a];
    }
    f.fk = pl->d_fk + kofs;
    f.td = td + kofs;
    f.b3 = pl->b3;
    f.b2 = pl->b2;
    f.b3_col = (size_t)pl->max_lines * f.F3;
    f.b2_col = (size_t)pl->max_planes * f.F2 * f.F3;
    f.ncol = ncol;
    f.vmode = vmode;
    f.use_vd = use_vd;
    f.v = pl->prec == 0 ? (const void*)pl->v64 : (const void*)pl->v32;
    f.vd = pl->prec == 0 ? (const void*)pl->vd64 : (const void*)pl->vd32;
    f.s = s;
    const int ch1 = (f.F3 + f.lpb[1] - 1) / f.lpb[1], ch0 = (f.F3 + f.lpb[0] - 1) / f.lpb[0];
    const dim3 ga((pl->max_lines + f.lpb[2] - 1) / f.lpb[2], ncol, nk);
    const dim3 gb(pl->max_planes * ch1, ncol, nk);
    const dim3 gc(f.F2 * ch0, ncol, nk);
    if (pl->fx) {
        const int own = vmode != 0 || use_vd;
        if (own) k_fx_v<<<f.F2 * ch0, FFT_THREADS, 0, st>>>(f, pl->vq[1], pl->vqe[1]);
        f.vq = pl->vq[own];
        f.vqe = pl->vqe[own];
        f.ma = pl->ma;
        f.mb = pl->mb;
        f.mc = pl->mc;
        f.lines_max = pl->max_lines;
        f.planes_max = pl->max_planes;
        for (int a = 0; a < 3; ++a) f.qb[a] = fx_bits(pl->F[a]);
        if (fused) {
            const dim3 gp(pl->max_planes, ncol, nk);
            const size_t psm = fft_plane_smem(f.F2, f.F3, sizeof(zq));
            k_fx_plane<<<gp, FFT_PTHREADS, psm, st>>>(f, 0);
            k_fx_c<<<gc, FFT_THREADS, fft_smem(f.F1, sizeof(zq)), st>>>(f);
            k_fx_plane<<<gp, FFT_PTHREADS, psm, st>>>(f, 1);
            return 3 + own;
        }
        k_fx_a<<<ga, FFT_THREADS, fft_smem(f.F3, sizeof(zq)), st>>>(f);
        k_fx_bd<<<gb, FFT_THREADS, fft_smem(f.F2, sizeof(zq)), st>>>(f, 0);
        k_fx_c<<<gc, FFT_THREADS, fft_smem(f.F1, sizeof(zq)), st>>>(f);
        k_fx_bd<<<gb, FFT_THREADS, fft_smem(f.F2, sizeof(zq)), st>>>(f, 1);
        k_fx_e<<<ga, FFT_THREADS, fft_smem(f.F3, sizeof(zq)), st>>>(f);
        return 5 + own;
    }
    if (fused) {
        const dim3 gp(pl->max_planes, ncol, nk);
        if (pl->prec == 0) {
            const size_t psm = fft_plane_smem(f.F2, f.F3, sizeof(zd));
            k_fft_plane<zd><<<gp, FFT_PTHREADS, psm, st>>>(f, 0);
            k_fft_c<zd><<<gc, FFT_THREADS, fft_smem(f.F1, sizeof(zd)), st>>>(f);
            k_fft_plane<zd><<<gp, FFT_PTHREADS, psm, st>>>(f, 1);
        } else {
            const size_t psm = fft_plane_smem(f.F2, f.F3, sizeof(zf));
            k_fft_plane<zf><<<gp, FFT_PTHREADS, psm, st>>>(f, 0);
            k_fft_c<zf><<<gc, FFT_THREADS, fft_smem(f.F1, sizeof(zf)), st>>>(f);
            k_fft_plane<zf><<<gp, FFT_PTHREADS, psm, st>>>(f, 1);
        }
        return 3;
    }
    if (pl->prec == 0) {
        k_fft_a<zd><<<ga, FFT_THREADS, fft_smem(f.F3, sizeof(zd)), st>>>(f);
        k_fft_bd<zd><<<gb, FFT_THREADS, fft_smem(f.F2, sizeof(zd)), st>>>(f, 0);
        k_fft_c<zd><<<gc, FFT_THREADS, fft_smem(f.F1, sizeof(zd)), st>>>(f);
        k_fft_bd<zd><<<gb, FFT_THREADS, fft_smem(f.F2, sizeof(zd)), st>>>(f, 1);
        k_fft_e<zd><<<ga, FFT_THREADS, fft_smem(f.F3, sizeof(zd)), st>>>(f);
    } else {
        k_fft_a<zf><<<ga, FFT_THREADS, fft_smem(f.F3, sizeof(zf)), st>>>(f);
        k_fft_bd<zf><<<gb, FFT_THREADS, fft_smem(f.F2, sizeof(zf)), st>>>(f, 0);
        k_fft_c<zf><<<gc, FFT_THREADS, fft_smem(f.F1, sizeof(zf)), st>>>(f);
        k_fft_bd<zf><<<gb, FFT_THREADS, fft_smem(f.F2, sizeof(zf)), st>>>(f, 1);
        k_fft_e<zf><<<ga, FFT_THREADS, fft_smem(f.F3, sizeof(zf)), st>>>(f);
    }
    return 5;
}

int launch_fft_conv(const FftPlan* pl, const ToepDesc* td, int kofs, int nk, int ncol, int vmode, int use_vd,
                    const double* s, cudaStream_t st) {
    return launch_fft_any(pl, pl->fused, td, kofs, nk, ncol, vmode, use_vd, s, st);
}

// Set-up autotuner: times the five-launch and the plane-fused three-launch
// sets on the operator's own descriptors (three runs each after one warm-up)
// and keeps the faster.
// RTTDDFT_FFT_LAUNCHES=5 or =3 in the environment fixes the choice (both sets
// compute the same sums; the tests run each).
int fft_tune(FftPlan* pl, const ToepDesc* td, int ncol, cudaStream_t st) {
    const int elt = pl->prec == 0 ? (int)sizeof(zd) : (int)sizeof(zf);
    if (fft_plane_smem(pl->F[1], pl->F[2], elt) > FFT_PLANE_SMEM_MAX) {
        pl->fused = 0;
        return 0;
    }
    const char* force = getenv("RTTDDFT_FFT_LAUNCHES");
    if (force && (force[0] == '3' || force[0] == '5') && force[1] == 0) {
        pl->fused = force[0] == '3' ? 1 : 0;
        return 0;
    }
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return -1;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return -1;
    }
    float ms[2] = {0.f, 0.f};
    for (int v = 0; v < 2; ++v) {
        launch_fft_any(pl, v, td, 0, pl->nk, ncol, 0, 0, nullptr, st, 1);
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; ++r) launch_fft_any(pl, v, td, 0, pl->nk, ncol, 0, 0, nullptr, st, 1);
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        cudaEventElapsedTime(&ms[v], e0, e1);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    pl->ms_split = ms[0] / 3;
    pl->ms_fused = ms[1] / 3;
    pl->fused = ms[1] < ms[0] ? 1 : 0;
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------- Hartree feedback
// launch arguments of the FP64 density passes
static FftArgs fft_args64(const FftPlan* pl, const ToepDesc* td, int kofs, int ncol) {
    FftArgs f;
    f.F1 = pl->F[0];
    f.F2 = pl->F[1];
    f.F3 = pl->F[2];
    for (int a = 0; a < 3; ++a) {
        f.nst[a] = pl->nst[a];
        fft_stages(f, pl, a);
        f.lpb[a] = fft_lpb(pl->F[a]);
        f.w[a] = (const void*)pl->w64[a];
    }
    f.fk = pl->d_fk + kofs;
    f.td = td + kofs;
    f.b3 = pl->prec == 0 ? pl->b3 : (void*)pl->b3d;
    f.b2 = pl->prec == 0 ? pl->b2 : (void*)pl->b2d;
    f.b3_col = (size_t)pl->max_lines * f.F3;
    f.b2_col = (size_t)pl->max_planes * f.F2 * f.F3;
    f.ncol = ncol;
    f.vmode = 0;
    f.use_vd = 0;
    f.v = nullptr;
    f.vd = nullptr;
    f.s = nullptr;
    return f;
}

// Set up the density feedback: grids for n, its starting value and the
// potential change; recip rows are the reciprocal vectors b_i (1/bohr).
int fft_hartree_init(FftPlan* pl, const double recip[9], const int vt_dim[3], double omega, double bound, int ns,
                     cudaStream_t st, std::string* why) {
    const size_t n3 = (size_t)pl->F[0] * pl->F[1] * pl->F[2];
    bool ok = true;
    if (cudaMalloc((void**)&pl->rho, n3 * sizeof(zd)) != cudaSuccess ||
        cudaMalloc((void**)&pl->rho0, n3 * sizeof(zd)) != cudaSuccess ||
        cudaMalloc((void**)&pl->l1, sizeof(double)) != cudaSuccess)
        ok = false;
    if (ok && !pl->vd64) ok = cudaMalloc((void**)&pl->vd64, n3 * sizeof(zd)) == cudaSuccess;
    if (ok && pl->prec != 0 && !pl->vd32) ok = cudaMalloc((void**)&pl->vd32, n3 * sizeof(zf)) == cudaSuccess;
    if (ok && pl->prec != 0) {
        // FP64 buffers for the N_s columns of the density
        const size_t c3 = (size_t)pl->max_lines * pl->F[2], c2 = (size_t)pl->max_planes * pl->F[1] * pl->F[2];
        ok = cudaMalloc((void**)&pl->b3d, std::max<size_t>((size_t)pl->nk * ns * c3, 1) * sizeof(zd)) == cudaSuccess &&
             cudaMalloc((void**)&pl->b2d, std::max<size_t>((size_t)pl->nk * ns * c2, 1) * sizeof(zd)) == cudaSuccess;
    }
    if (!ok) {
        if (why) *why = "Hartree feedback: device allocation failed";
        return RTTDDFT_ERR_OOM;
    }
    cudaMemsetAsync(pl->l1, 0, sizeof(double), st);
    cudaMemsetAsync(pl->vd64, 0, n3 * sizeof(zd), st);
    if (pl->vd32) cudaMemsetAsync(pl->vd32, 0, n3 * sizeof(zf), st);
    const size_t psm = fft_plane_smem(pl->F[1], pl->F[2], sizeof(zd));
    pl->fused_d = (pl->prec == 0) ? pl->fused : (psm <= FFT_PLANE_SMEM_MAX ? 1 : 0);
    for (int i = 0; i < 9; ++i) pl->recip[i] = recip[i];
    for (int a = 0; a < 3; ++a) pl->e[a] = (vt_dim[a] - 1) / 2;
    pl->omega = omega;
    pl->bound = bound;
    pl->hartree = 1;
    const int mx = (int)fft_smem(std::max(pl->F[0], std::max(pl->F[1], pl->F[2])), (int)sizeof(zd));
    raise_smem((const void*)k_fft_density<zd>, mx);
    raise_smem((const void*)k_fft_full<zd>, mx);
    raise_smem((const void*)k_fft_a<zd>, mx);
    raise_smem((const void*)k_fft_bd<zd>, mx);
    if (pl->fused_d) raise_smem((const void*)k_fft_plane<zd>, (int)psm);
    if (cudaGetLastError() != cudaSuccess) {
        if (why) *why = "Hartree feedback: set-up failed";
        return RTTDDFT_ERR_CUDA;
    }
    return 0;
}

template <typename C>
static int density_launches(const FftPlan* pl, const FftArgs& f, int nk, const double* occ, const double* wk, C* rho,
                            cudaStream_t st) {
    const int ch0 = (f.F3 + f.lpb[0] - 1) / f.lpb[0], ch1 = (f.F3 + f.lpb[1] - 1) / f.lpb[1];
    int nl = 0;
    // the planes of every (k, state) column after the inverse transforms of axes 3 and 2
    if (pl->fused_d) {
        k_fft_plane<C><<<dim3(pl->max_planes, f.ncol, nk), FFT_PTHREADS, fft_plane_smem(f.F2, f.F3, sizeof(C)), st>>>(f, 0);
        ++nl;
    } else {
        k_fft_a<C><<<dim3((pl->max_lines + f.lpb[2] - 1) / f.lpb[2], f.ncol, nk), FFT_THREADS,
                     fft_smem(f.F3, sizeof(C)), st>>>(f);
        k_fft_bd<C><<<dim3(pl->max_planes * ch1, f.ncol, nk), FFT_THREADS, fft_smem(f.F2, sizeof(C)), st>>>(f, 0);
        nl += 2;
    }
    k_fft_density<C><<<f.F2 * ch0, FFT_THREADS, fft_smem(f.F1, sizeof(C)), st>>>(f, nk, occ, wk, 1.0 / pl->omega, rho);
    ++nl;
    // N(g) = sum_r n(r) e^{-2 pi i g.r/F}
    const int ga[3] = {f.F2 * ch0, f.F1 * ch1, (f.F1 * f.F2 + f.lpb[2] - 1) / f.lpb[2]};
    for (int a = 2; a >= 0; --a) {
        const int L = pl->F[a];
        k_fft_full<C><<<ga[a], FFT_THREADS, fft_smem(L, sizeof(C)), st>>>(f, rho, a, 0);
        ++nl;
    }
    return nl;
}

// The density of the current C (td: per k {C, .}) transformed to G space; with
// reference = 1 it becomes the starting density n(0).  Returns the launches.
int launch_fft_density(const FftPlan* pl, const ToepDesc* td, int nk, int ns, const double* occ, const double* wk,
                       int reference, cudaStream_t st) {
    const FftArgs f = fft_args64(pl, td, 0, ns);
    const size_t n3 = (size_t)pl->F[0] * pl->F[1] * pl->F[2];
    const int nl = density_launches<zd>(pl, f, nk, occ, wk, pl->rho, st);
    if (reference) cudaMemcpyAsync(pl->rho0, pl->rho, n3 * sizeof(zd), cudaMemcpyDeviceToDevice, st);
    return nl;
}

// After a step: the density of C_{k+1}, its Hartree potential change against
// n(0) on the table box, and that potential's grid image for the next step's
// operator and potential-change rebuild.  Returns the launches.
int launch_fft_hartree(const FftPlan* pl, const ToepDesc* td, int nk, int ns, const double* occ, const double* wk,
                       int* flag, cudaStream_t st) {
    int nl = launch_fft_density(pl, td, nk, ns, occ, wk, 0, st);
    const FftArgs f = fft_args64(pl, td, 0, ns);
    const double inv_f3 = 1.0 / ((double)pl->F[0] * pl->F[1] * pl->F[2]);
    const double* b = pl->recip;
    const int ch0 = (f.F3 + f.lpb[0] - 1) / f.lpb[0], ch1 = (f.F3 + f.lpb[1] - 1) / f.lpb[1];
    const int ga[3] = {f.F2 * ch0, f.F1 * ch1, (f.F1 * f.F2 + f.lpb[2] - 1) / f.lpb[2]};
    k_hartree<zd><<<152, 256, 0, st>>>(pl->rho, pl->rho0, pl->vd64, f.F1, f.F2, f.F3, pl->e[0], pl->e[1], pl->e[2],
                                       b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7], b[8], inv_f3, pl->l1);
    for (int a = 0; a < 3; ++a)
        k_fft_full<zd><<<ga[a], FFT_THREADS, fft_smem(pl->F[a], sizeof(zd)), st>>>(f, pl->vd64, a, 1);
    if (pl->prec != 0) {
        // the FP32 operator reads its copy of the grid image
        const size_t n3 = (size_t)f.F1 * f.F2 * f.F3;
        k_fft_to32<<<(int)std::min<size_t>((n3 + 255) / 256, 4096), 256, 0, st>>>(pl->vd64, pl->vd32, n3);
        ++nl;
    }
    k_hartree_check<<<1, 1, 0, st>>>(pl->l1, pl->bound, flag);
    return nl + 5;
}
