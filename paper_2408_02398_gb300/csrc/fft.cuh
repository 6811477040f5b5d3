// fft.cuh -- batched 1-D FFT passes over one axis of a 3-D array.
//
// Each CTA stages a tile of W lines of length L in shared memory (W a power
// of two), runs a mixed-radix Stockham FFT (radices 2, 3, 4, 5, 7, 8; the
// autosort variant so no bit reversal is needed) through two ping-pong
// buffers, and writes the tile back. Tiles of a strided axis are W lines
// that are adjacent in memory, so every one of the L rows of the tile is a
// contiguous run of W complex elements (coalesced); tiles of the contiguous
// axis are W whole lines. Loads go through a "prologue" functor and stores
// through a "store" functor, which is how the pointwise spectrum products,
// the real<->complex packing and the normalisation epilogues are fused into
// the passes.
//
// Index arithmetic is what bounds these kernels: the length is a run-time
// value, and with lines stored one after another (element j of line w at
// w ld + j) every load, butterfly and store divided by L, L / radix or W at
// run time, 320 issued instructions per complex element and pass at 270 and
// 315 against 56 in the register kernels. So the tile is kept transposed,
// element j of line w at j S + w: the lanes of a warp take the W lines of a
// butterfly first (shifts and masks; their twiddles are one broadcast read),
// a strided tile is copied without any index change (S = W), and the one
// quotient left per butterfly is a multiplication by a reciprocal from the
// plan. Contiguous tiles use S = W + 1 (odd), which keeps their copies
// along a line free of bank conflicts. Same schedules and arithmetic, the
// same results; ttm_correlate of 126 x 270 x 315 (n = 4, FP64 local sums)
// went from 8.24 to 6.64 ms, a batch of six sub-tomograms of 96 .. 176 per
// axis x two templates from 12.90 to 8.65 ms.
//
// Direction DIR = -1 computes sum_j x_j exp(-2 pi i jk/L) (forward),
// DIR = +1 the unnormalised inverse.
#pragma once

#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ttm_common.cuh"
#include "df64.cuh"

namespace ttm {

// Complex values as stored in HBM: the pass precision itself, or FP16 /
// BF16 pairs that are widened to FP32 on load (the arithmetic stays FP32).
__device__ __forceinline__ float2 load_cx(const float2& v) { return v; }
__device__ __forceinline__ double2 load_cx(const double2& v) { return v; }
__device__ __forceinline__ dcx load_cx(const dcx& v) { return v; }
__device__ __forceinline__ float2 load_cx(const __half2& v) { return __half22float2(v); }
__device__ __forceinline__ float2 load_cx(const __nv_bfloat162& v) { return __bfloat1622float2(v); }
__device__ __forceinline__ void store_cx(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void store_cx(__half2* p, float2 v) { *p = __float22half2_rn(v); }
__device__ __forceinline__ void store_cx(__nv_bfloat162* p, float2 v) { *p = __float22bfloat162_rn(v); }

constexpr int kMaxStages = 24;

// A transform length with its radix schedule and its twiddle table
// tw[m] = exp(-2 pi i m / L), m in [0, L), in the pass precision.
struct LenPlan {
    int L;
    int nst;
    int rad[kMaxStages];
    const void* tw;
    uint32_t mag[kMaxStages];  // ceil(2^32 / product of the radices before a stage), set by with_magic
    int num_sms = 1;  // SMs of the device that runs the passes
    int tile_w = 0;   // lines per CTA of the shared-memory passes (0: default)
    int no_reg = 0;   // 1: use the shared-memory passes even where register kernels exist
};

// sin/cos of 2 pi m / R for the odd radices (mathematical constants)
struct OddRadixConst {
    static constexpr double c3 = -0.5;
    static constexpr double s3 = 0.86602540378443864676372317075294;
    static constexpr double c5_1 = 0.30901699437494742410229341718282;
    static constexpr double s5_1 = 0.95105651629515357211643933337938;
    static constexpr double c5_2 = -0.80901699437494742410229341718282;
    static constexpr double s5_2 = 0.58778525229247312916870595463907;
    static constexpr double c7_1 = 0.62348980185873353052500488400424;
    static constexpr double s7_1 = 0.78183148246802980870844452667406;
    static constexpr double c7_2 = -0.22252093395631440428890256449679;
    static constexpr double s7_2 = 0.97492791218182360701813168299393;
    static constexpr double c7_3 = -0.90096886790241912623610231950745;
    static constexpr double s7_3 = 0.43388373911755812047576833284836;
    static constexpr double sqrt_half = 0.70710678118654752440084436210485;
};

// ---------------------------------------------------------- butterflies --

// Sum and difference of two complex values: for FP32 one packed instruction
// for both parts (a - b as a fused multiply-add by -1, the same rounding),
// which halves the issue slots of a butterfly's additions. PK = false takes
// the scalar instructions, the same results: operands have to lie in aligned
// register pairs, and where a pass forms its values part by part the moves
// into pairs can cost more (fs_c2r_packed).
template <bool PK, typename C> __device__ __forceinline__ C padd(C a, C b)
{
    if constexpr (PK && std::is_same<C, float2>::value) return __fadd2_rn(a, b);
    else return cadd(a, b);
}
template <bool PK, typename C> __device__ __forceinline__ C psub(C a, C b)
{
    if constexpr (PK && std::is_same<C, float2>::value) return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
    else return csub(a, b);
}

template <int DIR, bool PK = true, typename C> __device__ __forceinline__ void dft2(C* v)
{
    C a = v[0], b = v[1];
    v[0] = padd<PK>(a, b);
    v[1] = psub<PK>(a, b);
}

template <int DIR, bool PK = true, typename C> __device__ __forceinline__ void dft4(C& a0, C& a1, C& a2, C& a3)
{
    C t0 = padd<PK>(a0, a2), t1 = psub<PK>(a0, a2);
    C t2 = padd<PK>(a1, a3), t3 = cmul_diri<DIR>(psub<PK>(a1, a3));
    a0 = padd<PK>(t0, t2);
    a2 = psub<PK>(t0, t2);
    a1 = cadd(t1, t3);
    a3 = csub(t1, t3);
}

// x * (h + DIR h i) = h (x.x - DIR x.y) + i h (x.y + DIR x.x): two adds and
// two products instead of a full complex product
template <int DIR, typename R> __device__ __forceinline__ cx<R> mul_w8_1(cx<R> x, R h)
{
    if constexpr (std::is_same<R, df64>::value) return mul_w8_df<DIR>(x, h, false);
    else return DIR < 0 ? mk<R>((x.x + x.y) * h, (x.y - x.x) * h) : mk<R>((x.x - x.y) * h, (x.y + x.x) * h);
}
// x * (-h + DIR h i) = h (-x.x - DIR x.y) + i h (DIR x.x - x.y)
template <int DIR, typename R> __device__ __forceinline__ cx<R> mul_w8_3(cx<R> x, R h)
{
    if constexpr (std::is_same<R, df64>::value) return mul_w8_df<DIR>(x, h, true);
    else return DIR < 0 ? mk<R>((x.y - x.x) * h, (-x.x - x.y) * h) : mk<R>((-x.x - x.y) * h, (x.x - x.y) * h);
}

template <int DIR, typename R, bool PK = true> __device__ __forceinline__ void dft8(cx<R>* v)
{
    cx<R> e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    cx<R> o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<DIR, PK>(e0, e1, e2, e3);
    dft4<DIR, PK>(o0, o1, o2, o3);
    const R h = (R)OddRadixConst::sqrt_half;
    // w8^1 = h(1 + DIR i), w8^2 = DIR i, w8^3 = h(-1 + DIR i)
    if constexpr (PK && std::is_same<R, float>::value) {
        // the products by h are fused into the additions that take them
        const float2 p = DIR < 0 ? make_float2(o1.x + o1.y, o1.y - o1.x) : make_float2(o1.x - o1.y, o1.y + o1.x);
        const float2 q = DIR < 0 ? make_float2(o3.y - o3.x, -o3.x - o3.y) : make_float2(-o3.x - o3.y, o3.x - o3.y);
        const float2 hh = make_float2(h, h), mh = make_float2(-h, -h);
        const float2 t2 = cmul_diri<DIR>(o2);
        v[0] = padd<PK>(e0, o0); v[4] = psub<PK>(e0, o0);
        v[1] = __ffma2_rn(p, hh, e1); v[5] = __ffma2_rn(p, mh, e1);
        v[2] = cadd(e2, t2); v[6] = csub(e2, t2);
        v[3] = __ffma2_rn(q, hh, e3); v[7] = __ffma2_rn(q, mh, e3);
        return;
    }
    cx<R> t1 = mul_w8_1<DIR, R>(o1, h);
    cx<R> t2 = cmul_diri<DIR>(o2);
    cx<R> t3 = mul_w8_3<DIR, R>(o3, h);
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, t1); v[5] = csub(e1, t1);
    v[2] = cadd(e2, t2); v[6] = csub(e2, t2);
    v[3] = cadd(e3, t3); v[7] = csub(e3, t3);
}

// Odd radices in their symmetric form: with t_r = x_r + x_{R-r} and
// d_r = x_r - x_{R-r} (r = 1..(R-1)/2),
//   X_0 = x_0 + sum_r t_r,
//   X_k, X_{R-k} = A_k +- DIR i B_k,  A_k = x_0 + sum_r t_r cos(2 pi rk/R),
//                                      B_k = sum_r d_r sin(2 pi rk/R),
// so every product is a real constant times a complex value and each
// cosine / sine term is shared by the output pair (k, R - k).
template <int DIR, typename R> __device__ __forceinline__ cx<R> pm_diri(cx<R> a, cx<R> b, bool plus)
{
    // a + DIR i b (plus) or a - DIR i b
    const cx<R> ib = cmul_diri<DIR>(b);
    return plus ? cadd(a, ib) : csub(a, ib);
}

template <int DIR, typename R> __device__ __forceinline__ void dft3(cx<R>* v)
{
    const cx<R> t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const cx<R> x0 = v[0];
    v[0] = cadd(x0, t);
    const cx<R> A = csub(x0, cscale(t, (R)0.5));
    const cx<R> B = cscale(d, (R)OddRadixConst::s3);
    v[1] = pm_diri<DIR, R>(A, B, true);
    v[2] = pm_diri<DIR, R>(A, B, false);
}

template <int DIR, typename R> __device__ __forceinline__ void dft5(cx<R>* v)
{
    const R c1 = (R)OddRadixConst::c5_1, c2 = (R)OddRadixConst::c5_2;
    const R s1 = (R)OddRadixConst::s5_1, s2 = (R)OddRadixConst::s5_2;
    const cx<R> x0 = v[0];
    const cx<R> t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const cx<R> d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
    v[0] = cadd(x0, cadd(t1, t2));
    // cos 4 pi/5 = c2, cos 8 pi/5 = c1; sin 8 pi/5 = -s1
    const cx<R> A1 = cadd(x0, cadd(cscale(t1, c1), cscale(t2, c2)));
    const cx<R> A2 = cadd(x0, cadd(cscale(t1, c2), cscale(t2, c1)));
    const cx<R> B1 = cadd(cscale(d1, s1), cscale(d2, s2));
    const cx<R> B2 = csub(cscale(d1, s2), cscale(d2, s1));
    v[1] = pm_diri<DIR, R>(A1, B1, true);
    v[4] = pm_diri<DIR, R>(A1, B1, false);
    v[2] = pm_diri<DIR, R>(A2, B2, true);
    v[3] = pm_diri<DIR, R>(A2, B2, false);
}

template <int DIR, typename R> __device__ __forceinline__ void dft7(cx<R>* v)
{
    const R c1 = (R)OddRadixConst::c7_1, c2 = (R)OddRadixConst::c7_2, c3 = (R)OddRadixConst::c7_3;
    const R s1 = (R)OddRadixConst::s7_1, s2 = (R)OddRadixConst::s7_2, s3 = (R)OddRadixConst::s7_3;
    const cx<R> x0 = v[0];
    const cx<R> t1 = cadd(v[1], v[6]), t2 = cadd(v[2], v[5]), t3 = cadd(v[3], v[4]);
    const cx<R> d1 = csub(v[1], v[6]), d2 = csub(v[2], v[5]), d3 = csub(v[3], v[4]);
    v[0] = cadd(x0, cadd(t1, cadd(t2, t3)));
    // angles 2 pi rk / 7 reduced: (r k mod 7) in {1,2,3} keeps its sine, in
    // {4,5,6} takes minus the sine of 7 - (r k mod 7)
    const cx<R> A1 = cadd(x0, cadd(cscale(t1, c1), cadd(cscale(t2, c2), cscale(t3, c3))));
    const cx<R> A2 = cadd(x0, cadd(cscale(t1, c2), cadd(cscale(t2, c3), cscale(t3, c1))));
    const cx<R> A3 = cadd(x0, cadd(cscale(t1, c3), cadd(cscale(t2, c1), cscale(t3, c2))));
    const cx<R> B1 = cadd(cscale(d1, s1), cadd(cscale(d2, s2), cscale(d3, s3)));
    const cx<R> B2 = csub(cscale(d1, s2), cadd(cscale(d2, s3), cscale(d3, s1)));
    const cx<R> B3 = cadd(csub(cscale(d1, s3), cscale(d2, s1)), cscale(d3, s2));
    v[1] = pm_diri<DIR, R>(A1, B1, true);
    v[6] = pm_diri<DIR, R>(A1, B1, false);
    v[2] = pm_diri<DIR, R>(A2, B2, true);
    v[5] = pm_diri<DIR, R>(A2, B2, false);
    v[3] = pm_diri<DIR, R>(A3, B3, true);
    v[4] = pm_diri<DIR, R>(A3, B3, false);
}

template <int RAD, int DIR, typename R, bool PK = true> __device__ __forceinline__ void dft(cx<R>* v)
{
    if constexpr (RAD == 2) dft2<DIR, PK>(v);
    else if constexpr (RAD == 3) dft3<DIR, R>(v);
    else if constexpr (RAD == 4) dft4<DIR, PK>(v[0], v[1], v[2], v[3]);
    else if constexpr (RAD == 5) dft5<DIR, R>(v);
    else if constexpr (RAD == 7) dft7<DIR, R>(v);
    else dft8<DIR, R, PK>(v);
    // double-float butterflies add without renormalising (df64.cuh): once
    // per output here
    if constexpr (std::is_same<R, df64>::value) {
#pragma unroll
        for (int r = 0; r < RAD; r++) v[r] = renormalise(v[r]);
    }
}

// ----------------------------------------------------------- stages --

// One Stockham stage of radix RAD on the W = 2^LW lines of a tile (element j
// of line w at j S + w) from `in` to `out`. Ns = product of the radices of
// the earlier stages, mag = ceil(2^32 / Ns) (j < 2^16, so the high word of
// j mag is j / Ns exactly), step = L / (Ns RAD).
template <int RAD, int DIR, typename R>
__device__ __forceinline__ void stockham_stage(const cx<R>* __restrict__ in, cx<R>* __restrict__ out,
                                               int L, int S, int LW, int Ns, uint32_t mag, int step,
                                               const cx<R>* __restrict__ tw)
{
    const int nb = L / RAD;
    const int w = threadIdx.x & ((1 << LW) - 1);
    for (int j = threadIdx.x >> LW; j < nb; j += blockDim.x >> LW) {
        const int k = Ns > 1 ? j - (int)__umulhi((uint32_t)j, mag) * Ns : 0;
        const cx<R>* src = in + j * S + w;
        cx<R> v[RAD];
#pragma unroll
        for (int r = 0; r < RAD; r++) v[r] = src[r * nb * S];
        if (Ns > 1) {
            const cx<R>* tk = tw;
#pragma unroll
            for (int r = 1; r < RAD; r++) {
                tk += k * step;
                cx<R> t_ = *tk;
                if (DIR > 0) t_ = cconj(t_);
                v[r] = cmul(v[r], t_);
            }
        }
        dft<RAD, DIR, R>(v);
        cx<R>* dst = out + ((j - k) * RAD + k) * S + w;
#pragma unroll
        for (int r = 0; r < RAD; r++) dst[r * Ns * S] = v[r];
    }
}

// Full transform of the 2^LW lines in a (scratch b); returns the buffer that
// holds the result. Ends with __syncthreads().
template <int DIR, typename R>
__device__ cx<R>* smem_fft(cx<R>* a, cx<R>* b, int S, int LW, const LenPlan& pl, const cx<R>* tw)
{
    int Ns = 1, step = pl.L;
    const int L = pl.L;
    for (int s = 0; s < pl.nst; s++) {
        const uint32_t mag = pl.mag[s];
        switch (pl.rad[s]) {
            case 2: step /= 2; stockham_stage<2, DIR, R>(a, b, L, S, LW, Ns, mag, step, tw); break;
            case 3: step /= 3; stockham_stage<3, DIR, R>(a, b, L, S, LW, Ns, mag, step, tw); break;
            case 4: step /= 4; stockham_stage<4, DIR, R>(a, b, L, S, LW, Ns, mag, step, tw); break;
            case 5: step /= 5; stockham_stage<5, DIR, R>(a, b, L, S, LW, Ns, mag, step, tw); break;
            case 7: step /= 7; stockham_stage<7, DIR, R>(a, b, L, S, LW, Ns, mag, step, tw); break;
            default: step /= 8; stockham_stage<8, DIR, R>(a, b, L, S, LW, Ns, mag, step, tw); break;
        }
        Ns *= pl.rad[s];
        __syncthreads();
        cx<R>* t = a; a = b; b = t;
    }
    return a;
}

template <typename R>
__device__ __forceinline__ void load_twiddles(cx<R>* tws, const LenPlan& pl)
{
    const cx<R>* g = reinterpret_cast<const cx<R>*>(pl.tw);
    for (int i = threadIdx.x; i < pl.L; i += blockDim.x) tws[i] = g[i];
}

// Stages n tile elements into shared memory with kLoadBatch global loads
// per thread issued before any of their shared-memory stores, so that a
// thread has that many loads in flight instead of waiting on each in turn:
// get(idx) loads element idx, put(idx, v) stores it into the tile.
constexpr int kLoadBatch = 8;
template <typename T, class Get, class Put>
__device__ __forceinline__ void stage_tile(int n, Get get, Put put)
{
    for (int base = threadIdx.x; base < n; base += kLoadBatch * blockDim.x) {
        T v[kLoadBatch];
#pragma unroll
        for (int u = 0; u < kLoadBatch; u++) {
            const int idx = base + u * (int)blockDim.x;
            if (idx < n) v[u] = get(idx);
        }
#pragma unroll
        for (int u = 0; u < kLoadBatch; u++) {
            const int idx = base + u * (int)blockDim.x;
            if (idx < n) put(idx, v[u]);
        }
    }
}

// ------------------------------------------------------------ functors --

template <typename R> struct ProIdentity {
    __device__ __forceinline__ cx<R> operator()(cx<R> v, int64_t, int64_t, int) const { return v; }
};

template <typename R> struct StoreTo {
    cx<R>* out;
    int64_t os, s;  // outer stride, element stride (inner stride is 1)
    __device__ __forceinline__ void operator()(cx<R> v, int64_t o, int64_t i, int j) const
    {
        out[o * os + i + (int64_t)j * s] = v;
    }
};

// Geometry of a strided axis: line (o, i) has elements o*os + i + j*s,
// j < L; i < inner are adjacent lines, o < outer.
struct StridedAxis {
    int64_t inner, outer, os, s;
};

// ------------------------------------------------------------ kernels --

constexpr int kSmemFftThreads = 256;

// Stages elements x0, x0 + G, ... < n of one line with kLoadBatch global
// loads issued before any of their shared-memory stores (see stage_tile)
template <typename T, class Get, class Put>
__device__ __forceinline__ void stage_line(int x0, int G, int n, Get get, Put put)
{
    for (int base = x0; base < n; base += kLoadBatch * G) {
        T v[kLoadBatch];
#pragma unroll
        for (int u = 0; u < kLoadBatch; u++)
            if (base + u * G < n) v[u] = get(base + u * G);
#pragma unroll
        for (int u = 0; u < kLoadBatch; u++)
            if (base + u * G < n) put(base + u * G, v[u]);
    }
}

// Shared memory: 2 * L * W + L complex elements (W = 2^LW lines, S = W).
template <typename R, int DIR, class Pro, class Store, typename In = cx<R>>
__global__ void __launch_bounds__(kSmemFftThreads) k_fft_strided(const In* __restrict__ in, StridedAxis ax, LenPlan pl,
                                                     int LW, Pro pro, Store store)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = pl.L, W = 1 << LW;
    cx<R>* bufa = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* bufb = bufa + L * W;
    cx<R>* tws = bufb + L * W;
    const int64_t tiles_per_outer = (ax.inner + W - 1) >> LW;
    const int64_t o = blockIdx.x / tiles_per_outer;
    const int64_t i = ((blockIdx.x - o * tiles_per_outer) << LW) + (threadIdx.x & (W - 1));
    const bool act = i < ax.inner;
    load_twiddles<R>(tws, pl);
    const In* src = in + o * ax.os + i;
    stage_tile<cx<R>>(
        W * L,
        [&](int idx) {
            const int j = idx >> LW;
            return act ? pro(load_cx(src[(int64_t)j * ax.s]), o, i, j) : mk<R>(0, 0);
        },
        [&](int idx, cx<R> v) { bufa[idx] = v; });
    __syncthreads();
    cx<R>* res = smem_fft<DIR, R>(bufa, bufb, W, LW, pl, tws);
    if (act)
        for (int idx = threadIdx.x; idx < W * L; idx += kSmemFftThreads) store(res[idx], o, i, idx >> LW);
}

// Contiguous lines: line l has elements l*L + j (l < nlines). The functors
// get (o = l, i = 0, j). 256 / W consecutive threads work on one line.
template <typename R, int DIR, class Pro, class Store>
__global__ void __launch_bounds__(kSmemFftThreads) k_fft_contig(const cx<R>* __restrict__ in, int64_t nlines, LenPlan pl,
                                                    int LW, int S, Pro pro, Store store)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = pl.L, G = kSmemFftThreads >> LW;
    cx<R>* bufa = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* bufb = bufa + L * S;
    cx<R>* tws = bufb + L * S;
    const int w = threadIdx.x / G, x0 = threadIdx.x & (G - 1);
    const int64_t l = ((int64_t)blockIdx.x << LW) + w;
    const bool act = l < nlines;
    load_twiddles<R>(tws, pl);
    stage_line<cx<R>>(
        x0, G, L, [&](int j) { return act ? pro(in[l * L + j], l, 0, j) : mk<R>(0, 0); },
        [&](int j, cx<R> v) { bufa[j * S + w] = v; });
    __syncthreads();
    cx<R>* res = smem_fft<DIR, R>(bufa, bufb, S, LW, pl, tws);
    if (act)
        for (int j = x0; j < L; j += G) store(res[j * S + w], l, 0, j);
}

// Forward real-to-complex along the contiguous axis, two real rows per
// complex line: z = a + i b, Z = FFT(z), A(k) = (Z(k) + conj Z(-k)) / 2,
// B(k) = (Z(k) - conj Z(-k)) / (2i), k in [0, X/2]. `src(row, x)` yields the
// real input (so padding / wrapping / type conversion fuse into the load).
template <typename R, class Src>
__global__ void __launch_bounds__(kSmemFftThreads) k_r2c_rows(Src src, int64_t nrows, cx<R>* __restrict__ out, LenPlan pl,
                                                  int LW, int S)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int X = pl.L, Xh = X / 2 + 1, G = kSmemFftThreads >> LW;
    cx<R>* bufa = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* bufb = bufa + X * S;
    cx<R>* tws = bufb + X * S;
    const int w = threadIdx.x / G, x0 = threadIdx.x & (G - 1);
    const int64_t ra = ((int64_t)blockIdx.x << (LW + 1)) + 2 * w, rb = ra + 1;
    load_twiddles<R>(tws, pl);
    stage_line<cx<R>>(
        x0, G, X,
        [&](int x) { return mk<R>(ra < nrows ? src(ra, x) : (R)0, rb < nrows ? src(rb, x) : (R)0); },
        [&](int x, cx<R> v) { bufa[x * S + w] = v; });
    __syncthreads();
    cx<R>* res = smem_fft<-1, R>(bufa, bufb, S, LW, pl, tws);
    for (int k = x0; k < Xh; k += G) {
        cx<R> zk = res[k * S + w];
        cx<R> zn = res[(k == 0 ? 0 : X - k) * S + w];
        // A = (zk + conj zn)/2 ; B = (zk - conj zn)/(2i)
        cx<R> A = mk<R>((zk.x + zn.x) * (R)0.5, (zk.y - zn.y) * (R)0.5);
        cx<R> d = mk<R>(zk.x - zn.x, zk.y + zn.y);
        cx<R> B = mk<R>(d.y * (R)0.5, -d.x * (R)0.5);
        if (ra < nrows) out[ra * Xh + k] = A;
        if (rb < nrows) out[rb * Xh + k] = B;
    }
}

// Inverse complex-to-real along the contiguous axis, two half-spectrum rows
// per complex line: Z(k) = A(k) + i B(k) for k <= X/2 and
// Z(k) = conj A(X-k) + i conj B(X-k) above, with the imaginary parts of the
// k = 0 (and k = X/2 for even X) bins dropped as a C2R transform does;
// IFFT(Z) = a + i b. `sink(batch, row, x, value)` consumes the real outputs
// (normalisation / max epilogues); nbatch arrays of nrows rows follow each
// other in `in`.
template <typename R, class Sink, typename In = cx<R>>
__global__ void __launch_bounds__(kSmemFftThreads) k_c2r_rows(const In* __restrict__ in, int64_t nrows, Sink sink,
                                                  LenPlan pl, int LW, int S, int nbatch)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int X = pl.L, Xh = X / 2 + 1, G = kSmemFftThreads >> LW;
    cx<R>* bufa = reinterpret_cast<cx<R>*>(smem_raw);
    cx<R>* bufb = bufa + X * S;
    cx<R>* tws = bufb + X * S;
    // batch index fastest so that the CTAs sharing rows (and the rows of any
    // per-voxel factor the sink reads) run together
    const int batch = blockIdx.x % nbatch;
    const int64_t tile = blockIdx.x / nbatch;
    const int w = threadIdx.x / G, x0 = threadIdx.x & (G - 1);
    const int64_t ra = (tile << (LW + 1)) + 2 * w, rb = ra + 1;
    const bool va = ra < nrows, vb = rb < nrows;
    const In* ba = in + ((int64_t)batch * nrows + ra) * Xh;
    const In* bb = ba + Xh;
    load_twiddles<R>(tws, pl);
    struct Pair { cx<R> A, B; };
    stage_line<Pair>(
        x0, G, Xh,
        [&](int k) {
            Pair p;
            p.A = va ? load_cx(ba[k]) : mk<R>(0, 0);
            p.B = vb ? load_cx(bb[k]) : mk<R>(0, 0);
            return p;
        },
        [&](int k, Pair p) {
            if (k == 0 || (2 * k == X)) { p.A.y = 0; p.B.y = 0; }
            // Z(k) = A + iB
            bufa[k * S + w] = mk<R>(p.A.x - p.B.y, p.A.y + p.B.x);
            // Z(X-k) = conj A + i conj B, for the bins not covered above
            const int kk = X - k;
            if (k >= 1 && kk >= Xh) bufa[kk * S + w] = mk<R>(p.A.x + p.B.y, -p.A.y + p.B.x);
        });
    __syncthreads();
    cx<R>* res = smem_fft<+1, R>(bufa, bufb, S, LW, pl, tws);
    for (int x = x0; x < X; x += G) {
        const cx<R> v = res[x * S + w];
        if (va) sink(batch, ra, x, v.x);
        if (vb) sink(batch, rb, x, v.y);
    }
}

// ------------------------------------------------------------ host side --

// Radix schedule for L (7-smooth); returns false otherwise.
bool factor_length(int L, LenPlan& pl);

// Tile of a shared-memory pass of length L: W = 2^LW lines per CTA, element
// stride S (W, or W + 1 for tiles copied along their lines), and its
// dynamic shared memory in bytes.
struct TileShape {
    int W, LW, S;
    size_t smem;
};
TileShape choose_tile(int L, size_t elem_bytes, int min_w, int max_w, bool along_lines);
// the plan's tuned tile width if it has one (rounded down to a power of two,
// within the shared-memory budget), else choose_tile
TileShape plan_tile(const LenPlan& pl, size_t elem_bytes, int min_w, int max_w, bool along_lines);
// the plan with the reciprocals that its schedule needs
LenPlan with_magic(LenPlan pl);

}  // namespace ttm

namespace ttm {

// Device twiddle tables, one per (length, precision), owned by a context.
// twiddle precision: FP32, FP64, or double-float pairs
enum TwKind { TW_F32 = 0, TW_F64 = 1, TW_DF64 = 2 };

class TwiddleCache {
  public:
    ~TwiddleCache();
    const void* get(int L, int kind);
    int num_sms = 1;  // of the context's device, handed to the plans

  private:
    struct Entry { int L; int kind; void* ptr; };
    Entry* entries_ = nullptr;
    int n_ = 0, cap_ = 0;
};

// LenPlan for L with the twiddles of the given precision (TwKind).
LenPlan make_len_plan(TwiddleCache& tc, int L, int kind);

template <typename K>
inline void set_smem(K kernel, size_t bytes)
{
    if (bytes > 48 * 1024)
        TTM_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

// strided-axis pass (lines adjacent along the inner index)
template <typename R, int DIR, class Pro, class Store, typename In = cx<R>>
inline void launch_strided(const In* in, StridedAxis ax, const LenPlan& pl, Pro pro, Store store,
                           cudaStream_t st)
{
    TileShape ts = plan_tile(pl, sizeof(cx<R>), 4, 16, false);
    auto k = k_fft_strided<R, DIR, Pro, Store, In>;
    set_smem(k, ts.smem);
    int64_t grid = ax.outer * ceil_div(ax.inner, ts.W);
    TTM_REQUIRE(grid < (1ll << 31), E_SHAPE, "strided pass grid too large");
    k<<<(unsigned)grid, kSmemFftThreads, ts.smem, st>>>(in, ax, with_magic(pl), ts.LW, pro, store);
    TTM_LAUNCH_CHECK();
}

template <typename R, int DIR, class Pro, class Store>
inline void launch_contig(const cx<R>* in, int64_t nlines, const LenPlan& pl, Pro pro, Store store,
                          cudaStream_t st)
{
    TileShape ts = plan_tile(pl, sizeof(cx<R>), 1, 8, true);
    auto k = k_fft_contig<R, DIR, Pro, Store>;
    set_smem(k, ts.smem);
    int64_t grid = ceil_div(nlines, ts.W);
    k<<<(unsigned)grid, kSmemFftThreads, ts.smem, st>>>(in, nlines, with_magic(pl), ts.LW, ts.S, pro, store);
    TTM_LAUNCH_CHECK();
}

template <typename R, class Src>
inline void launch_r2c_rows(Src src, int64_t nrows, cx<R>* out, const LenPlan& pl, cudaStream_t st)
{
    TileShape ts = choose_tile(pl.L, sizeof(cx<R>), 1, 8, true);
    auto k = k_r2c_rows<R, Src>;
    set_smem(k, ts.smem);
    int64_t grid = ceil_div(nrows, 2 * ts.W);
    k<<<(unsigned)grid, kSmemFftThreads, ts.smem, st>>>(src, nrows, out, with_magic(pl), ts.LW, ts.S);
    TTM_LAUNCH_CHECK();
}

template <typename R, class Sink, typename In = cx<R>>
inline void launch_c2r_rows(const In* in, int64_t nrows, Sink sink, const LenPlan& pl, int nbatch,
                            cudaStream_t st)
{
    TileShape ts = plan_tile(pl, sizeof(cx<R>), 1, 8, true);
    auto k = k_c2r_rows<R, Sink, In>;
    set_smem(k, ts.smem);
    int64_t grid = ceil_div(nrows, 2 * ts.W) * nbatch;
    TTM_REQUIRE(grid < (1ll << 31), E_SHAPE, "c2r pass grid too large");
    k<<<(unsigned)grid, kSmemFftThreads, ts.smem, st>>>(in, nrows, sink, with_magic(pl), ts.LW, ts.S, nbatch);
    TTM_LAUNCH_CHECK();
}

}  // namespace ttm
