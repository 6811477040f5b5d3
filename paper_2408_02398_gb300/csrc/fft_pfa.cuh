// fft_pfa.cuh -- FP64 transforms of the local sums by the prime-factor
// algorithm (Good 1958, Thomas 1963).
//
// What bounds an FP64 pass on this GPU is the FP64 pipe: 1.7 lane operations
// per clock and SM measured, 1/64 of the FP32 rate, so a pass costs its FP64
// instructions and nothing else (521 of 535 G/s at X = 315 in the mixed-radix
// Stockham passes; memory 0.4 TB/s). So these passes spend integer
// instructions to save FP64 ones: L = 2^a 3^b 5^c 7^d is split into its
// coprime parts g, whose transforms need no twiddles between them. With the
// Chinese-remainder map of the input, n -> (n mod g)_g, and the map
// k = sum_g (L/g) k_g mod L of the output,
//   W_L^{n k} = prod_g W_g^{n_g k_g}.
// Inside a part the radices 8, 4, 2 / 9, 3 / 5 / 7 run as Stockham stages
// (twiddles only there), with butterflies whose products by constants are
// all fused into additions. FP64 instructions per element: 36 -> 26 at 315,
// 34 -> 25 at 270, 30 -> 21 at 126; 39 -> 27 at 512 against the register
// four-step. ttm_correlate of 126 x 270 x 315 (n = 4, FP64 local sums)
// 6.38 -> 5.56 ms, the same w to the last FP32 bit; a 64^3 match unchanged
// (157 us: 64 = 8 x 8 has nothing to save).
// The two index maps are their own inverses' duals: an inverse transform
// that takes its input in the forward one's output layout (rows k_g) and
// leaves its output in the remainder layout needs no permutation between
// them (local sums, z pass).
#pragma once

#include "fft.cuh"

namespace ttm {

constexpr int kPfaStages = 16;

// one stage: radix rad on the part of length g whose rows are G apart
struct PfaStage {
    int rad, G, g, Ns, nb, step;          // nb = g / rad, step = L / (Ns rad)
    uint32_t mG, mNb, mNs;                // ceil(2^32 / .) of G, nb, Ns (0 for 1)
};
// tw: exp(-2 pi i m / L), then the maps as uint16: crt[n], rur[k] (rows of
// input n / output k), kof[row] (k of a row)
struct PfaPlan {
    int L, nst;
    const double2* tw;
    const uint16_t *crt, *rur, *kof;
    PfaStage st[kPfaStages];
};
PfaPlan pfa_plan(const LenPlan& pl);
// the maps of length L, in the order crt, rur, kof
void pfa_maps(int L, uint16_t* maps);

__device__ __forceinline__ int pfa_div(int x, int d, uint32_t m) { return d == 1 ? x : (int)__umulhi((uint32_t)x, m); }

// ---------------------------------------------------------- butterflies --
// S = DIR * sin: x +- i DIR B is folded into the fused multiply-adds

template <int DIR> __device__ __forceinline__ void pfa_dft3(double2& a, double2& b, double2& c)
{
    const double s = DIR * OddRadixConst::s3;
    const double tx = b.x + c.x, ty = b.y + c.y, dx = b.x - c.x, dy = b.y - c.y;
    const double ax = fma(-0.5, tx, a.x), ay = fma(-0.5, ty, a.y);
    a.x += tx;
    a.y += ty;
    b.x = fma(-s, dy, ax); b.y = fma(s, dx, ay);
    c.x = fma(s, dy, ax);  c.y = fma(-s, dx, ay);
}

template <int DIR> __device__ __forceinline__ void pfa_dft5(double2* v)
{
    const double c1 = OddRadixConst::c5_1, c2 = OddRadixConst::c5_2;
    const double s1 = DIR * OddRadixConst::s5_1, s2 = DIR * OddRadixConst::s5_2;
    const double2 x0 = v[0];
    const double2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]), d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
    v[0] = cadd(x0, cadd(t1, t2));
    const double a1x = fma(c2, t2.x, fma(c1, t1.x, x0.x)), a1y = fma(c2, t2.y, fma(c1, t1.y, x0.y));
    const double a2x = fma(c1, t2.x, fma(c2, t1.x, x0.x)), a2y = fma(c1, t2.y, fma(c2, t1.y, x0.y));
    const double b1x = fma(s2, d2.x, s1 * d1.x), b1y = fma(s2, d2.y, s1 * d1.y);
    const double b2x = fma(-s1, d2.x, s2 * d1.x), b2y = fma(-s1, d2.y, s2 * d1.y);
    v[1] = make_double2(a1x - b1y, a1y + b1x);
    v[4] = make_double2(a1x + b1y, a1y - b1x);
    v[2] = make_double2(a2x - b2y, a2y + b2x);
    v[3] = make_double2(a2x + b2y, a2y - b2x);
}

template <int DIR> __device__ __forceinline__ void pfa_dft7(double2* v)
{
    const double c1 = OddRadixConst::c7_1, c2 = OddRadixConst::c7_2, c3 = OddRadixConst::c7_3;
    const double s1 = DIR * OddRadixConst::s7_1, s2 = DIR * OddRadixConst::s7_2, s3 = DIR * OddRadixConst::s7_3;
    const double2 x0 = v[0];
    const double2 t1 = cadd(v[1], v[6]), t2 = cadd(v[2], v[5]), t3 = cadd(v[3], v[4]);
    const double2 d1 = csub(v[1], v[6]), d2 = csub(v[2], v[5]), d3 = csub(v[3], v[4]);
    v[0] = cadd(x0, cadd(t1, cadd(t2, t3)));
    auto A = [&](double p, double q, double r) {
        return make_double2(fma(r, t3.x, fma(q, t2.x, fma(p, t1.x, x0.x))), fma(r, t3.y, fma(q, t2.y, fma(p, t1.y, x0.y))));
    };
    auto B = [&](double p, double q, double r) {
        return make_double2(fma(r, d3.x, fma(q, d2.x, p * d1.x)), fma(r, d3.y, fma(q, d2.y, p * d1.y)));
    };
    auto out = [&](int k, double2 a, double2 b) {
        v[k] = make_double2(a.x - b.y, a.y + b.x);
        v[7 - k] = make_double2(a.x + b.y, a.y - b.x);
    };
    // 2 pi r k / 7: (r k mod 7) in {4, 5, 6} takes minus the sine of 7 - (r k mod 7)
    out(1, A(c1, c2, c3), B(s1, s2, s3));
    out(2, A(c2, c3, c1), B(s2, -s3, -s1));
    out(3, A(c3, c1, c2), B(s3, -s1, s2));
}

template <int DIR> __device__ __forceinline__ void pfa_dft8(double2* v)
{
    double2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<DIR>(e0, e1, e2, e3);
    dft4<DIR>(o0, o1, o2, o3);
    const double h = OddRadixConst::sqrt_half;
    // o1 h (1 + DIR i) and o3 h (-1 + DIR i), the products by h fused below
    const double2 p = make_double2(o1.x - DIR * o1.y, o1.y + DIR * o1.x);
    const double2 q = make_double2(-o3.x - DIR * o3.y, DIR * o3.x - o3.y);
    const double2 r = cmul_diri<DIR>(o2);
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[2] = cadd(e2, r);  v[6] = csub(e2, r);
    v[1] = make_double2(fma(h, p.x, e1.x), fma(h, p.y, e1.y));
    v[5] = make_double2(fma(-h, p.x, e1.x), fma(-h, p.y, e1.y));
    v[3] = make_double2(fma(h, q.x, e3.x), fma(h, q.y, e3.y));
    v[7] = make_double2(fma(-h, q.x, e3.x), fma(-h, q.y, e3.y));
}

// exp(DIR 2 pi i / 9), its square and its fourth power
struct Ninth {
    static constexpr double c1 = 0.76604444311897803520239265055542, s1 = 0.64278760968653932632264340990726;
    static constexpr double c2 = 0.17364817766693034885171662676931, s2 = 0.98480775301220805936674302458952;
    static constexpr double c4 = -0.93969262078590838405410927732473, s4 = 0.34202014332566873304409961468226;
};
template <int DIR> __device__ __forceinline__ void pfa_dft9(double2* v)
{
#pragma unroll
    for (int p = 0; p < 3; p++) pfa_dft3<DIR>(v[p], v[p + 3], v[p + 6]);
    // v[p + 3 k1]: times w9^{p k1}, then a transform over p
    const double2 w1 = make_double2(Ninth::c1, DIR * Ninth::s1), w2 = make_double2(Ninth::c2, DIR * Ninth::s2),
                  w4 = make_double2(Ninth::c4, DIR * Ninth::s4);
    v[4] = cmul(v[4], w1);
    v[5] = cmul(v[5], w2);
    v[7] = cmul(v[7], w2);
    v[8] = cmul(v[8], w4);
#pragma unroll
    for (int k1 = 0; k1 < 3; k1++) pfa_dft3<DIR>(v[3 * k1], v[3 * k1 + 1], v[3 * k1 + 2]);
    // X[k1 + 3 k2] is at 3 k1 + k2: transpose
    double2 t;
    t = v[1]; v[1] = v[3]; v[3] = t;
    t = v[2]; v[2] = v[6]; v[6] = t;
    t = v[5]; v[5] = v[7]; v[7] = t;
}

template <int RAD, int DIR> __device__ __forceinline__ void pfa_dft(double2* v)
{
    if constexpr (RAD == 2) dft2<DIR>(v);
    else if constexpr (RAD == 3) pfa_dft3<DIR>(v[0], v[1], v[2]);
    else if constexpr (RAD == 4) dft4<DIR>(v[0], v[1], v[2], v[3]);
    else if constexpr (RAD == 5) pfa_dft5<DIR>(v);
    else if constexpr (RAD == 7) pfa_dft7<DIR>(v);
    else if constexpr (RAD == 8) pfa_dft8<DIR>(v);
    else pfa_dft9<DIR>(v);
}

// --------------------------------------------------------------- stages --

// one Stockham stage inside a part, on the 2^LW lines of a tile (row q of
// line w at (q << LW) + w)
template <int RAD, int DIR>
__device__ __forceinline__ void pfa_stage(const double2* __restrict__ in, double2* __restrict__ out, int L, int LW,
                                          const PfaStage& s, const double2* __restrict__ tw)
{
    const int w = threadIdx.x & ((1 << LW) - 1);
    const int is = (s.G * s.nb) << LW, os = (s.G * s.Ns) << LW;
    for (int b = threadIdx.x >> LW; b < L / RAD; b += blockDim.x >> LW) {
        const int t = pfa_div(b, s.G, s.mG), low = b - t * s.G;
        const int high = pfa_div(t, s.nb, s.mNb), j = t - high * s.nb;
        const int k = j - pfa_div(j, s.Ns, s.mNs) * s.Ns;
        const int base = low + high * s.G * s.g;
        const double2* src = in + ((base + s.G * j) << LW) + w;
        double2 v[RAD];
#pragma unroll
        for (int r = 0; r < RAD; r++) v[r] = src[r * is];
        if (s.Ns > 1) {
            const double2* tk = tw;
#pragma unroll
            for (int r = 1; r < RAD; r++) {
                tk += k * s.step;
                double2 t_ = *tk;
                if (DIR > 0) t_.y = -t_.y;
                v[r] = cmul(v[r], t_);
            }
        }
        pfa_dft<RAD, DIR>(v);
        double2* dst = out + ((base + s.G * ((j - k) * RAD + k)) << LW) + w;
#pragma unroll
        for (int r = 0; r < RAD; r++) dst[r * os] = v[r];
    }
}

// the transform of the tile in a (scratch b); returns the buffer that holds
// the result and ends with __syncthreads()
template <int DIR>
__device__ double2* pfa_fft(double2* a, double2* b, int LW, const PfaPlan& pl, const double2* tw)
{
    const int L = pl.L;
    for (int i = 0; i < pl.nst; i++) {
        const PfaStage& s = pl.st[i];
        switch (s.rad) {
            case 2: pfa_stage<2, DIR>(a, b, L, LW, s, tw); break;
            case 3: pfa_stage<3, DIR>(a, b, L, LW, s, tw); break;
            case 4: pfa_stage<4, DIR>(a, b, L, LW, s, tw); break;
            case 5: pfa_stage<5, DIR>(a, b, L, LW, s, tw); break;
            case 7: pfa_stage<7, DIR>(a, b, L, LW, s, tw); break;
            case 8: pfa_stage<8, DIR>(a, b, L, LW, s, tw); break;
            default: pfa_stage<9, DIR>(a, b, L, LW, s, tw); break;
        }
        __syncthreads();
        double2* t = a; a = b; b = t;
    }
    return a;
}

__device__ __forceinline__ void pfa_twiddles(double2* tws, const PfaPlan& pl)
{
    for (int i = threadIdx.x; i < pl.L; i += blockDim.x) tws[i] = pl.tw[i];
}

// -------------------------------------------------------------- kernels --
// shared memory: (2 W + 1) L double2

// strided axis, functors as in k_fft_strided
template <int DIR, class Pro, class Store>
__global__ void __launch_bounds__(kSmemFftThreads)
k_pfa_strided(const double2* __restrict__ in, StridedAxis ax, const __grid_constant__ PfaPlan pl, int LW, Pro pro,
              Store store)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = pl.L, W = 1 << LW;
    double2* bufa = reinterpret_cast<double2*>(smem_raw);
    double2* bufb = bufa + L * W;
    double2* tws = bufb + L * W;
    const int64_t tiles = (ax.inner + W - 1) >> LW;
    const int64_t o = blockIdx.x / tiles;
    const int w = threadIdx.x & (W - 1);
    const int64_t i = ((blockIdx.x - o * tiles) << LW) + w;
    const bool act = i < ax.inner;
    pfa_twiddles(tws, pl);
    const double2* src = in + o * ax.os + i;
    stage_tile<double2>(
        W * L,
        [&](int idx) {
            const int j = idx >> LW;
            return act ? pro(src[(int64_t)j * ax.s], o, i, j) : make_double2(0, 0);
        },
        [&](int idx, double2 v) { bufa[((int)__ldg(pl.crt + (idx >> LW)) << LW) + w] = v; });
    __syncthreads();
    const double2* res = pfa_fft<DIR>(bufa, bufb, LW, pl, tws);
    if (act)
        for (int idx = threadIdx.x; idx < W * L; idx += blockDim.x) store(res[idx], o, i, (int)__ldg(pl.kof + (idx >> LW)));
}

// contiguous lines, functors as in k_fft_contig; blockDim / W consecutive
// threads work on one line
template <int DIR, class Pro, class Store>
__global__ void __launch_bounds__(kSmemFftThreads)
k_pfa_contig(const double2* __restrict__ in, int64_t nlines, const __grid_constant__ PfaPlan pl, int LW, Pro pro,
             Store store)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = pl.L, W = 1 << LW, G = blockDim.x >> LW;
    double2* bufa = reinterpret_cast<double2*>(smem_raw);
    double2* bufb = bufa + L * W;
    double2* tws = bufb + L * W;
    const int w = threadIdx.x / G, x0 = threadIdx.x & (G - 1);
    const int64_t l = ((int64_t)blockIdx.x << LW) + w;
    const bool act = l < nlines;
    pfa_twiddles(tws, pl);
    stage_line<double2>(
        x0, G, L, [&](int j) { return act ? pro(in[l * L + j], l, 0, j) : make_double2(0, 0); },
        [&](int j, double2 v) { bufa[((int)__ldg(pl.crt + j) << LW) + w] = v; });
    __syncthreads();
    const double2* res = pfa_fft<DIR>(bufa, bufb, LW, pl, tws);
    if (act)
        for (int j = x0; j < L; j += G) store(res[((int)__ldg(pl.rur + j) << LW) + w], l, 0, j);
}

// z pass of the local sums, in place: forward, times mask(v, 0, column, kz),
// inverse, on W adjacent columns
template <class Mask>
__global__ void __launch_bounds__(kSmemFftThreads)
k_pfa_zmask(double2* __restrict__ zd, int64_t ncols, const __grid_constant__ PfaPlan pl, int LW, Mask mask)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = pl.L, W = 1 << LW;
    double2* bufa = reinterpret_cast<double2*>(smem_raw);
    double2* bufb = bufa + L * W;
    double2* tws = bufb + L * W;
    const int w = threadIdx.x & (W - 1);
    const int64_t c = ((int64_t)blockIdx.x << LW) + w;
    const bool act = c < ncols;
    pfa_twiddles(tws, pl);
    stage_tile<double2>(
        W * L, [&](int idx) { return act ? zd[(int64_t)(idx >> LW) * ncols + c] : make_double2(0, 0); },
        [&](int idx, double2 v) { bufa[((int)__ldg(pl.crt + (idx >> LW)) << LW) + w] = v; });
    __syncthreads();
    double2* p = pfa_fft<-1>(bufa, bufb, LW, pl, tws);
    double2* q = p == bufa ? bufb : bufa;
    if (act)
        for (int idx = threadIdx.x; idx < W * L; idx += blockDim.x)
            p[idx] = mask(p[idx], 0, c, (int)__ldg(pl.kof + (idx >> LW)));
    __syncthreads();
    const double2* r = pfa_fft<+1>(p, q, LW, pl, tws);
    if (act)
        for (int idx = threadIdx.x; idx < W * L; idx += blockDim.x) {
            const int z = idx >> LW;
            zd[(int64_t)z * ncols + c] = r[((int)__ldg(pl.crt + z) << LW) + w];
        }
}

// ----------------------------------------------------------------- host --

// tile of W = 2^lw lines: the widest (up to 16) that leaves two CTAs per SM
// their shared memory, narrowed while fewer than four CTAs per SM remain
// (every SM's FP64 pipe is the bound, so the CTAs have to spread evenly:
// 64 x 64 lines in tiles of 16 are 256 CTAs for 152 SMs)
inline int pfa_tile(int num_sms, int L, int64_t lines, int64_t outer, int min_lw)
{
    auto bytes = [&](int lw) { return ((2ull << lw) + 1) * L * sizeof(double2); };
    int lw = 4;
    while (lw > min_lw && bytes(lw) > 112 * 1024) lw--;
    while (lw > 2 && ceil_div(lines, 1ll << lw) * outer < 4 * (int64_t)num_sms) lw--;
    return lw;
}
inline size_t pfa_smem(int L, int lw) { return ((2ull << lw) + 1) * L * sizeof(double2); }
inline int pfa_threads(int L, int lw) { return ((int64_t)L << lw) <= 1024 ? 128 : kSmemFftThreads; }

template <int DIR, class Pro, class Store>
inline void launch_pfa_strided(const double2* in, StridedAxis ax, const LenPlan& pl, Pro pro, Store store,
                               cudaStream_t st)
{
    const int lw = pfa_tile(pl.num_sms, pl.L, ax.inner, ax.outer, 2);
    auto k = k_pfa_strided<DIR, Pro, Store>;
    const size_t smem = pfa_smem(pl.L, lw);
    set_smem(k, smem);
    const int64_t grid = ax.outer * ceil_div(ax.inner, 1ll << lw);
    TTM_REQUIRE(grid < (1ll << 31), E_SHAPE, "strided pass grid too large");
    k<<<(unsigned)grid, pfa_threads(pl.L, lw), smem, st>>>(in, ax, pfa_plan(pl), lw, pro, store);
    TTM_LAUNCH_CHECK();
}

template <int DIR, class Pro, class Store>
inline void launch_pfa_contig(const double2* in, int64_t nlines, const LenPlan& pl, Pro pro, Store store,
                              cudaStream_t st)
{
    const int lw = pfa_tile(pl.num_sms, pl.L, nlines, 1, 0);
    auto k = k_pfa_contig<DIR, Pro, Store>;
    const size_t smem = pfa_smem(pl.L, lw);
    set_smem(k, smem);
    k<<<(unsigned)ceil_div(nlines, 1ll << lw), pfa_threads(pl.L, lw), smem, st>>>(in, nlines, pfa_plan(pl), lw, pro, store);
    TTM_LAUNCH_CHECK();
}

template <class Mask>
inline void launch_pfa_zmask(double2* zd, int64_t ncols, const LenPlan& pl, Mask mask, cudaStream_t st)
{
    const int lw = pfa_tile(pl.num_sms, pl.L, ncols, 1, 1);
    auto k = k_pfa_zmask<Mask>;
    const size_t smem = pfa_smem(pl.L, lw);
    set_smem(k, smem);
    k<<<(unsigned)ceil_div(ncols, 1ll << lw), pfa_threads(pl.L, lw), smem, st>>>(zd, ncols, pfa_plan(pl), lw, mask);
    TTM_LAUNCH_CHECK();
}

}  // namespace ttm
