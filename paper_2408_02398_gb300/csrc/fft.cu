// fft.cu -- host side of the FFT passes: radix schedules, tile shapes and
// twiddle tables.
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "fft.cuh"

namespace ttm {

bool factor_length(int L, LenPlan& pl)
{
    pl.L = L;
    pl.nst = 0;
    pl.tw = nullptr;
    if (L < 1) return false;
    int rest = L;
    // largest radices first; a trailing power of two below 8 becomes one
    // radix-4 or radix-2 stage
    while (rest % 8 == 0 && pl.nst < kMaxStages) { pl.rad[pl.nst++] = 8; rest /= 8; }
    if (rest % 4 == 0) { pl.rad[pl.nst++] = 4; rest /= 4; }
    if (rest % 2 == 0) { pl.rad[pl.nst++] = 2; rest /= 2; }
    const int odd[3] = {7, 5, 3};
    for (int r : odd)
        while (rest % r == 0 && pl.nst < kMaxStages) { pl.rad[pl.nst++] = r; rest /= r; }
    if (L == 1) { pl.rad[pl.nst++] = 2; return false; }
    return rest == 1;
}

static TileShape tile_of(int L, size_t elem_bytes, int LW, bool along_lines)
{
    TileShape t;
    t.LW = LW;
    t.W = 1 << LW;
    t.S = along_lines && t.W > 1 ? t.W + 1 : t.W;
    t.smem = (2 * (size_t)t.S * L + L) * elem_bytes;
    return t;
}

static int floor_log2(int v)
{
    int l = 0;
    while ((2 << l) <= v) l++;
    return l;
}

TileShape choose_tile(int L, size_t elem_bytes, int min_w, int max_w, bool along_lines)
{
    const size_t budget = 112 * 1024;  // two CTAs per SM
    int lw = floor_log2(max_w);
    while ((1 << lw) > min_w && tile_of(L, elem_bytes, lw, along_lines).smem > budget) lw--;
    return tile_of(L, elem_bytes, lw, along_lines);
}

TileShape plan_tile(const LenPlan& pl, size_t elem_bytes, int min_w, int max_w, bool along_lines)
{
    if (pl.tile_w >= min_w && pl.tile_w <= max_w) {
        const TileShape t = tile_of(pl.L, elem_bytes, floor_log2(pl.tile_w), along_lines);
        if (t.smem <= 200 * 1024) return t;
    }
    return choose_tile(pl.L, elem_bytes, min_w, max_w, along_lines);
}

LenPlan with_magic(LenPlan pl)
{
    uint64_t Ns = 1;
    for (int s = 0; s < pl.nst; s++) {
        pl.mag[s] = Ns > 1 ? (uint32_t)(((1ull << 32) + Ns - 1) / Ns) : 0u;
        Ns *= (uint64_t)pl.rad[s];
    }
    return pl;
}

TwiddleCache::~TwiddleCache()
{
    for (int i = 0; i < n_; i++) cudaFree(entries_[i].ptr);
    std::free(entries_);
}

const void* TwiddleCache::get(int L, int kind)
{
    for (int i = 0; i < n_; i++)
        if (entries_[i].L == L && entries_[i].kind == kind) return entries_[i].ptr;
    // exp(-2 pi i m / L) from the exact fraction m / L, in double precision
    std::vector<double> re(L), im(L);
    for (int m = 0; m < L; m++) {
        double a = 2.0 * M_PI * (double)m / (double)L;
        re[m] = std::cos(a);
        im[m] = -std::sin(a);
    }
    void* d = nullptr;
    const size_t esz = kind == TW_F32 ? sizeof(float2) : sizeof(double2);
    const size_t bytes = (size_t)L * esz;
    TTM_CUDA_TRY(cudaMalloc(&d, bytes));
    if (kind == TW_F64) {
        std::vector<double2> h(L);
        for (int m = 0; m < L; m++) h[m] = make_double2(re[m], im[m]);
        TTM_CUDA_TRY(cudaMemcpy(d, h.data(), bytes, cudaMemcpyHostToDevice));
    } else if (kind == TW_DF64) {
        // (re.hi, re.lo, im.hi, im.lo)
        std::vector<float4> h(L);
        for (int m = 0; m < L; m++) {
            float rh = (float)re[m], ih = (float)im[m];
            h[m] = make_float4(rh, (float)(re[m] - (double)rh), ih, (float)(im[m] - (double)ih));
        }
        TTM_CUDA_TRY(cudaMemcpy(d, h.data(), bytes, cudaMemcpyHostToDevice));
    } else {
        std::vector<float2> h(L);
        for (int m = 0; m < L; m++) h[m] = make_float2((float)re[m], (float)im[m]);
        TTM_CUDA_TRY(cudaMemcpy(d, h.data(), bytes, cudaMemcpyHostToDevice));
    }
    if (n_ == cap_) {
        cap_ = cap_ ? 2 * cap_ : 8;
        entries_ = (Entry*)std::realloc(entries_, sizeof(Entry) * cap_);
    }
    entries_[n_++] = Entry{L, kind, d};
    return d;
}

LenPlan make_len_plan(TwiddleCache& tc, int L, int kind)
{
    LenPlan pl;
    TTM_REQUIRE(factor_length(L, pl), E_SHAPE,
                "transform length " + std::to_string(L) + " is not a product of 2, 3, 5 and 7");
    pl.tw = tc.get(L, kind);
    return pl;
}

}  // namespace ttm
