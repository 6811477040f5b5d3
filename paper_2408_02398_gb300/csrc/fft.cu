// fft.cu -- host side of the FFT passes: radix schedules, tile shapes and
// twiddle tables.
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "fft_pfa.cuh"

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

// the coprime parts of a 7-smooth L, in the order of their rows
static int pfa_parts(int L, int* g, int* p)
{
    int n = 0;
    for (int r : {2, 3, 5, 7}) {
        int q = 1;
        while (L % r == 0) { L /= r; q *= r; }
        if (q > 1) { g[n] = q; p[n++] = r; }
    }
    return n;
}

void pfa_maps(int L, uint16_t* maps)
{
    uint16_t *crt = maps, *rur = maps + L, *kof = maps + 2 * L;
    int g[4], p[4];
    const int n = pfa_parts(L, g, p);
    int inv[4] = {0, 0, 0, 0};  // (L/g)^-1 mod g
    for (int i = 0; i < n; i++)
        while ((int64_t)inv[i] * (L / g[i]) % g[i] != 1 % g[i]) inv[i]++;
    for (int j = 0; j < L; j++) {
        int rc = 0, rr = 0, G = 1;
        for (int i = 0; i < n; i++) {
            // j = sum (L/g) k_g mod L: k_g = j (L/g)^-1 mod g
            rc += G * (j % g[i]);
            rr += G * (int)((int64_t)j * inv[i] % g[i]);
            G *= g[i];
        }
        crt[j] = (uint16_t)rc;
        rur[j] = (uint16_t)rr;
        kof[rr] = (uint16_t)j;
    }
}

PfaPlan pfa_plan(const LenPlan& pl)
{
    PfaPlan q{};
    const int L = pl.L;
    q.L = L;
    q.tw = reinterpret_cast<const double2*>(pl.tw);
    q.crt = reinterpret_cast<const uint16_t*>(q.tw + L);
    q.rur = q.crt + L;
    q.kof = q.rur + L;
    auto magic = [](int d) { return d > 1 ? (uint32_t)(((1ull << 32) + d - 1) / d) : 0u; };
    int g[4], p[4], G = 1;
    const int n = pfa_parts(L, g, p);
    for (int i = 0; i < n; i++) {
        int rest = g[i], Ns = 1;
        while (rest > 1) {
            int r = p[i];
            if (r == 2) r = rest % 8 == 0 ? 8 : (rest % 4 == 0 ? 4 : 2);
            if (r == 3 && rest % 9 == 0) r = 9;
            PfaStage& s = q.st[q.nst++];
            s = PfaStage{r, G, g[i], Ns, g[i] / r, L / (Ns * r), magic(G), magic(g[i] / r), magic(Ns)};
            Ns *= r;
            rest /= r;
        }
        G *= g[i];
    }
    return q;
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
    // FP64: the three index maps of the prime-factor passes follow the twiddles
    const size_t maps = kind == TW_F64 ? (3 * (size_t)L * sizeof(uint16_t) + esz - 1) / esz * esz : 0;
    const size_t bytes = (size_t)L * esz + maps;
    TTM_CUDA_TRY(cudaMalloc(&d, bytes));
    if (kind == TW_F64) {
        std::vector<double2> h(bytes / sizeof(double2));
        for (int m = 0; m < L; m++) h[m] = make_double2(re[m], im[m]);
        pfa_maps(L, reinterpret_cast<uint16_t*>(h.data() + L));
        TTM_CUDA_TRY(cudaMemcpy(d, h.data(), bytes, cudaMemcpyHostToDevice));
    } else if (kind == TW_DF64) {
        // (re.hi, im.hi, re.lo, im.lo)
        std::vector<float4> h(L);
        for (int m = 0; m < L; m++) {
            float rh = (float)re[m], ih = (float)im[m];
            h[m] = make_float4(rh, ih, (float)(re[m] - (double)rh), (float)(im[m] - (double)ih));
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
    pl.num_sms = tc.num_sms;
    return pl;
}

}  // namespace ttm
