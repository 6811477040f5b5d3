// ttm_refine.cu -- position refinement of TTM peaks (TTM-ref, Sec. 3.3 and
// Alg. 3). For each peak x_i the voxels of the ball ||x - x_i|| <= r_s are
// scored by the LNCC at their own optimal rotation,
//   c(x) = w(x) sum_z t'(R(q*(x))^T z) g(x + z),
// in real space (the template window around x, trilinear samples of the
// normalised template t', zero outside its grid), and the peak moves to the
// best of them. q*(x) is the quaternion map of the d' = 4 maximiser; g and
// w are the filtered tomogram and local normaliser of the plan's last
// correlation (Eq. 2, Eq. 3).
//
// One CTA per (peak, candidate): its threads stride over template voxels
// with FP32 samples and partial sums, reduced in FP64. The candidates of a
// peak are the peak itself, then the other ball voxels in (z, y, x) order;
// the first strictly higher LNCC in that order is kept (Alg. 3). Candidates
// outside the valid box (whose template window leaves the tomogram) are not
// scored.
//
// What bounds it is instruction issue, then the gathers of t' from L1: 300
// peaks x 123 candidates of a 40^3 template are 2.4e9 samples. A rotation
// keeps lengths, so a sample farther than r + sqrt 3 (plus the soft width)
// from the centre is zero: the host lists the offsets inside (36 % of 40^3),
// each with its offset in g, and t' lies in a frame of zeros kRefPad wide,
// so a sample is four loads of x pairs without a bounds test. Floor and fraction come
// from one addition of 2^23 rounded down. The call took 20.7 ms with every
// voxel sampled, 6.5 with the list and single loads, 4.3 with pairs.
#include <algorithm>
#include <cmath>
#include <vector>

#include "ttm_internal.h"

namespace ttm {

constexpr int kRefThreads = 256;
// width of the frame of zeros around t': the support ends sqrt 3 beyond a
// mask that fits the template grid, and a sample reads one voxel further
constexpr int kRefPad = 3;

struct RefGeom {
    int Z, Y, X;                 // working grid of g and w
    int b[6];                    // valid box (z0, z1, y0, y1, x0, x1)
    int tz, ty, tx;              // template grid
    int64_t V;                   // Z * Y * X (component stride of the quaternion map)
};

// one listed template voxel: offsets + 128 in bytes 0 (x), 1 (y), 2 (z), and
// its linear offset in g
struct RefVoxel {
    uint32_t xyz;
    int gofs;
};

__device__ __forceinline__ float trilinear32(const float2* __restrict__ v, int tz, int ty, int tx, float fx, float fy,
                                             float fz)
{
    const float x0 = floorf(fx), y0 = floorf(fy), z0 = floorf(fz);
    const float ax = fx - x0, ay = fy - y0, az = fz - z0;
    const int ix = (int)x0, iy = (int)y0, iz = (int)z0;
    const int py = tx + 2 * kRefPad, pz = (ty + 2 * kRefPad) * py;
    float acc = 0.f;
#pragma unroll
    for (int dz = 0; dz <= 1; dz++)
#pragma unroll
        for (int dy = 0; dy <= 1; dy++)
#pragma unroll
            for (int dx = 0; dx <= 1; dx++) {
                const int xx = ix + dx, yy = iy + dy, zz = iz + dz;
                if (xx < 0 || xx >= tx || yy < 0 || yy >= ty || zz < 0 || zz >= tz) continue;
                const float wgt = (dx ? ax : 1.f - ax) * (dy ? ay : 1.f - ay) * (dz ? az : 1.f - az);
                acc += wgt * v[(int64_t)(zz + kRefPad) * pz + (yy + kRefPad) * py + xx + kRefPad].x;
            }
    return acc;
}

// floor of v in [0, 2^22) as 2^23 + floor(v): the integer is in the low bits
__device__ __forceinline__ float floor_biased(float v) { return __fadd_rd(v, 8388608.f); }
// byte k of w as a float minus 128
__device__ __forceinline__ float byte_offset(uint32_t w, int k)
{
    return __int_as_float(0x4B000000 | ((w >> (8 * k)) & 0xFFu)) - 8388736.f;
}

// grid (n_cand, P): candidate j of peak i; writes the LNCC (or -inf outside
// the valid box) and the candidate's quaternion. tp: t' in its frame of
// zeros; list: the n_list offsets that a rotation can bring into t'
__global__ void __launch_bounds__(kRefThreads)
k_refine_lncc(const float* __restrict__ g, const float* __restrict__ w, const float* __restrict__ orient,
              const float2* __restrict__ tp, const RefVoxel* __restrict__ list, int n_list,
              const int64_t* __restrict__ peaks, const int* __restrict__ offs, int n_cand, RefGeom geo,
              double* __restrict__ c_out, float4* __restrict__ q_out)
{
    __shared__ double red[kRefThreads / 32];
    const int j = blockIdx.x, i = blockIdx.y;
    const int64_t pk = peaks[i];
    const int px = (int)(pk % geo.X), py = (int)((pk / geo.X) % geo.Y), pz = (int)(pk / ((int64_t)geo.X * geo.Y));
    const int z = pz + offs[3 * j], y = py + offs[3 * j + 1], x = px + offs[3 * j + 2];
    const int64_t slot = (int64_t)i * n_cand + j;
    const bool inside = z >= geo.b[0] && z < geo.b[1] && y >= geo.b[2] && y < geo.b[3] && x >= geo.b[4] && x < geo.b[5];
    if (!inside) {  // uniform over the CTA
        if (threadIdx.x == 0) {
            c_out[slot] = -INFINITY;
            q_out[slot] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        return;
    }
    const int64_t v = ((int64_t)z * geo.Y + y) * geo.X + x;
    const float qw = orient[v], qx = orient[geo.V + v], qy = orient[2 * geo.V + v], qz = orient[3 * geo.V + v];
    // R(q), row-major, acting on (x, y, z) column vectors
    const float R0 = 1.f - 2.f * (qy * qy + qz * qz), R1 = 2.f * (qx * qy - qw * qz), R2 = 2.f * (qx * qz + qw * qy);
    const float R3 = 2.f * (qx * qy + qw * qz), R4 = 1.f - 2.f * (qx * qx + qz * qz), R5 = 2.f * (qy * qz - qw * qx);
    const float R6 = 2.f * (qx * qz - qw * qy), R7 = 2.f * (qy * qz + qw * qx), R8 = 1.f - 2.f * (qx * qx + qy * qy);
    const int cz = geo.tz / 2, cy = geo.ty / 2, cx = geo.tx / 2;
    const float* gv = g + v;
    float acc = 0.f;
    const float nq = qw * qw + qx * qx + qy * qy + qz * qz;
    if (n_list > 0 && fabsf(nq - 1.f) < 1e-4f) {  // uniform over the CTA
        const int sy = geo.tx + 2 * kRefPad, sz = (geo.ty + 2 * kRefPad) * sy;
        const unsigned mx = geo.tx + 2 * kRefPad - 2, my = geo.ty + 2 * kRefPad - 2, mz = geo.tz + 2 * kRefPad - 2;
        const float ox0 = (float)(cx + kRefPad), oy0 = (float)(cy + kRefPad), oz0 = (float)(cz + kRefPad);
#pragma unroll 2
        for (int t = threadIdx.x; t < n_list; t += kRefThreads) {
            const uint2 e = __ldg(reinterpret_cast<const uint2*>(list) + t);
            const float gval = __ldg(gv + (int)e.y);
            const float ox = byte_offset(e.x, 0), oy = byte_offset(e.x, 1), oz = byte_offset(e.x, 2);
            // t'_R(o) = t'(R^T o)
            const float fx = R0 * ox + R3 * oy + R6 * oz + ox0, fy = R1 * ox + R4 * oy + R7 * oz + oy0,
                        fz = R2 * ox + R5 * oy + R8 * oz + oz0;
            const float bx = floor_biased(fx), by = floor_biased(fy), bz = floor_biased(fz);
            const float ax = fx - (bx - 8388608.f), ay = fy - (by - 8388608.f), az = fz - (bz - 8388608.f);
            // (the clamps never act for a unit quaternion; they keep the loads inside for any other)
            const unsigned ix = min(__float_as_uint(bx) & 0x7FFFFFu, mx), iy = min(__float_as_uint(by) & 0x7FFFFFu, my),
                           iz = min(__float_as_uint(bz) & 0x7FFFFFu, mz);
            const float2* p = tp + (iz * sz + iy * sy + ix);
            const float2 p00 = __ldg(p), p01 = __ldg(p + sy), p10 = __ldg(p + sz), p11 = __ldg(p + sz + sy);
            const float v00 = fmaf(ax, p00.y - p00.x, p00.x), v01 = fmaf(ax, p01.y - p01.x, p01.x);
            const float v10 = fmaf(ax, p10.y - p10.x, p10.x), v11 = fmaf(ax, p11.y - p11.x, p11.x);
            const float v0 = fmaf(ay, v01 - v00, v00), v1 = fmaf(ay, v11 - v10, v10);
            const float tv = fmaf(az, v1 - v0, v0);
            // (no sample beside the support: a value of g there, infinite or NaN, does not enter)
            if (tv != 0.f) acc = fmaf(tv, gval, acc);
        }
    } else {
        // not a unit quaternion (or a template too large for the list): every voxel of the template grid
        const int nt = geo.tz * geo.ty * geo.tx;
        for (int t = threadIdx.x; t < nt; t += blockDim.x) {
            const int tx_ = t % geo.tx, ty_ = (t / geo.tx) % geo.ty, tz_ = t / (geo.tx * geo.ty);
            const float ox = (float)(tx_ - cx), oy = (float)(ty_ - cy), oz = (float)(tz_ - cz);
            const float sx = R0 * ox + R3 * oy + R6 * oz, sy = R1 * ox + R4 * oy + R7 * oz,
                        sz = R2 * ox + R5 * oy + R8 * oz;
            const float tv = trilinear32(tp, geo.tz, geo.ty, geo.tx, sx + cx, sy + cy, sz + cz);
            if (tv != 0.f) acc += tv * __ldg(gv + ((int64_t)(tz_ - cz) * geo.Y + (ty_ - cy)) * geo.X + (tx_ - cx));
        }
    }
    double d = acc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < kRefThreads / 32; k++) s += red[k];
        c_out[slot] = (double)w[v] * s;
        q_out[slot] = make_float4(qw, qx, qy, qz);
    }
}

// the first candidate of each peak with the highest LNCC (one warp per peak;
// a NaN never replaces a kept one): its index, LNCC and quaternion
struct RefPick {
    float4 q;
    int j;
    float c;
};
__global__ void k_refine_pick(const double* __restrict__ c, const float4* __restrict__ q, int n_cand, int P,
                              RefPick* __restrict__ out)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= P) return;
    const double* ci = c + (int64_t)i * n_cand;
    double best = ci[0];
    int bj = 0;
    for (int j = lane; j < n_cand; j += 32)
        if (ci[j] > best) { best = ci[j]; bj = j; }
    if (best == best) {  // the peak's own LNCC is a number
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (ob > best || (ob == best && oj < bj)) { best = ob; bj = oj; }
        }
    }
    if (lane == 0) {
        RefPick r;
        r.q = q[(int64_t)i * n_cand + bj];
        r.j = bj;
        r.c = (float)ci[bj];
        out[i] = r;
    }
}

// t' in FP32 inside its frame of zeros, each voxel beside its x neighbour
__global__ void k_pad_template(const double* __restrict__ a, int tz, int ty, int tx, float2* __restrict__ b)
{
    const int px = tx + 2 * kRefPad, py = ty + 2 * kRefPad, n = (tz + 2 * kRefPad) * py * px;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int x = i % px - kRefPad, y = (i / px) % py - kRefPad, z = i / (px * py) - kRefPad;
        const bool in = y >= 0 && y < ty && z >= 0 && z < tz;
        const double* row = a + ((int64_t)z * ty + y) * tx;
        b[i] = make_float2(in && x >= 0 && x < tx ? (float)row[x] : 0.f,
                           in && x >= -1 && x < tx - 1 ? (float)row[x + 1] : 0.f);
    }
}

// the offsets of the template grid within the reach of t' under a rotation
// (empty where they or their offsets in g do not fit the entries)
static std::vector<RefVoxel> reach_list(const RefGeom& geo, double reach)
{
    std::vector<RefVoxel> l;
    const int64_t far = (int64_t)(reach + 1) * ((int64_t)geo.Y * geo.X + geo.X + 1);
    if (reach > 126 || far >= (1ll << 31)) return l;
    const int cz = geo.tz / 2, cy = geo.ty / 2, cx = geo.tx / 2;
    for (int z = -cz; z < geo.tz - cz; z++)
        for (int y = -cy; y < geo.ty - cy; y++)
            for (int x = -cx; x < geo.tx - cx; x++)
                if ((double)(x * x + y * y + z * z) <= reach * reach)
                    l.push_back(RefVoxel{(uint32_t)(x + 128) | (uint32_t)(y + 128) << 8 | (uint32_t)(z + 128) << 16,
                                         (z * geo.Y + y) * geo.X + x});
    return l;
}

// Alg. 3's candidate set: the peak, then the rest of the ball in (z, y, x) order
static std::vector<int> ball_offsets(double rs)
{
    std::vector<int> o = {0, 0, 0};
    const int R = (int)std::floor(rs);
    for (int dz = -R; dz <= R; dz++)
        for (int dy = -R; dy <= R; dy++)
            for (int dx = -R; dx <= R; dx++) {
                if (dz == 0 && dy == 0 && dx == 0) continue;
                if ((double)(dz * dz + dy * dy + dx * dx) > rs * rs) continue;
                o.push_back(dz); o.push_back(dy); o.push_back(dx);
            }
    return o;
}

}  // namespace ttm

using namespace ttm;

extern "C" ttm_status ttm_refine_peaks(ttm_plan* plan, const float* d_tmpl, const float* d_orient,
                                       const int64_t* h_peaks, int P, double r_s, int64_t* h_idx, float* h_quat,
                                       float* h_lncc, void* stream)
{
    if (!plan) return TTM_E_INVALID_ARG;
    try {
        TTM_REQUIRE(d_tmpl && d_orient && (P == 0 || (h_peaks && h_idx && h_quat && h_lncc)), E_INVALID_ARG,
                    "null pointer argument");
        TTM_REQUIRE(plan->fp.dprime == 4, E_UNSUPPORTED, "refinement needs the rotation map of the d' = 4 form");
        TTM_REQUIRE(P >= 0 && P <= 65535 && r_s >= 0 && r_s <= 16, E_INVALID_ARG,
                    "P must be in [0, 65535] and r_s in [0, 16]");
        if (P == 0) return TTM_OK;
        TTM_CUDA_TRY(cudaSetDevice(plan->ctx->device));
        cudaStream_t st = (cudaStream_t)stream;
        const Prep& p = plan->prep;
        RefGeom geo;
        geo.Z = p.Z; geo.Y = p.Y; geo.X = p.X;
        ttm_plan_valid_box(plan, geo.b);
        geo.tz = p.tz; geo.ty = p.ty; geo.tx = p.tx;
        geo.V = (int64_t)p.Z * p.Y * p.X;
        for (int i = 0; i < P; i++) {
            const int64_t v = h_peaks[i];
            TTM_REQUIRE(v >= 0 && v < geo.V, E_INVALID_ARG, "peak index outside the grid");
            const int x = (int)(v % p.X), y = (int)((v / p.X) % p.Y), z = (int)(v / ((int64_t)p.X * p.Y));
            TTM_REQUIRE(z >= geo.b[0] && z < geo.b[1] && y >= geo.b[2] && y < geo.b[3] && x >= geo.b[4] &&
                            x < geo.b[5],
                        E_INVALID_ARG, "peak outside the valid box");
        }
        // t' in FP32 (Eq. 4, the same normalisation as the tensor field)
        DevBuf tp64, tp32;
        normalise_template_dev(plan->ctx, d_tmpl, p.tz, p.ty, p.tx, plan->fp, tp64, st, p.mask_t.as<double>());
        const int nt = (p.tz + 2 * kRefPad) * (p.ty + 2 * kRefPad) * (p.tx + 2 * kRefPad);
        tp32.alloc((size_t)nt * sizeof(float2));
        k_pad_template<<<(unsigned)std::min<int64_t>(1024, ceil_div(nt, 256)), 256, 0, st>>>(
            tp64.as<double>(), p.tz, p.ty, p.tx, tp32.as<float2>());
        TTM_LAUNCH_CHECK();
        // |q|^2 = 1 - d brings an offset in by up to 2 d of its length: 0.03
        // covers d = 1e-4 up to a reach of 126, and the rounding of FP32 coordinates
        const std::vector<RefVoxel> list =
            reach_list(geo, plan->fp.mask_radius + plan->fp.mask_soft_width + std::sqrt(3.0) + 0.03);
        const std::vector<int> offs = ball_offsets(r_s);
        const int n_cand = (int)offs.size() / 3;
        const size_t slots = (size_t)P * n_cand;
        DevBuf d_q, d_c, d_pick, d_peaks, d_list, d_offs;
        d_q.alloc(slots * sizeof(float4));
        d_c.alloc(slots * sizeof(double));
        d_pick.alloc((size_t)P * sizeof(RefPick));
        d_peaks.alloc((size_t)P * sizeof(int64_t));
        d_list.alloc(list.size() * sizeof(RefVoxel));
        d_offs.alloc(offs.size() * sizeof(int));
        if (!list.empty())
            TTM_CUDA_TRY(cudaMemcpyAsync(d_list.p, list.data(), list.size() * sizeof(RefVoxel), cudaMemcpyHostToDevice, st));
        TTM_CUDA_TRY(cudaMemcpyAsync(d_offs.p, offs.data(), offs.size() * sizeof(int), cudaMemcpyHostToDevice, st));
        TTM_CUDA_TRY(cudaMemcpyAsync(d_peaks.p, h_peaks, (size_t)P * sizeof(int64_t), cudaMemcpyHostToDevice, st));
        k_refine_lncc<<<dim3((unsigned)n_cand, (unsigned)P), kRefThreads, 0, st>>>(
            p.g32.as<float>(), p.w.as<float>(), d_orient, tp32.as<float2>(), d_list.as<RefVoxel>(), (int)list.size(),
            d_peaks.as<int64_t>(), d_offs.as<int>(), n_cand, geo, d_c.as<double>(), d_q.as<float4>());
        TTM_LAUNCH_CHECK();
        k_refine_pick<<<(unsigned)ceil_div(P, 8), 256, 0, st>>>(d_c.as<double>(), d_q.as<float4>(), n_cand, P,
                                                               d_pick.as<RefPick>());
        TTM_LAUNCH_CHECK();
        std::vector<RefPick> pick((size_t)P);
        TTM_CUDA_TRY(cudaMemcpyAsync(pick.data(), d_pick.p, (size_t)P * sizeof(RefPick), cudaMemcpyDeviceToHost, st));
        TTM_CUDA_TRY(cudaStreamSynchronize(st));
        for (int i = 0; i < P; i++) {
            const int best = pick[i].j;
            const int64_t v = h_peaks[i];
            const int x = (int)(v % p.X), y = (int)((v / p.X) % p.Y), z = (int)(v / ((int64_t)p.X * p.Y));
            h_idx[i] = ((int64_t)(z + offs[3 * best]) * p.Y + (y + offs[3 * best + 1])) * p.X + (x + offs[3 * best + 2]);
            h_quat[4 * i] = pick[i].q.x;
            h_quat[4 * i + 1] = pick[i].q.y;
            h_quat[4 * i + 2] = pick[i].q.z;
            h_quat[4 * i + 3] = pick[i].q.w;
            h_lncc[i] = pick[i].c;
        }
        return TTM_OK;
    } catch (const Error& e) {
        return (ttm_status)fail(plan->ctx, e);
    }
}
