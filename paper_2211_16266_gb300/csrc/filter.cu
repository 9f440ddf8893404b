// Geometric-consistency filter kernel and the standalone camera-model kernels
// (bilinear fetch, projection) behind pmsp_sample_bilinear and pmsp_project.
//
// Paper Sec. III: once five depth maps are available the current one is
// checked against its neighbours' depth maps and outliers are removed. A
// reference pixel with range d is lifted to 3-D, projected into neighbour j,
// the range stored at the nearest pixel there is lifted back and reprojected
// into the reference; the view agrees if the reprojection error (longitude
// difference wrapped to half a panorama) is below max_px. The pixel keeps
// its range when at least min_views views agree. FP32.
//
// Bound by FP32 issue: two projections (four arctangents) and a bearing per pixel
// and neighbour, against 4 bytes read. The bearing needs sines and cosines of the
// neighbour pixel's row and column only, so each block tabulates them once, for
// every panorama size among the maps (usually one: 23 KB at 1920x960), and walks
// the image with a fixed grid, each warp taking 32 pixels of a row at a time. 1920x960
// against 4 maps, a call alone: 79.7 -> 69.8 us with the tables, 64.9 with the wrap and
// the distance as comparisons, 61.5 by warps (the rows in strips of 512 left warps idle
// at most widths), against 7.6 us for its 52 MB. Among other calls: 75.7 -> 57.3 us; 514x257
// and 8 maps 19.3 -> 11.4.
#include <algorithm>

#include "camera.cuh"
#include "common.cuh"
#include "filter_thresholds.h"

namespace pmsp {

__device__ __forceinline__ float3 apply(const float* R, const float* t, float3 X) {
    return make_float3(fmaf(R[0], X.x, fmaf(R[1], X.y, fmaf(R[2], X.z, t[0]))),
                       fmaf(R[3], X.x, fmaf(R[4], X.y, fmaf(R[5], X.z, t[1]))),
                       fmaf(R[6], X.x, fmaf(R[7], X.y, fmaf(R[8], X.z, t[2]))));
}

constexpr int FILTER_WARPS = 16, FILTER_THREADS = 32 * FILTER_WARPS, FILTER_BLOCKS = 3;  // resident blocks per SM
// Shared memory of the bearing tables in all, for the resident blocks to fit an SM. Maps whose
// sizes need more get their bearings computed per pixel.
constexpr size_t FILTER_TABLE_BYTES = 72 * 1024;

// (sin, cos) of the latitudes of a panorama's rows, then of the longitudes of its
// columns, by the expressions of pixel_bearing; table 0 is the reference's.
struct FilterTables {
    int W[PMSP_MAX_SOURCES + 1], H[PMSP_MAX_SOURCES + 1];  // panorama size of each table
    int at[PMSP_MAX_SOURCES + 1];                          // its offset (float2)
    int of[PMSP_MAX_SOURCES];                              // table of each neighbour
    int n;
};

template <bool TABLES>
__global__ void __launch_bounds__(FILTER_THREADS, FILTER_BLOCKS)
    filter_kernel(const __grid_constant__ FilterParams P, const __grid_constant__ FilterTables T) {
    extern __shared__ float2 bearings[];
    if constexpr (TABLES) {
        for (int t = 0; t < T.n; ++t)
            for (int k = threadIdx.x; k < T.H[t] + T.W[t]; k += blockDim.x) {
                float sn, cs;
                if (k < T.H[t])
                    sincospif(0.5f - (2.0f * k + 1.0f) / (2.0f * T.H[t]), &sn, &cs);
                else
                    sincospif((2.0f * (k - T.H[t]) + 1.0f) / T.W[t] - 1.0f, &sn, &cs);
                bearings[T.at[t] + k] = make_float2(sn, cs);
            }
        __syncthreads();
    }
    auto bearing = [&](int t, int u, int v, int W, int H) {
        if constexpr (TABLES) {
            const float2 r = bearings[T.at[t] + v], c = bearings[T.at[t] + H + u];
            return make_float3(r.y * c.x, -r.x, r.y * c.y);
        } else {
            return pixel_bearing(u, v, W, H);
        }
    };
    // a warp takes 32 pixels of a row at a time
    const int strips = (P.W + 31) / 32, warps = blockDim.x >> 5;
    const float su = P.W * 0.15915494309189535f, ou = 0.5f * P.W - 0.5f;
    const float sv = -P.H * 0.3183098861837907f, ov = 0.5f * P.H - 0.5f;
    for (int w = blockIdx.x * warps + (threadIdx.x >> 5); w < strips * P.H; w += gridDim.x * warps) {
        const int y = w / strips, x = (w - y * strips) * 32 + (threadIdx.x & 31);
        if (x >= P.W) continue;
        const size_t i = (size_t)y * P.W + x;
        const float d = P.depth_in[i];
        int cnt = 0;
        if (d > 0.f) {
            const float3 rp = bearing(0, x, y, P.W, P.H);
            const float3 X = make_float3(d * rp.x, d * rp.y, d * rp.z);
            for (int j = 0; j < P.n; ++j) {
                const FilterView& V = P.nb[j];
                const float3 Y = apply(V.Rf, V.tf, X);
                float uc, vc;
                project_dir_fast(Y.x, Y.y, Y.z, V.su, V.ou, V.sv, V.ov, uc, vc);
                // |lon| <= pi: the rounded column lies within one of [0, W)
                int ui = (int)floorf(uc + 0.5f);
                ui = ui < 0 ? ui + V.W : (ui >= V.W ? ui - V.W : ui);
                ui = clamp_index(ui, V.W - 1);
                const int vi = clamp_index((int)floorf(vc + 0.5f), V.H - 1);
                const float dj = V.depth[(size_t)vi * V.W + ui];
                if (!(dj > 0.f)) continue;
                const float3 rq = bearing(T.of[j], ui, vi, V.W, V.H);
                const float3 Z = apply(V.Rb, V.tb, make_float3(dj * rq.x, dj * rq.y, dj * rq.z));
                float u2, v2;
                project_dir_fast(Z.x, Z.y, Z.z, su, ou, sv, ov, u2, v2);
                float du = u2 - (float)x;
                du = du >= P.wrap_hi ? du - P.W : (du < P.wrap_lo ? du + P.W : du);  // into half a panorama
                const float dv = v2 - (float)y;
                if (du * du + dv * dv < P.max_sq) ++cnt;  // the distance is below max_px
            }
        }
        P.depth_out[i] = (d > 0.f && cnt >= P.min_views) ? d : 0.f;
        if (P.agree) P.agree[i] = cnt;
    }
}

cudaError_t launch_filter_kernel(const FilterParams& params, cudaStream_t stream) {
    FilterParams p = params;
    const FilterThresholds at = filter_thresholds(p.W, p.max_px);
    p.wrap_hi = at.wrap_hi;
    p.wrap_lo = at.wrap_lo;
    p.max_sq = at.max_sq;
    for (int j = 0; j < p.n; ++j) {
        FilterView& V = p.nb[j];
        V.su = V.W * 0.15915494309189535f;
        V.ou = 0.5f * V.W - 0.5f;
        V.sv = -V.H * 0.3183098861837907f;
        V.ov = 0.5f * V.H - 0.5f;
    }
    FilterTables T{};
    size_t entries = 0;
    auto table_of = [&](int W, int H) {
        for (int t = 0; t < T.n; ++t)
            if (T.W[t] == W && T.H[t] == H) return t;
        T.W[T.n] = W;
        T.H[T.n] = H;
        T.at[T.n] = (int)entries;
        entries += (size_t)W + H;
        return T.n++;
    };
    table_of(p.W, p.H);
    for (int j = 0; j < p.n; ++j) T.of[j] = table_of(p.nb[j].W, p.nb[j].H);
    const size_t bytes = entries * sizeof(float2);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // Strips of 32 pixels, FILTER_WARPS of them at a time in a resident block; where there are
    // fewer than the resident warps, smaller blocks on more SMs.
    const long long strips = (long long)((p.W + 31) / 32) * p.H, resident = (long long)FILTER_BLOCKS * sms;
    const int warps = (int)std::min<long long>(FILTER_WARPS, (strips + resident - 1) / resident);
    const long long blocks = std::min(resident, (strips + warps - 1) / warps);
    // A block's tables cost as many bearings as the sizes have rows and columns: they
    // pay where a block has that many pixel-neighbours to look up (us a call, direct and
    // tabulated: 1920x960 and 1 map, 1.4 look-ups an entry, 25.7 and 21.8; 960x480 and
    // 1 map, 0.7, 7.8 and 7.5; 256x128 and 4 maps, 0.75, 4.7 and 4.9).
    const long long per_block = (long long)p.W * p.H * p.n / blocks;
    if (bytes <= FILTER_TABLE_BYTES && per_block >= (long long)entries) {
        if (bytes > 48 * 1024) {
            e = cudaFuncSetAttribute(filter_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FILTER_TABLE_BYTES);
            if (e != cudaSuccess) return e;
        }
        filter_kernel<true><<<(unsigned)blocks, 32 * warps, bytes, stream>>>(p, T);
    } else {
        // (nothing to share: blocks of up to 4 warps, whose slots are free again sooner; 1920x960
        // and 1 map 25.7 us, of 16 warps 26.9)
        const int few = std::min(warps, 4);
        filter_kernel<false><<<(unsigned)std::min<long long>((strips + few - 1) / few, 1ll << 30), 32 * few, 0, stream>>>(p, T);
    }
    return cudaGetLastError();
}

__global__ void sample_kernel(cudaTextureObject_t tex, float inv_w, float inv_h, int n, const float* uc,
                              const float* vc, float* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = sample_bilinear(tex, inv_w, inv_h, uc[i], vc[i]);
}

cudaError_t launch_sample_kernel(cudaTextureObject_t tex, int W, int H, int n, const float* uc,
                                 const float* vc, float* out, cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    sample_kernel<<<(n + 255) / 256, 256, 0, stream>>>(tex, 1.0f / W, 1.0f / H, n, uc, vc, out);
    return cudaGetLastError();
}

__global__ void project_kernel(int n, const float* dirs, float su, float ou, float sv, float ov, float* uc,
                               float* vc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) project_dir_fast(dirs[3 * i], dirs[3 * i + 1], dirs[3 * i + 2], su, ou, sv, ov, uc[i], vc[i]);
}

cudaError_t launch_project_kernel(int W, int H, int n, const float* dirs, float* uc, float* vc,
                                  cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    project_kernel<<<(n + 255) / 256, 256, 0, stream>>>(n, dirs, W * 0.15915494309189535f, 0.5f * W - 0.5f,
                                                        -H * 0.3183098861837907f, 0.5f * H - 0.5f, uc, vc);
    return cudaGetLastError();
}

}  // namespace pmsp
