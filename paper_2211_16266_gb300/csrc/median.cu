// Median post-filter of a depth map (paper Sec. III-C, item 2: a median
// filter runs over a copy of the depth image and ranges that deviate from the
// filtered copy by more than a threshold are removed).
//
// For a pixel with range d > 0, the valid ranges (> 0) of its (2R+1)^2
// window (columns wrapped at the seam, rows outside the panorama left out)
// are sorted and the lower median m, the element of rank floor((n-1)/2), is
// taken; d is removed when |d - m| > tau * m in FP32. Every decision reads the
// unfiltered input, so the output buffer must not alias it.
//
// The decision needs no median. In order of value the window's valid ranges are
// those that would be too low a median for d, those that would keep it, and those
// that would be too high, so d stays exactly if the median's rank falls among the
// middle ones: if at most `rank` are too low and at most n - 1 - rank too high.
// (Too low: fl(d - x) falls and fl(tau x) rises with x. Too high, for tau <= 1/4:
// x - d is exact up to 2 d and grows faster than fl(tau x), by more than its
// rounding as ulp(tau x) <= ulp(x) / 4; beyond 2 d it exceeds x / 2.) Counting is
// five FP32-pipe instructions per entry, each entry's comparison a multiply-add
// that saturates to 0 or 1, where sorting takes 191 compare-exchanges of two
// instructions on the half-rate pipe for the 25 of a 5x5 window. A thread serves
// four pixels of a column, so an entry is loaded and scaled once for up to four.
// Bound by FP32 issue (74 % of the slots; 255 instructions per pixel, 180 of them on
// that pipe): 1920x960, 5x5: 40.8 -> 18.3 us, against 2.2 us for its 15 MB.
//
// Blocks that hold a valid range outside [2^-30, 2^30], where the scaled
// comparison could lose its sign, and calls with tau > 1/4 sort: invalid entries
// as +inf, Batcher's odd-even merge network (fixed compare-exchange sequence,
// unrolled, so the values never leave registers), the median picked by rank.
// Both are exact: the result equals a plain sort bit for bit.
#include "common.cuh"

namespace pmsp {

namespace {

constexpr int MT_W = 32, MT_H = 8, MT_V = 4;  // threads of a block, pixels of a thread (one column)

constexpr int pow2_at_least(int n) {
    int p = 1;
    while (p < n) p <<= 1;
    return p;
}

// Batcher's odd-even merge sort network on N = 2^m keys: the compare-exchange
// pairs in order, built at compile time so every register index is a constant.
template <int N>
struct MergeNetwork {
    static constexpr int size() {
        int c = 0;
        for (int p = 1; p < N; p <<= 1)
            for (int k = p; k >= 1; k >>= 1)
                for (int j = k % p; j + k < N; j += 2 * k)
                    for (int i = 0; i < k && i + j + k < N; ++i)
                        if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) ++c;
        return c;
    }
    int lo[size()], hi[size()];
    constexpr MergeNetwork() : lo(), hi() {
        int c = 0;
        for (int p = 1; p < N; p <<= 1)
            for (int k = p; k >= 1; k >>= 1)
                for (int j = k % p; j + k < N; j += 2 * k)
                    for (int i = 0; i < k && i + j + k < N; ++i)
                        if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) {
                            lo[c] = i + j;
                            hi[c] = i + j + k;
                            ++c;
                        }
    }
};

template <int N>
__device__ __forceinline__ void odd_even_merge_sort(float (&a)[N]) {
    constexpr MergeNetwork<N> net{};
#pragma unroll
    for (int c = 0; c < MergeNetwork<N>::size(); ++c) {
        const float x = a[net.lo[c]], y = a[net.hi[c]];
        a[net.lo[c]] = fminf(x, y);
        a[net.hi[c]] = fmaxf(x, y);
    }
}

// Output of the pixel whose window starts at `win` (row pitch SW), by sorting.
template <int R, int SW>
__device__ __forceinline__ float median_sorted(const float* win, float tau) {
    constexpr int K = (2 * R + 1) * (2 * R + 1);
    constexpr int N = pow2_at_least(K);
    const float d = win[R * SW + R];
    float a[N];
    int n = 0;
#pragma unroll
    for (int dy = 0; dy <= 2 * R; ++dy)
#pragma unroll
        for (int dx = 0; dx <= 2 * R; ++dx) {
            const float x = win[dy * SW + dx];
            const bool ok = x > 0.f;
            a[dy * (2 * R + 1) + dx] = ok ? x : __int_as_float(0x7f800000);
            n += ok;
        }
#pragma unroll
    for (int k = K; k < N; ++k) a[k] = __int_as_float(0x7f800000);
    odd_even_merge_sort<N>(a);
    const int rank = (n - 1) >> 1;
    float m = a[0];
#pragma unroll
    for (int k = 1; k < K; ++k)
        if (k == rank) m = a[k];
    const float diff = fabsf(__fsub_rn(d, m)), lim = __fmul_rn(tau, m);
    return diff > lim ? 0.f : d;
}

template <int R>
__global__ void __launch_bounds__(MT_W * MT_H) median_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                           int W, int H, float tau) {
    constexpr int TH = MT_H * MT_V, SW = MT_W + 2 * R, SH = TH + 2 * R;
    constexpr float BIG = 1.2089258e24f;  // 2^80
    __shared__ float tile[SH * SW];       // NaN: no valid range
    const int x0 = blockIdx.x * MT_W, y0 = blockIdx.y * TH;
    const int tid = threadIdx.y * MT_W + threadIdx.x;
    bool odd = tau > 0.25f;
    for (int k = tid; k < SH * SW; k += MT_W * MT_H) {
        const int sy = k / SW, sx = k - sy * SW;
        const int y = y0 + sy - R;
        int x = x0 + sx - R;
        if (W >= SW) {
            x = x < 0 ? x + W : (x >= W ? x - W : x);
        } else {
            x %= W;
            if (x < 0) x += W;
        }
        const float v = (y >= 0 && y < H) ? in[(size_t)y * W + x] : 0.f;  // rows outside: no value
        tile[k] = v > 0.f ? v : __int_as_float(0x7fffffff);
        odd = odd || (v > 0.f && !(v >= 9.3132257e-10f && v <= 1.0737418e9f));
    }
    odd = __syncthreads_or(odd);
    const int u = x0 + threadIdx.x, v0 = y0 + threadIdx.y * MT_V;
    if (u >= W || v0 >= H) return;
    const float* win = tile + threadIdx.y * MT_V * SW + threadIdx.x;  // of the thread's first pixel
    float d[MT_V];
#pragma unroll
    for (int p = 0; p < MT_V; ++p) d[p] = win[(p + R) * SW + R];
    float res[MT_V];
    if (odd) {
#pragma unroll 1
        for (int p = 0; p < MT_V; ++p) {
            float r = 0.f;
            if (v0 + p < H && win[(p + R) * SW + R] > 0.f) r = median_sorted<R, SW>(win + p * SW, tau);
            if (v0 + p < H) out[(size_t)(v0 + p) * W + u] = r;
        }
        return;
    }
    float n[MT_V], low[MT_V], high[MT_V];  // valid entries; too low, too high ones (whole numbers)
#pragma unroll
    for (int p = 0; p < MT_V; ++p) n[p] = low[p] = high[p] = 0.f;
#pragma unroll
    for (int r = 0; r < MT_V + 2 * R; ++r) {
        float row_n = 0.f;
#pragma unroll
        for (int c = 0; c <= 2 * R; ++c) {
            const float x = win[r * SW + c];
            row_n += __saturatef(x * BIG);
            const float lim = __fmul_rn(tau, x) * -BIG;
#pragma unroll
            for (int p = 0; p < MT_V; ++p)
                if (r >= p && r <= p + 2 * R) {
                    const float s = __fsub_rn(d[p], x);
                    low[p] += __saturatef(fmaf(s, BIG, lim));
                    high[p] += __saturatef(fmaf(s, -BIG, lim));
                }
        }
#pragma unroll
        for (int p = 0; p < MT_V; ++p)
            if (r >= p && r <= p + 2 * R) n[p] += row_n;
    }
#pragma unroll
    for (int p = 0; p < MT_V; ++p) {
        const float rank = floorf(0.5f * (n[p] - 1.0f));
        res[p] = d[p] > 0.f && low[p] <= rank && high[p] <= n[p] - 1.0f - rank ? d[p] : 0.f;
        if (v0 + p < H) out[(size_t)(v0 + p) * W + u] = res[p];
    }
}

}  // namespace

cudaError_t launch_median_kernel(const float* in, float* out, int W, int H, int radius, float tau,
                                 cudaStream_t stream) {
    const dim3 block(MT_W, MT_H), grid((W + MT_W - 1) / MT_W, (H + MT_H * MT_V - 1) / (MT_H * MT_V));
    switch (radius) {
        case 1: median_kernel<1><<<grid, block, 0, stream>>>(in, out, W, H, tau); break;
        case 2: median_kernel<2><<<grid, block, 0, stream>>>(in, out, W, H, tau); break;
        case 3: median_kernel<3><<<grid, block, 0, stream>>>(in, out, W, H, tau); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace pmsp
