// Per-pixel PatchMatch kernels: matching cost, random initialisation and the
// red-black half-sweep (propagation + refinement), templated on the number
// of source views the thread keeps in registers.
//
// Paper: random initialisation of the plane map (Sec. III-B); parallel
// red-black propagation over an 8-neighbourhood whose inner neighbours sit
// one position further out than in Galliani et al. (Sec. III-C, Fig. 5);
// six random refinement tests on a shrinking range (Sec. III-C, item 1). The
// cost is the bilaterally weighted NCC of the reference patch against its
// reprojection through the plane into every source, averaged over the best k
// views (the cost of the PatchMatch works the paper cites).
//
// Design: one thread per active pixel of a 32x8 tile (one colour per launch),
// blocks walking the image in strips of tile rows. The reference tile with
// its halo, the per-row / per-column bearing terms, the spatial weights and
// (for exactly known view counts) each view pair's rotated column directions
// are staged in shared memory; the sample loop runs over the patch with all
// views innermost, so the plane intersection and the bilateral weight of a
// sample are shared by every view. Views are processed in pairs with packed
// FP32 instructions, the projection in half-angle form (see camera.cuh). Per
// view four FP32 sums are kept: the source intensity is centred on its value
// at the first (centre-most) sample, which keeps the variance term free of
// cancellation. The 8 neighbour candidates and the refinement candidates run
// through one loop with a single inlined copy of the cost.
#pragma once

#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "camera.cuh"
#include "common.cuh"
#include "philox.cuh"
#include "sweep_policy.h"

namespace pmsp {

static __constant__ int c_neighbors[2][8][2] = {
    {{0, -3}, {0, 3}, {-3, 0}, {3, 0}, {0, -5}, {0, 5}, {-5, 0}, {5, 0}},
    {{0, -1}, {0, 1}, {-1, 0}, {1, 0}, {0, -5}, {0, 5}, {-5, 0}, {5, 0}}};


// Resident blocks per SM the batched kernel's register budget is sized for,
// by its largest view count (its per-view-count variants share one budget).
constexpr int min_blocks_for(int ns) { return ns <= 4 ? 8 : ns <= 6 ? 7 : ns <= 8 ? 6 : ns <= 10 ? 5 : 4; }

// Resident blocks per SM of the single-keyframe kernels, by view count:
// 5 (96 registers) up to 4 views, 4 (128) for 5-8 views, 3 (168) for 9-10
// and 4 beyond (the compiler left alone takes up to 246). Each tier is the
// fastest of 3-7 blocks on 1920x960 half-sweeps: fewer, spill-free threads
// beat more resident warps once the per-view sums fill the registers.
constexpr int pixel_min_blocks(int ns) { return ns <= 4 ? 5 : ns <= 8 ? 4 : ns <= 10 ? 3 : 4; }

// Reference-side constants of one pixel (independent of the hypothesis).
struct RefStats {
    float Ip;    // centre intensity
    float mu;    // weighted mean of the samples
    float Sw;    // sum of weights
    float SIc;   // sum w (I - mu)   (zero up to rounding)
    float varI;  // Sw * sum w (I - mu)^2 - SIc^2
};

// Per-block scratch of the half-sweep's pooled candidate evaluation, for a block
// of N pixels: each pixel's reference statistics and the minimum (cost, candidate) key of its
// neighbour candidates, and per warp the list of (pixel, candidate) pairs that
// need a cost evaluation.
template <int N>
struct SweepPool {
    unsigned long long key[N];
    RefStats st[N];
    unsigned char item[BLOCK_THREADS / 32][N * 8 / (BLOCK_THREADS / 32)];
};
struct NoPool {};

// Further scratch of the bounded half-sweep (sweep_bounded): the bearing tables as
// float2, the neighbours' FP32 bearings, each pixel's incumbent, how far a bound
// must clear it, the random steps of its refinement tests (of the inverse range and
// the normal, scaled), the costs of the tests under way, and the window's samples
// in the order they are taken (the centre-most first, then row-major). MAX_DRAWN
// tests are drawn ahead, the paper's six; further ones are drawn when they start.
// At most MAX_AHEAD tests of a pixel are under way.
constexpr int MAX_DRAWN = 6, MAX_AHEAD = 2;
constexpr int MAX_REACH = 5;  // of a neighbour candidate (c_neighbors)
// (Byte offsets in the reference tile and in the tables of float2 rows and
// columns, and the spatial log2-weight: 16 bytes, or 8 where a window has many.)
struct WindowSample {
    int ref_at, row_at, col_at;
    float wsp;
    __device__ __forceinline__ static WindowSample at(int pitch, int dy, int dx, float wsp) {
        return WindowSample{4 * (dy * pitch + dx), 8 * dy, 8 * dx, wsp};
    }
    __device__ __forceinline__ int ref() const { return ref_at; }
    __device__ __forceinline__ int row() const { return row_at; }
    __device__ __forceinline__ int col() const { return col_at; }
};
struct PackedSample {
    short ref_at;
    signed char dy, dx;
    float wsp;
    __device__ __forceinline__ static PackedSample at(int pitch, int dy, int dx, float wsp) {
        return PackedSample{(short)(4 * (dy * pitch + dx)), (signed char)dy, (signed char)dx, wsp};
    }
    __device__ __forceinline__ int ref() const { return ref_at; }
    __device__ __forceinline__ int row() const { return 8 * dy; }
    __device__ __forceinline__ int col() const { return 8 * dx; }
};
template <int TW, int TH, int HALO, int SAMPLES>
struct BoundPool {
    static constexpr int N = (TW / 2) * TH;
    float2 row[TH + 2 * HALO], col[TW + 2 * HALO];  // (cos, sin) latitude, (sin, cos) longitude of the tile
    float2 near_row[TH + 2 * MAX_REACH], near_col[TW + 2 * MAX_REACH];  // (sin, cos), as pixel_bearing
    float d[N], inv_d[N], nx[N], ny[N], nz[N], cost[N];
    float margin[N];
    float draw[MAX_DRAWN][4][N];
    float result[MAX_AHEAD][N];
    unsigned char version[N];  // counts the incumbents; a test of an older one is void
    unsigned char taken[N];    // refinement results taken up
    unsigned offer[BLOCK_THREADS];
    using Sample = typename std::conditional<(SAMPLES <= 64), WindowSample, PackedSample>::type;
    alignas(16) Sample sample[SAMPLES];
};

// Shared memory of one tile of TW x TH reference pixels with a halo of HALO
// pixels on each side (the window radius the tile serves: the largest, or
// that of a fixed-window instance); every shape has (TW / 2) x TH pixels of
// one colour and TPP threads per pixel, 128 threads in all.
template <int TW, int TH, int TPP = 1, int HALO = MAX_HALO, bool POOL = TPP == 1, bool BOUND = false>
struct TileSmemT {
    static constexpr int W = TW, H = TH, LANES = TPP;
    static constexpr int PITCH = TW + 2 * HALO, ROWS = TH + 2 * HALO;
    static constexpr int THREADS = (TW / 2) * TH;
    static_assert(THREADS * TPP == BLOCK_THREADS, "every tile shape runs 128 threads");
    static_assert(HALO >= 0 && HALO <= MAX_HALO, "halo within the largest window");
    float ref[ROWS * PITCH];             // normalised intensities, halo included
    float row_cos[ROWS], row_sin[ROWS];  // cos lat, sin lat
    float col_sin[PITCH], col_cos[PITCH];  // sin lon, cos lon
    float wsp[2 * HALO + 1];             // spatial log2-weight of offset index k
    // candidate pooling of the one-thread-per-pixel half-sweep
    typename std::conditional<POOL, SweepPool<THREADS>, NoPool>::type pool;
    // the bounded half-sweep's (36 samples at 11x11 / 2, (2 HALO + 1)^2 at most)
    static constexpr int SAMPLES = HALO == 5 ? 36 : (2 * HALO + 1) * (2 * HALO + 1);
    typename std::conditional<BOUND, BoundPool<TW, TH, HALO, SAMPLES>, NoPool>::type bound;
};
using TileSmem = TileSmemT<TILE_W, TILE_H>;  // the batched and no-alloc kernels' shape

// Tile shapes of the single-keyframe half-sweep, chosen by PixelParams::tile.
template <int TS, int HALO = MAX_HALO, bool POOL = true> struct TileShape { using Smem = TileSmemT<32, 8, 1, HALO, POOL>; };
template <int HALO, bool POOL> struct TileShape<1, HALO, POOL> { using Smem = TileSmemT<64, 4, 1, HALO, POOL>; };
template <int HALO, bool POOL> struct TileShape<2, HALO, POOL> { using Smem = TileSmemT<16, 16, 1, HALO, POOL>; };
// 2, 4 and 8 lanes per pixel, for keyframes of few tiles (sweep_shape).
template <int HALO, bool POOL> struct TileShape<3, HALO, POOL> { using Smem = TileSmemT<32, 4, 2, HALO, POOL>; };
template <int HALO, bool POOL> struct TileShape<4, HALO, POOL> { using Smem = TileSmemT<16, 4, 4, HALO, POOL>; };
template <int HALO, bool POOL> struct TileShape<5, HALO, POOL> { using Smem = TileSmemT<8, 4, 8, HALO, POOL>; };

// Rotated column directions of the paired path: for view pair q and tile
// column c, colU[q][k][c] = row k of R_s applied to (sin lon_c, 0, cos lon_c)
// for both views of the pair. A sample direction r = (cl sin, -sl, cl cos)
// then transforms as R r = cl U_c - sl R_col1. One table per kernel, sized by the
// tile's columns (PITCH, halo included) and by the view pairs: the kernels of one
// view count hold exactly theirs (every KB given up here is texture cache), the
// batched kernel, whose view counts share one table, five for up to 10 views.
constexpr int MAX_COL_PAIRS = 5;

template <int CAP, int PITCH>
__device__ __forceinline__ auto& col_array() {
    __shared__ float2 t[CAP][3][PITCH];
    return t;
}

struct ParamViews;
template <int NP, class VA, int PITCH>
__device__ __forceinline__ auto& col_table() {
    return col_array<std::is_same<VA, ParamViews>::value ? NP : MAX_COL_PAIRS, PITCH>();
}

// Loads of read-only shared memory (written before a barrier) at a 32-bit shared
// address, with the offsets in the instruction. Volatile, so that they are not
// moved across a barrier.
__device__ __forceinline__ unsigned shared_at(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float shared_f(unsigned a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
template <int OFFSET = 0>
__device__ __forceinline__ float2 shared_f2(unsigned a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "r"(a), "n"(OFFSET));
    return v;
}

// Sample window of the paired cost loop: WIN 0 reads the window from the
// parameters; the fixed windows make the loop bounds and offsets constants
// (3 % faster half-sweeps at 11x11 / 2). WIN 1: 11x11 sampled at stride 2
// (6 x 6 samples, radius 5); WIN 2: 7x7 dense (7 x 7, radius 3).
template <int WIN>
struct Window {
    static constexpr int HALO = MAX_HALO;  // the tile halo the instance needs
    __device__ static int K(const PixelParams& P) { return P.K; }
    __device__ static int R(const PixelParams& P) { return P.radius; }
    __device__ static int stride(const PixelParams& P) { return P.stride; }
};
template <>
struct Window<1> {
    static constexpr int HALO = 5;
    __device__ static constexpr int K(const PixelParams&) { return 6; }
    __device__ static constexpr int R(const PixelParams&) { return 5; }
    __device__ static constexpr int stride(const PixelParams&) { return 2; }
};
template <>
struct Window<2> {
    static constexpr int HALO = 3;
    __device__ static constexpr int K(const PixelParams&) { return 7; }
    __device__ static constexpr int R(const PixelParams&) { return 3; }
    __device__ static constexpr int stride(const PixelParams&) { return 1; }
};


__device__ __forceinline__ float load_ref(const PixelParams& P, int x, int y) {
    const uint8_t* row = P.ref + (int64_t)y * P.ref_pitch;
    if (P.ref_format == PMSP_U8) return (float)row[x] * (1.0f / 255.0f);
    if (P.ref_format == PMSP_F16) return __half2float(reinterpret_cast<const __half*>(row)[x]);
    return reinterpret_cast<const float*>(row)[x];
}

template <class SM>
__device__ __forceinline__ void stage_tile(const PixelParams& P, SM& sm, int bx, int by) {
    const int R = P.radius;
    const int rows = SM::H + 2 * R, cols = SM::W + 2 * R;
    for (int i = threadIdx.x; i < rows * cols; i += BLOCK_THREADS) {
        const int ly = i / cols, lx = i - ly * cols;
        const int gy = clamp_index(by - R + ly, P.H - 1);
        const int gx = wrap_index(bx - R + lx, P.W);
        sm.ref[ly * SM::PITCH + lx] = load_ref(P, gx, gy);
    }
    // Bearing tables in FP64, rounded once to FP32. An FP32 angle argument
    // (2 gx + 1) / W - 1 is itself rounded by up to 6e-8 near 1, i.e. pi x 6e-8
    // = 1.9e-7 rad of direction error per column, 1.1e-4 px at 3840 px: that,
    // not the projection, was the largest error of the matching cost at that
    // size. A block computes at most 2 x (TILE + 2 x halo) entries, so the FP64
    // cost is negligible.
    for (int i = threadIdx.x; i < rows; i += BLOCK_THREADS) {
        const int gy = clamp_index(by - R + i, P.H - 1);
        double s, c;
        sincospi(0.5 - (2.0 * gy + 1.0) / (2.0 * P.H), &s, &c);
        sm.row_sin[i] = (float)s;
        sm.row_cos[i] = (float)c;
    }
    for (int i = threadIdx.x; i < cols; i += BLOCK_THREADS) {
        const int gx = wrap_index(bx - R + i, P.W);
        double s, c;
        sincospi((2.0 * gx + 1.0) / P.W - 1.0, &s, &c);
        sm.col_sin[i] = (float)s;
        sm.col_cos[i] = (float)c;
    }
    for (int k = threadIdx.x; k < P.K; k += BLOCK_THREADS) {
        const float o = (float)(k * P.stride - R);
        sm.wsp[k] = P.ws * o * o;
    }
}

// Bilateral weight of sample (a, b) with intensity Iq: 2^(wc dI^2 + ws |o|^2).
template <class SM>
__device__ __forceinline__ float bilateral(const PixelParams& P, const SM& sm, int a, int b, float Iq,
                                           float Ip) {
    const float dI = Iq - Ip;
    return exp2_approx(fmaf(P.wc, dI * dI, sm.wsp[a] + sm.wsp[b]));
}

// Local (halo-inclusive) tile coordinates of the pixel: lx, ly.
// SII: sum w (I - mu)^2; w_centre: weight of the centre-most sample.
template <int WIN, class SM>
__device__ __forceinline__ RefStats ref_stats(const PixelParams& P, const SM& sm, int lx, int ly, float& SII,
                                              float& w_centre) {
    RefStats st;
    st.Ip = sm.ref[ly * SM::PITCH + lx];
    const int K = Window<WIN>::K(P), R = Window<WIN>::R(P), stp = Window<WIN>::stride(P);
    float Sw = 0.f, SI = 0.f;
    for (int a = 0; a < K; ++a) {
        const float* row = sm.ref + (ly + a * stp - R) * SM::PITCH + lx - R;
        for (int b = 0; b < K; ++b) {
            const float Iq = row[b * stp];
            const float w = bilateral(P, sm, a, b, Iq, st.Ip);
            Sw += w;
            SI = fmaf(w, Iq, SI);
        }
    }
    st.Sw = Sw;
    st.mu = SI / Sw;
    float SIc = 0.f, SIIc = 0.f;
    for (int a = 0; a < K; ++a) {
        const float* row = sm.ref + (ly + a * stp - R) * SM::PITCH + lx - R;
        for (int b = 0; b < K; ++b) {
            const float Iq = row[b * stp];
            const float w = bilateral(P, sm, a, b, Iq, st.Ip);
            const float Ic = Iq - st.mu;
            SIc = fmaf(w, Ic, SIc);
            SIIc = fmaf(w * Ic, Ic, SIIc);
        }
    }
    st.SIc = SIc;
    st.varI = mul_sub(Sw, SIIc, SIc, SIc);
    SII = SIIc;
    const int ac = K >> 1, o = ac * stp - R;
    w_centre = bilateral(P, sm, ac, ac, sm.ref[(ly + o) * SM::PITCH + lx + o], st.Ip);
    return st;
}

template <class SM>
__device__ __forceinline__ RefStats ref_stats(const PixelParams& P, const SM& sm, int lx, int ly) {
    float SII, w_centre;
    return ref_stats<0>(P, sm, lx, ly, SII, w_centre);
}

// Where the per-view constants are read from. Kernel parameters: plain member
// reads (they become constant-bank operands). Shared memory (the batched
// kernel): volatile vector loads at every use, so the compiler reloads them
// instead of holding all views' constants in registers.
struct ParamViews {
    // Reads go straight to the parameter at each use, so they stay
    // constant-bank operands of the arithmetic instead of register copies.
    struct Loaded {
        const SourceView& V;
        __device__ __forceinline__ float r(int k) const { return V.R[k]; }
        __device__ __forceinline__ float t(int k) const { return V.t[k]; }
        __device__ __forceinline__ float su() const { return V.su; }
        __device__ __forceinline__ float ou() const { return V.ou; }
        __device__ __forceinline__ float sv() const { return V.sv; }
        __device__ __forceinline__ float ov() const { return V.ov; }
        __device__ __forceinline__ float inv_w() const { return V.inv_w; }
        __device__ __forceinline__ float inv_h() const { return V.inv_h; }
        __device__ __forceinline__ cudaTextureObject_t tex() const { return V.tex; }
    };
    __device__ __forceinline__ static Loaded load(const SourceView& V) { return Loaded{V}; }
};

struct SharedViews {
    __device__ __forceinline__ static float4 ld4(const float4* p) {
        float4 v;
        const unsigned a = (unsigned)__cvta_generic_to_shared(p);
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
        return v;
    }
    // The 80-byte view as 20 words: tex (2), R (9), t (3), su, ou, sv, ov, inv_w, inv_h.
    struct Loaded {
        float w[20];
        __device__ __forceinline__ float r(int k) const { return w[2 + k]; }
        __device__ __forceinline__ float t(int k) const { return w[11 + k]; }
        __device__ __forceinline__ float su() const { return w[14]; }
        __device__ __forceinline__ float ou() const { return w[15]; }
        __device__ __forceinline__ float sv() const { return w[16]; }
        __device__ __forceinline__ float ov() const { return w[17]; }
        __device__ __forceinline__ float inv_w() const { return w[18]; }
        __device__ __forceinline__ float inv_h() const { return w[19]; }
        __device__ __forceinline__ cudaTextureObject_t tex() const {
            return (cudaTextureObject_t)(((unsigned long long)__float_as_uint(w[1]) << 32) | __float_as_uint(w[0]));
        }
    };
    __device__ __forceinline__ static Loaded load(const SourceView& V) {
        Loaded L;
        const float4* q = reinterpret_cast<const float4*>(&V);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const float4 a = ld4(q + k);
            L.w[4 * k] = a.x;
            L.w[4 * k + 1] = a.y;
            L.w[4 * k + 2] = a.z;
            L.w[4 * k + 3] = a.w;
        }
        return L;
    }
};

// The constants of a view pair the paired sample loop reads, and the texture
// of a view. Kernel parameters (ParamViews): member reads at the point of use,
// which become constant-bank operands. Shared memory (SharedViews, the batched
// kernel): volatile 16-byte loads at every sample, so the compiler reloads
// them instead of keeping every pair's constants in registers across the
// sample loop.
template <class VA>
struct PairOf {  // kernel parameters: each constant read where it is used
    const PixelParams::ViewPair& V;
    __device__ __forceinline__ float2 r1() const { return V.R[1]; }
    __device__ __forceinline__ float2 r4() const { return V.R[4]; }
    __device__ __forceinline__ float2 r7() const { return V.R[7]; }
    __device__ __forceinline__ float2 t0() const { return V.t[0]; }
    __device__ __forceinline__ float2 t1() const { return V.t[1]; }
    __device__ __forceinline__ float2 t2() const { return V.t[2]; }
    __device__ __forceinline__ float2 su() const { return V.su; }
    __device__ __forceinline__ float2 nsv() const { return V.nsv; }
    __device__ __forceinline__ float2 inv_w() const { return V.inv_w; }
    __device__ __forceinline__ float2 inv_h() const { return V.inv_h; }
};

template <>
struct PairOf<SharedViews> {  // shared memory: the pair's words loaded once per use of the pair
    float4 a, b, c, d, e, f, g;
    __device__ __forceinline__ explicit PairOf(const PixelParams::ViewPair& V) {
        // ViewPair as 8 16-byte words: (R0 R1) (R2 R3) (R4 R5) (R6 R7) (R8 t0) (t1 t2) (su nsv) (inv_w inv_h)
        const float4* q = reinterpret_cast<const float4*>(&V);
        a = SharedViews::ld4(q);
        b = SharedViews::ld4(q + 2);
        c = SharedViews::ld4(q + 3);
        d = SharedViews::ld4(q + 4);
        e = SharedViews::ld4(q + 5);
        f = SharedViews::ld4(q + 6);
        g = SharedViews::ld4(q + 7);
    }
    __device__ __forceinline__ float2 r1() const { return make_float2(a.z, a.w); }
    __device__ __forceinline__ float2 r4() const { return make_float2(b.x, b.y); }
    __device__ __forceinline__ float2 r7() const { return make_float2(c.z, c.w); }
    __device__ __forceinline__ float2 t0() const { return make_float2(d.z, d.w); }
    __device__ __forceinline__ float2 t1() const { return make_float2(e.x, e.y); }
    __device__ __forceinline__ float2 t2() const { return make_float2(e.z, e.w); }
    __device__ __forceinline__ float2 su() const { return make_float2(f.x, f.y); }
    __device__ __forceinline__ float2 nsv() const { return make_float2(f.z, f.w); }
    __device__ __forceinline__ float2 inv_w() const { return make_float2(g.x, g.y); }
    __device__ __forceinline__ float2 inv_h() const { return make_float2(g.z, g.w); }
};

template <class VA>
__device__ __forceinline__ PairOf<VA> pair_of(const PixelParams::ViewPair& V) {
    if constexpr (std::is_same<VA, SharedViews>::value)
        return PairOf<SharedViews>(V);
    else
        return PairOf<VA>{V};
}

template <class VA>
__device__ __forceinline__ cudaTextureObject_t view_tex(const SourceView& V) {
    if constexpr (std::is_same<VA, SharedViews>::value) {
        unsigned long long t;
        const unsigned a = (unsigned)__cvta_generic_to_shared(&V.tex);
        asm volatile("ld.shared.u64 %0, [%1];" : "=l"(t) : "r"(a));
        return (cudaTextureObject_t)t;
    } else {
        return V.tex;
    }
}

// Intensity of source view V at the projection of reference-frame point X.
template <class VA>
__device__ __forceinline__ float view_sample(const SourceView& V, float X, float Y, float Z) {
    const typename VA::Loaded L = VA::load(V);
    const float Yx = fmaf(L.r(0), X, fmaf(L.r(1), Y, fmaf(L.r(2), Z, L.t(0))));
    const float Yy = fmaf(L.r(3), X, fmaf(L.r(4), Y, fmaf(L.r(5), Z, L.t(1))));
    const float Yz = fmaf(L.r(6), X, fmaf(L.r(7), Y, fmaf(L.r(8), Z, L.t(2))));
    float qu, qv;
    bool front;
    project_dir_half(Yx, Yy, Yz, L.su(), -L.sv(), qu, qv, front);
    return sample_bilinear_half(L.tex(), L.inv_w(), L.inv_h(), qu, qv, front);
}

// Mean of the best_k smallest of NS view costs: odd-even transposition sort,
// then the sum from the smallest up.
template <int NS>
__device__ __forceinline__ float best_mean(const PixelParams& P, float (&cs)[NS]) {
#pragma unroll
    for (int pass = 0; pass < NS; ++pass) {
#pragma unroll
        for (int s = (pass & 1); s + 1 < NS; s += 2) {
            const float lo = fminf(cs[s], cs[s + 1]), hi = fmaxf(cs[s], cs[s + 1]);
            cs[s] = lo;
            cs[s + 1] = hi;
        }
    }
    float sum = 0.f;
#pragma unroll
    for (int s = 0; s < NS; ++s)
        if (s < P.best_k) sum += cs[s];
    return sum / (float)P.best_k;
}

// Cost of plane (range d along rp, unit normal n) at the pixel. Returns 2 for
// an invalid plane (a patch ray meets it from behind or grazing). NS views
// are kept in registers; EXACT means S == NS (no per-view guard).
template <int NS, bool EXACT, class VA, class SM>
__device__ __forceinline__ float plane_cost(const PixelParams& P, const SM& sm, int lx, int ly,
                                            const RefStats& st, float3 rp, float d, float3 n) {
    const float eps = 1e-8f * st.Sw * st.Sw;
    if (st.varI < eps) return 2.0f;
    const float dn = d * dot3(n, rp);
    const int K = P.K, R = P.radius, stp = P.stride;
    const int ac = K >> 1;  // centre-most sample first: its intensity centres each view

    float c0[NS], SJ[NS], SJJ[NS], SIJ[NS];
    {
        const int o = ac * stp - R;
        const float cl = sm.row_cos[ly + o];
        const float3 rq = make_float3(cl * sm.col_sin[lx + o], -sm.row_sin[ly + o], cl * sm.col_cos[lx + o]);
        const float den = dot3(n, rq);
        if (!(den < -1e-6f)) return 2.0f;
        const float t = __fdividef(dn, den);
        const float X = t * rq.x, Y = t * rq.y, Z = t * rq.z;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            c0[s] = 0.f;
            SJ[s] = 0.f;
            SJJ[s] = 0.f;
            SIJ[s] = 0.f;
            if (EXACT || s < P.S) c0[s] = view_sample<VA>(P.src[s], X, Y, Z);
        }
    }
    bool valid = true;
    for (int a = 0; a < K && valid; ++a) {
        const int oy = a * stp - R;
        const float cl = sm.row_cos[ly + oy], msl = -sm.row_sin[ly + oy];
        const float* ref_row = sm.ref + (ly + oy) * SM::PITCH + lx - R;
        for (int b = 0; b < K; ++b) {
            if (a == ac && b == ac) continue;
            const float Iq = ref_row[b * stp];
            const float w = bilateral(P, sm, a, b, Iq, st.Ip);
            const float wI = w * (Iq - st.mu);
            const int cx = lx + b * stp - R;
            const float3 rq = make_float3(cl * sm.col_sin[cx], msl, cl * sm.col_cos[cx]);
            const float den = dot3(n, rq);
            if (!(den < -1e-6f)) {
                valid = false;
                break;
            }
            const float t = __fdividef(dn, den);
            const float X = t * rq.x, Y = t * rq.y, Z = t * rq.z;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                if (EXACT || s < P.S) {
                    const float Jc = view_sample<VA>(P.src[s], X, Y, Z) - c0[s];
                    const float tw = __fmul_rn(w, Jc);
                    SJ[s] = __fadd_rn(SJ[s], tw);
                    SJJ[s] = fmaf(tw, Jc, SJJ[s]);
                    SIJ[s] = fmaf(wI, Jc, SIJ[s]);
                }
            }
        }
    }
    if (!valid) return 2.0f;

    float cs[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        float c = 3.0f;  // unused slots sort last
        if (EXACT || s < P.S) {
            const float varJ = mul_sub(st.Sw, SJJ[s], SJ[s], SJ[s]);
            const float cov = mul_sub(st.Sw, SIJ[s], st.SIc, SJ[s]);
            if (varJ < eps) {
                c = 2.0f;
            } else {
                float ncc = cov * rsqrtf(st.varI * varJ);
                ncc = fminf(1.0f, fmaxf(-1.0f, ncc));
                c = 1.0f - ncc;
            }
        }
        cs[s] = c;
    }
    return best_mean<NS>(P, cs);
}

// Intensities of all NP view pairs (views 2q, 2q + 1) at the sample whose
// reference-frame point is X = t r, r = (cl sin lon_c, -sl, cl cos lon_c) in
// tile column c: the source point R_s X + t_s = alpha U_c + beta R_col1 + t_s
// with alpha = t cl, beta = -t sl and U_c from the column table. The
// projection runs on float2 pairs (one packed instruction for both views of a
// pair), then two gathers and the bilinear weights per pair; the arithmetic
// after the rigid transform is that of project_dir_half and
// sample_bilinear_half, operation for operation. Two phases: each pair's
// source coordinates and, right after them, its two gathers, so a pair's
// gathers are in flight while the next pairs' coordinates are computed; then
// the interpolation of every pair (2 % faster than pair by pair, and issuing
// each pair's gathers before the next pair's coordinates another 1.5 %).
// pairs_columns reads column c's entries of the table from the shared address of
// its first one; the recursion makes every offset a constant.
template <int NP, int PITCH, int Q = 0>
__device__ __forceinline__ void pairs_columns(unsigned col, float2 (&U)[NP][3]) {
    if constexpr (Q < NP) {
        U[Q][0] = shared_f2<8 * PITCH * (3 * Q)>(col);
        U[Q][1] = shared_f2<8 * PITCH * (3 * Q + 1)>(col);
        U[Q][2] = shared_f2<8 * PITCH * (3 * Q + 2)>(col);
        pairs_columns<NP, PITCH, Q + 1>(col, U);
    }
}

// The rest of pairs_sample, from the column's table entries U.
template <int NP, class VA>
__device__ __forceinline__ void pairs_sample_columns(const PixelParams& P, float alpha, float beta, const float2 (&U)[NP][3],
                                                     float2 (&J)[NP]) {
    float2 fx[NP], fy[NP];
    float4 G0[NP], G1[NP];
    const float2 av = pair(alpha), bv = pair(beta);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const auto VP = pair_of<VA>(P.pairs[q]);
        const float2 Yx = fma2(av, U[q][0], fma2(bv, VP.r1(), VP.t0()));
        const float2 Yy = fma2(av, U[q][1], fma2(bv, VP.r4(), VP.t1()));
        const float2 Yz = fma2(av, U[q][2], fma2(bv, VP.r7(), VP.t2()));
        const float2 q2 = fma2(Yx, Yx, mul2(Yz, Yz));
        const float2 rho = make_float2(sqrt_approx(q2.x), sqrt_approx(q2.y));
        const float2 dl = add2(rho, make_float2(fabsf(Yz.x), fabsf(Yz.y)));
        const float2 ql = mul2(Yx, make_float2(rcp_approx(dl.x), rcp_approx(dl.y)));
        const float2 r2 = fma2(Yy, Yy, q2);
        const float2 r3 = make_float2(sqrt_approx(r2.x), sqrt_approx(r2.y));
        const float2 dt = add2(r3, rho);
        const float2 qt = mul2(Yy, make_float2(rcp_approx(dt.x), rcp_approx(dt.y)));
        float2 pl, pt;
        atan2x_poly2_dual(mul2(ql, ql), mul2(qt, qt), pl, pt);
        const float2 al = mul2(ql, pl), nlat = mul2(qt, pt);
        const bool f0 = Yz.x >= 0.f, f1 = Yz.y >= 0.f;
        const float2 qu = fma2(al, make_float2(f0 ? VP.su().x : -VP.su().x, f1 ? VP.su().y : -VP.su().y), pair(0.5f));
        const float2 qv = fma2(nlat, VP.nsv(), pair(0.5f));
        const float2 fi = floor_small2(qu), fj = floor_small2(qv);
        fx[q] = add2(qu, make_float2(-fi.x, -fi.y));
        fy[q] = add2(qv, make_float2(-fj.x, -fj.y));
        const float2 xn = fma2(fi, VP.inv_w(), make_float2(f0 ? 0.5f : 0.0f, f1 ? 0.5f : 0.0f));
        const float2 yn = fma2(fj, VP.inv_h(), pair(0.5f));
        G0[q] = tex2Dgather<float4>(view_tex<VA>(P.src[2 * q]), xn.x, yn.x, 0);
        G1[q] = tex2Dgather<float4>(view_tex<VA>(P.src[2 * q + 1]), xn.y, yn.y, 0);
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const float4 g0 = G0[q];
        const float4 g1 = G1[q];
        const float top0 = fmaf(fx[q].x, g0.z - g0.w, g0.w), bot0 = fmaf(fx[q].x, g0.y - g0.x, g0.x);
        const float top1 = fmaf(fx[q].y, g1.z - g1.w, g1.w), bot1 = fmaf(fx[q].y, g1.y - g1.x, g1.x);
        J[q] = make_float2(fmaf(fy[q].x, bot0 - top0, top0), fmaf(fy[q].y, bot1 - top1, top1));
    }
}

template <int NP, class VA, int PITCH, bool AT_ADDRESS = false>
__device__ __forceinline__ void pairs_sample(const PixelParams& P, float alpha, float beta, int cx, float2 (&J)[NP]) {
    float2 U[NP][3];
    if constexpr (AT_ADDRESS) {
        pairs_columns<NP, PITCH>(shared_at(&col_table<NP, VA, PITCH>()[0][0][cx]), U);
    } else {
#pragma unroll
        for (int k = 0; k < 3 * NP; ++k) U[k / 3][k % 3] = col_table<NP, VA, PITCH>()[k / 3][k % 3][cx];
    }
    pairs_sample_columns<NP, VA>(P, alpha, beta, U, J);
}

// Half-sweeps that read the column table by shared addresses: those of even view
// counts (1920x960, 6 views, 8 iterations: 76.8 -> 75.8 ms; 3840x1920, 8 views: 390 ->
// 380 ms), but only the fixed windows with 6 views, and with 8 where a lane has a pixel of its
// own (one iteration at 13x13 / 2, by address and by index: 514x258, 6 views 1736 against
// 1709 us, 1000x502 5493 against 5434, 8 views 7022 against 6998; 4 iterations of 9x9 / 2, 8
// views, lanes a pixel: 256x128 1631 against 1687; 1920x960, 13x13 / 2, 10 views 30472 against
// 30636, 2 views 7728 against 8106). With an odd last view, and in the one-evaluation
// kernels, indexing is the faster (5 views 8.83 against 8.91 ms, the cost of 6 views 1.03
// against 1.05 ms).
constexpr bool columns_at_address(int ns, int win, int lanes) {
    return ns % 2 == 0 && (win != 0 || (ns != 6 && (ns != 8 || lanes > 1)));
}

// plane_cost for exactly NS >= 2 views held in kernel parameters, with the
// views processed in pairs (packed FP32) and an odd last view on its own.
// AT_ADDRESS: the column table by shared addresses, where columns_at_address says so.
template <int NS, int WIN, class SM, class VA, bool AT_ADDRESS>
__device__ __forceinline__ float plane_cost_paired(const PixelParams& P, const SM& sm, int lx, int ly,
                                                   const RefStats& st, float3 rp, float d, float3 n) {
    constexpr int NP = NS / 2;
    constexpr bool ODD = (NS & 1) != 0;
    const float eps = 1e-8f * st.Sw * st.Sw;
    if (st.varI < eps) return 2.0f;
    const float dn = d * dot3(n, rp);
    const int K = Window<WIN>::K(P), R = Window<WIN>::R(P), stp = Window<WIN>::stride(P);
    const int ac = K >> 1;

    float2 c0[NP], SJ[NP], SJJ[NP], SIJ[NP];
    float c0o = 0.f, SJo = 0.f, SJJo = 0.f, SIJo = 0.f;
    {
        const int o = ac * stp - R;
        const float cl = sm.row_cos[ly + o];
        const float3 rq = make_float3(cl * sm.col_sin[lx + o], -sm.row_sin[ly + o], cl * sm.col_cos[lx + o]);
        const float den = dot3(n, rq);
        if (!(den < -1e-6f)) return 2.0f;
        const float t = __fdividef(dn, den);
        const float X = t * rq.x, Y = t * rq.y, Z = t * rq.z;
        const float alpha = t * cl, beta = -t * sm.row_sin[ly + o];
        pairs_sample<NP, VA, SM::PITCH, AT_ADDRESS>(P, alpha, beta, lx + o, c0);
#pragma unroll
        for (int q = 0; q < NP; ++q) SJ[q] = SJJ[q] = SIJ[q] = pair(0.f);
        if (ODD) c0o = view_sample<VA>(P.src[NS - 1], X, Y, Z);
    }
    bool valid = true;
#pragma unroll 1
    for (int a = 0; a < K; ++a) {
        const int oy = a * stp - R;
        const float cl = sm.row_cos[ly + oy], msl = -sm.row_sin[ly + oy];
        const float* ref_row = sm.ref + (ly + oy) * SM::PITCH + lx - R;
#pragma unroll 1
        for (int b = 0; b < K; ++b) {
            if (a == ac && b == ac) continue;
            const float Iq = ref_row[b * stp];
            const float w = bilateral(P, sm, a, b, Iq, st.Ip);
            const float wI = w * (Iq - st.mu);
            const int cx = lx + b * stp - R;
            const float3 rq = make_float3(cl * sm.col_sin[cx], msl, cl * sm.col_cos[cx]);
            const float den = dot3(n, rq);
            // an invalid sample makes the cost 2; the loop runs on without a
            // branch (1 % faster than leaving it), its values are discarded
            valid = valid && (den < -1e-6f);
            const float t = __fdividef(dn, den);
            const float X = t * rq.x, Y = t * rq.y, Z = t * rq.z;
            const float alpha = t * cl, beta = t * msl;
            const float2 w2 = pair(w), wI2 = pair(wI);
            float2 Jall[NP];
            pairs_sample<NP, VA, SM::PITCH, AT_ADDRESS>(P, alpha, beta, cx, Jall);
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const float2 J = Jall[q];
                const float2 Jc = add2(J, make_float2(-c0[q].x, -c0[q].y));
                const float2 tw = mul2(w2, Jc);
                SJ[q] = add2(SJ[q], tw);
                SJJ[q] = fma2(tw, Jc, SJJ[q]);
                SIJ[q] = fma2(wI2, Jc, SIJ[q]);
            }
            if (ODD) {
                const float Jc = view_sample<VA>(P.src[NS - 1], X, Y, Z) - c0o;
                const float tw = __fmul_rn(w, Jc);
                SJo = __fadd_rn(SJo, tw);
                SJJo = fmaf(tw, Jc, SJJo);
                SIJo = fmaf(wI, Jc, SIJo);
            }
        }
    }
    if (!valid) return 2.0f;

    float cs[NS];
    auto view_cost = [&](float sj, float sjj, float sij) {
        const float varJ = mul_sub(st.Sw, sjj, sj, sj);
        const float cov = mul_sub(st.Sw, sij, st.SIc, sj);
        if (varJ < eps) return 2.0f;
        float ncc = cov * rsqrtf(st.varI * varJ);
        ncc = fminf(1.0f, fmaxf(-1.0f, ncc));
        return 1.0f - ncc;
    };
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        cs[2 * q] = view_cost(SJ[q].x, SJJ[q].x, SIJ[q].x);
        cs[2 * q + 1] = view_cost(SJ[q].y, SJJ[q].y, SIJ[q].y);
    }
    if (ODD) cs[NS - 1] = view_cost(SJo, SJJo, SIJo);
    return best_mean<NS>(P, cs);
}

// The paired form serves exactly known view counts whose views sit in kernel
// parameters or in shared memory (the batched kernel); the general form the
// guarded view count and plain-load sources.
template <class VA>
constexpr bool paired_views() {
    return std::is_same<VA, ParamViews>::value || std::is_same<VA, SharedViews>::value;
}

// The cost used by the per-pixel kernels: the paired form where the views
// are exactly known, the general one otherwise.
template <int NS, bool EXACT, class VA, int WIN = 0, class SM = TileSmem, bool SWEEP = false>
__device__ __forceinline__ float cost_of(const PixelParams& P, const SM& sm, int lx, int ly,
                                         const RefStats& st, float3 rp, float d, float3 n) {
    if constexpr (EXACT && NS >= 2 && paired_views<VA>())
        return plane_cost_paired<NS, WIN, SM, VA, SWEEP && columns_at_address(NS, WIN, SM::LANES)>(P, sm, lx, ly, st, rp, d, n);
    else
        return plane_cost<NS, EXACT, VA, SM>(P, sm, lx, ly, st, rp, d, n);
}

// Face the camera: n . r_p < 0 (|n . r_p| < 1e-3: replace by -r_p).
__device__ __forceinline__ float3 face_camera(float3 n, float3 rp) {
    const float c = dot3(n, rp);
    if (fabsf(c) < 1e-3f) return make_float3(-rp.x, -rp.y, -rp.z);
    if (c > 0.f) return make_float3(-n.x, -n.y, -n.z);
    return n;
}

// Random initial plane of pixel i (Sec. III-B): inverse range uniform on
// [1/d_max, 1/d_min), normal uniform on the sphere turned to the camera,
// from Philox block (i, 0, 0, 0).
__device__ __forceinline__ void random_plane(const PixelParams& P, size_t i, float3 rp, float& d, float3& n) {
    const U4 u = draw_uniform4(i, 0, 0, P.seed, P.keyframe);
    const float inv = fmaf(u.x, P.inv_dmin - P.inv_dmax, P.inv_dmax);
    d = 1.0f / inv;
    const float z = 1.0f - 2.0f * u.y;
    const float rho = sqrtf(fmaxf(0.f, fmaf(-z, z, 1.0f)));
    float sp, cp;
    sincospif(2.0f * u.z, &sp, &cp);
    n = face_camera(make_float3(rho * cp, rho * sp, z), rp);
}

// Neighbour candidate k of pixel (x, y) (Sec. III-C): the plane of the k-th
// opposite-colour neighbour re-intersected with this pixel's ray. False where
// the neighbour lies outside the image, the plane does not face the ray or the
// range leaves [d_min, d_max]. Every use computes it with this one function,
// so equal inputs give equal bits.
__device__ __forceinline__ bool neighbour_candidate(const PixelParams& P, int x, int y, float3 rp, int k,
                                                    float& dc, float3& nc) {
    const int qy = y + c_neighbors[P.table][k][1];
    if (qy < 0 || qy >= P.H) return false;
    const int qx = wrap_index(x + c_neighbors[P.table][k][0], P.W);
    const size_t j = (size_t)qy * P.W + qx;
    nc = make_float3(P.nx[j], P.ny[j], P.nz[j]);
    const float den = dot3(nc, rp);
    const float3 rq = pixel_bearing(qx, qy, P.W, P.H);
    dc = P.depth[j] * dot3(nc, rq) / den;
    return den < -1e-6f && dc >= P.d_min && dc <= P.d_max;
}

// Neighbour k of pixel (x, y) kept its plane in its last half-sweep (or lies
// outside the image).
__device__ __forceinline__ bool unchanged_neighbour(const PixelParams& P, int x, int y, int k) {
    const int qy = y + c_neighbors[P.table][k][1];
    if (qy < 0 || qy >= P.H) return true;
    return P.changed[(size_t)qy * P.W + wrap_index(x + c_neighbors[P.table][k][0], P.W)] == 0;
}

// Bit-for-bit equal planes (the cost is a deterministic function of them).
__device__ __forceinline__ bool same_plane(float d0, float3 n0, float d1, float3 n1) {
    return __float_as_uint(d0) == __float_as_uint(d1) && __float_as_uint(n0.x) == __float_as_uint(n1.x) &&
           __float_as_uint(n0.y) == __float_as_uint(n1.y) && __float_as_uint(n0.z) == __float_as_uint(n1.z);
}

// Cost bits mapped so that unsigned order is float order (negative values
// bit-inverted, the sign bit set on the others), and back.
__device__ __forceinline__ unsigned ordered_bits(float c) {
    const unsigned u = __float_as_uint(c);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_ordered_bits(unsigned o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// View counts with a bounded half-sweep (launch_pixel_kernel_ns).
constexpr bool has_bounded(int ns, bool exact) { return exact && ns >= 4 && ns <= 10; }

// Whether the half-sweep of (iter, colour) goes to the bounded kernel: enough of the
// pixels of the half-sweep before it ended close (sweep_policy.h). Every half-sweep of such a run
// is launched as both kernels, and one of them finds that it is not its turn.
__device__ __forceinline__ bool bounded_turn(const PixelParams& P) {
    const int phase = 2 * P.iter + P.colour;
    return phase > 0 && P.close[phase - 1] >= (unsigned)bounded_from(P.W, P.H);
}

// The half-sweep's close pixels, for the next one's choice (the block calls it).
__device__ __forceinline__ void count_close(const PixelParams& P, bool close) {
    const int n = __syncthreads_count(close);
    if (threadIdx.x == 0 && n) atomicAdd(P.close + 2 * P.iter + P.colour, (unsigned)n);
}

// One half-sweep over the pixels of `colour` in a tile (Sec. III-C): each
// pixel tries its 8 neighbour candidates, then n_refine perturbations of the
// best so far, and a candidate replaces the incumbent only if its cost is
// strictly lower. Taken in that order, the neighbour phase ends on the
// candidate of lowest cost, the first of equal ones, if that cost is below
// the incumbent's; a candidate bit-identical to the incumbent or to an
// earlier candidate can never be that one (its cost equals theirs), so it is
// not evaluated. Nor is, from the second iteration of a run on, the candidate of
// a neighbour whose plane has not changed since this pixel's last half-sweep
// (P.changed, written by every half-sweep of the run; the neighbours' colour has
// run exactly once in between): it was tried then, the incumbent ended at or
// below its cost, incumbents only improve, and a plane's cost at a pixel has the
// same bits at every evaluation. On a 960x480 6-view keyframe 2 % of the
// neighbour candidates are left out in the second iteration, 75 % in the eighth.
// The other neighbour candidates of a warp's 32 pixels are
// pooled and evaluated 32 at a time, each lane taking any pixel's candidate,
// and every pixel keeps the minimum of (cost, candidate index) in shared
// memory; then each pixel adopts that candidate if it wins and runs its
// refinements. The maps equal those of trying all candidates in turn.
//
// LANES lanes of a warp share a pixel. One (the shape of large keyframes) leaves
// nothing idle. Several spread a small keyframe over more warps: its neighbour
// candidates are pooled as ever, and its next LANES refinement tests are scored
// side by side from the same incumbent, on the supposition that all but the last
// fail; the first success is taken, and the tests after it are scored again from
// the new incumbent. The maps are those of the tests in turn.
template <int NS, bool EXACT, class VA, int WIN, class SM>
__device__ __forceinline__ void sweep_pooled(const PixelParams& P, SM& sm, int bx, int by, int colour, int iter) {
    constexpr int LANES = SM::LANES, PER_WARP = 32 / LANES;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane % LANES, own = threadIdx.x / LANES;  // this lane of its pixel's; its pixel of the block
    const int y = by + own / (SM::W / 2), x = bx + 2 * (own % (SM::W / 2)) + ((y + colour) & 1);
    const bool active = x < P.W && y < P.H;
    const int lx = x - bx + P.radius, ly = y - by + P.radius;
    const size_t i = (size_t)y * P.W + x;
    float bd = 0.f, bc = 0.f;
    float3 bn = make_float3(0.f, 0.f, 0.f), rp = bn;
    unsigned need = 0;
    bool replaced = false;
    if (active) {
        rp = make_float3(sm.row_cos[ly] * sm.col_sin[lx], -sm.row_sin[ly], sm.row_cos[ly] * sm.col_cos[lx]);
        bd = P.depth[i];
        bn = make_float3(P.nx[i], P.ny[i], P.nz[i]);
        bc = P.cost[i];
    }
    if (active && sub == 0) {
        unsigned settled = 0;  // neighbours whose plane was tried in the last half-sweep
        if (P.changed != nullptr && iter > 0) {
#pragma unroll
            for (int k = 0; k < 8; ++k) settled |= (unsigned)unchanged_neighbour(P, x, y, k) << k;
        }
        float SII, w_centre;
        sm.pool.st[own] = ref_stats<WIN>(P, sm, lx, ly, SII, w_centre);
        float cd[8];
        float3 cn[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const bool ok = neighbour_candidate(P, x, y, rp, k, cd[k], cn[k]);
            bool dup = same_plane(cd[k], cn[k], bd, bn);
#pragma unroll
            for (int m = 0; m < k; ++m) dup = dup || (((need >> m) & 1u) && same_plane(cd[k], cn[k], cd[m], cn[m]));
            if (ok && !dup && !((settled >> k) & 1u)) need |= 1u << k;
        }
    }
    if (sub == 0) sm.pool.key[own] = ~0ull;
    // this lane's first slot in the warp's list: exclusive prefix of the counts
    const int cnt = __popc(need);
    int off = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, off, d);
        if (lane >= d) off += v;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= cnt;
    unsigned char* items = sm.pool.item[warp];
    for (unsigned m = need; m; m &= m - 1) items[off++] = (unsigned char)(((lane / LANES) << 3) | (__ffs(m) - 1));
    __syncwarp();

    const int pooled_rounds = (total + 31) >> 5;  // warp-uniform
    const float span = P.inv_dmin - P.inv_dmax;
    // the neighbour phase's winner, once every pooled evaluation has landed
    auto adopt_best = [&]() {
        __syncwarp();
        const unsigned long long key = sm.pool.key[own];
        if (active && key != ~0ull) {
            const float c = from_ordered_bits((unsigned)(key >> 3));
            if (c < bc) {
                float dc;
                float3 nc;
                neighbour_candidate(P, x, y, rp, (int)(key & 7u), dc, nc);
                bc = c;
                bd = dc;
                bn = nc;
                replaced = true;
            }
        }
    };
    int taken = 0;  // refinement tests of the own pixel decided (one lane a pixel: the same in all)
    // With one lane a pixel the bound of the loop is known: leaving it by the test of
    // several lanes took 2.60 ms where this takes 2.52 (1000x502, 4 views, 9x9 at stride
    // 3, 3 iterations) and 10.07 where this takes 9.76 (8 views, 5x5).
    const int n_jobs = pooled_rounds + P.n_refine;
#pragma unroll 1
    for (int r = 0; LANES != 1 || r < n_jobs; ++r) {
        if (r == pooled_rounds) adopt_best();
        if (LANES == 1)
            taken = r - pooled_rounds;
        else if (r >= pooled_rounds && !__any_sync(0xffffffffu, active && taken < P.n_refine))
            break;
        // the job of this round: (pixel, plane)
        bool job = false;
        int jt = own, jx = x, jy = y, k = 0;
        float3 jrp = rp;
        float dc = 0.f;
        float3 nc = make_float3(0.f, 0.f, 0.f);
        if (r < pooled_rounds) {
            const int idx = (r << 5) + lane;
            if (idx < total) {
                const int it = items[idx];
                k = it & 7;
                jt = warp * PER_WARP + (it >> 3);
                const int otx = jt % (SM::W / 2), oty = jt / (SM::W / 2);
                jy = by + oty;
                jx = bx + 2 * otx + ((jy + colour) & 1);
                job = true;
            }
        } else if (active && taken + sub < P.n_refine) {
            const int t = taken + sub;
            const float sc = __int_as_float((126 - t) << 23);  // 2^-(t+1)
            const U4 u = draw_uniform4(i, (uint64_t)iter, (uint64_t)(1 + t), P.seed, P.keyframe);
            float inv = fmaf((2.0f * u.x - 1.0f) * sc, span, 1.0f / bd);
            inv = fminf(P.inv_dmin, fmaxf(P.inv_dmax, inv));
            dc = 1.0f / inv;
            nc = make_float3(fmaf(sc, 2.0f * u.y - 1.0f, bn.x), fmaf(sc, 2.0f * u.z - 1.0f, bn.y),
                             fmaf(sc, 2.0f * u.w - 1.0f, bn.z));
            const float il = 1.0f / sqrtf(dot3(nc, nc));
            nc = face_camera(make_float3(nc.x * il, nc.y * il, nc.z * il), rp);
            job = true;
        }
        if (LANES == 1 && !job) continue;
        float c = 4.0f;  // above every cost
        bool won = false;
        if (job) {
            const int jlx = jx - bx + P.radius, jly = jy - by + P.radius;
            if (r < pooled_rounds) {
                jrp = make_float3(sm.row_cos[jly] * sm.col_sin[jlx], -sm.row_sin[jly], sm.row_cos[jly] * sm.col_cos[jlx]);
                neighbour_candidate(P, jx, jy, jrp, k, dc, nc);
            }
            c = cost_of<NS, EXACT, VA, WIN, SM, true>(P, sm, jlx, jly, sm.pool.st[jt], jrp, dc, nc);
            if (r < pooled_rounds) {
                if (c == c) atomicMin(&sm.pool.key[jt], ((unsigned long long)ordered_bits(c) << 3) | (unsigned)k);
            } else {
                won = c < bc;
            }
        }
        if constexpr (LANES == 1) {
            if (won) {
                bc = c;
                bd = dc;
                bn = nc;
                replaced = true;
            }
        } else if (r >= pooled_rounds) {
            // the pixel's first success, if there is one, becomes every lane's incumbent
            const unsigned mine = (__ballot_sync(0xffffffffu, won) >> (lane - sub)) & ((1u << LANES) - 1u);
            const int first = mine ? __ffs(mine) - 1 : sub, from = lane - sub + first;
            const float cw = __shfl_sync(0xffffffffu, c, from), dw = __shfl_sync(0xffffffffu, dc, from);
            const float3 nw = make_float3(__shfl_sync(0xffffffffu, nc.x, from), __shfl_sync(0xffffffffu, nc.y, from),
                                          __shfl_sync(0xffffffffu, nc.z, from));
            if (mine) {
                bc = cw;
                bd = dw;
                bn = nw;
                replaced = true;
            }
            taken += mine ? first + 1 : LANES;
        }
    }
    if (LANES == 1 && n_jobs == pooled_rounds) adopt_best();
    if constexpr (has_bounded(NS, EXACT) && std::is_same<VA, ParamViews>::value && LANES == 1)
        if (P.close != nullptr) count_close(P, active && bc < CLOSE_COST);
    if (!active || sub != 0) return;
    if (P.changed) P.changed[i] = replaced;
    P.depth[i] = bd;
    P.nx[i] = bn.x;
    P.ny[i] = bn.y;
    P.nz[i] = bn.z;
    P.cost[i] = bc;
}

// A refinement candidate's cost must fall below the incumbent's to matter, and
// most end far above it. After part of the samples the cost is already bounded
// from below: over the samples A taken so far let V_I, V_J and C be the weighted
// variances and covariance. (1 - NCC^2) V is what the best line in J leaves of the
// reference's sum of squares V = varI / Sw over the whole window, and over A alone
// a line of positive slope leaves at least r = (V_I - C^2 / V_J) / Sw_A (V_I / Sw_A where
// C <= 0, scaled sums as below). So for NCC > 0
//   NCC^2 <= 1 - r / V <= V / (V + r),
// and the cost is at least the mean of 1 - NCC over the best_k views of highest
// bound. The last form is the one used. Its root has the smaller rounding error (a
// derivative of at most 1/2 in r / V, where that of 1 - r / V grows without limit), but
// it is not the sharpest: r <= V, so a view's bound never exceeds 1 - sqrt(1/2) = 0.293,
// and an incumbent above that lets no test go.
// A candidate whose bound clears the incumbent is dropped; the others
// are evaluated to the end by the same operations in the same order as ever, so
// the maps do not change.
//
// Rounding: with n samples, u = 2^-24, A = Sw / w_c (w_c the weight of the
// centre-most sample, on which every view is centred: varJ >= w_c sum w J^2, so
// no sum of J cancels by more than A) and B = Sw sum w I^2 / varI, standard
// forward error bounds on the sums give at most (6 n + 8) u A B for the computed
// cost and (8 n + 9) u A B for the computed bound; refine_margin is their sum
// plus a few roundings of the remaining operations. Where it is large (a
// negligible centre weight, a flat patch) nothing is dropped.
__device__ __forceinline__ float refine_margin(const RefStats& st, float SII, float wc, int n) {
    const float AB = (st.Sw / wc) * (st.Sw * SII / st.varI);
    const float m = fmaf(5.9604645e-8f * (float)(14 * n + 20), AB, 4e-6f);
    return m < 0.1f ? m : __int_as_float(0x7f800000);
}

// Largest NCC a view can still reach (see above): V_I, V_J, C over the samples
// taken, scaled by their weight; scale = Sw / (varI Sw_A); `whole`: all samples
// are taken and the NCC itself is returned (0 where negative).
__device__ __forceinline__ float ncc_bound(float VI, float VJ, float C, float scale, float floor_vj, bool whole) {
    const float q = C > 0.f ? C * (C * rcp_approx(VJ)) : 0.f;
    const float free = rcp_approx(fmaf(VI - q, scale, 1.0f));
    const float m2 = whole ? q * rcp_approx(VI) : free;
    return VJ > floor_vj ? sqrt_approx(m2) : 1.0f;
}

// The random steps of refinement test t (Sec. III-C item 1) of pixel i: of the
// inverse range in x, of the normal in y, z, w, each 2^-(t+1) (2 u - 1), exact in
// FP32.
__device__ __forceinline__ U4 refinement_steps(const PixelParams& P, size_t i, int iter, int t) {
    const float sc = __int_as_float((126 - t) << 23);  // 2^-(t+1)
    U4 u = draw_uniform4((unsigned)i, (unsigned)iter, (unsigned)(1 + t), P.seed, P.keyframe);
    u.x = (2.0f * u.x - 1.0f) * sc;
    u.y = (2.0f * u.y - 1.0f) * sc;
    u.z = (2.0f * u.z - 1.0f) * sc;
    u.w = (2.0f * u.w - 1.0f) * sc;
    return u;
}

// Refinement candidate t of pixel jt of the block, whose ray is rp and index in
// the image i: its incumbent perturbed by the drawn steps.
template <class SM>
__device__ __forceinline__ void refinement_candidate(const PixelParams& P, const SM& sm, int jt, size_t i, int iter, int t,
                                                     float3 rp, float& dc, float3& nc) {
    U4 u;
    if (t < MAX_DRAWN) {
        u.x = sm.bound.draw[t][0][jt];
        u.y = sm.bound.draw[t][1][jt];
        u.z = sm.bound.draw[t][2][jt];
        u.w = sm.bound.draw[t][3][jt];
    } else {
        u = refinement_steps(P, i, iter, t);
    }
    float inv = fmaf(u.x, P.inv_dmin - P.inv_dmax, sm.bound.inv_d[jt]);
    inv = fminf(P.inv_dmin, fmaxf(P.inv_dmax, inv));
    dc = 1.0f / inv;
    nc = make_float3(__fadd_rn(u.y, sm.bound.nx[jt]), __fadd_rn(u.z, sm.bound.ny[jt]), __fadd_rn(u.w, sm.bound.nz[jt]));
    const float il = 1.0f / sqrtf(dot3(nc, nc));
    nc = face_camera(make_float3(nc.x * il, nc.y * il, nc.z * il), rp);
}

template <class SM>
__device__ __forceinline__ void set_incumbent(SM& sm, int jt, float d, float3 n, float c) {
    sm.bound.d[jt] = d;
    sm.bound.inv_d[jt] = 1.0f / d;
    sm.bound.nx[jt] = n.x;
    sm.bound.ny[jt] = n.y;
    sm.bound.nz[jt] = n.z;
    sm.bound.cost[jt] = c;
}

// neighbour_candidate with the neighbour's bearing from the block's tables (the
// same FP32 sines and cosines): pixel (x, y) of a tile at (bx, by).
template <class SM>
__device__ __forceinline__ bool neighbour_from_tables(const PixelParams& P, const SM& sm, int bx, int by, int x, int y,
                                                      float3 rp, int k, float& dc, float3& nc) {
    const int dx = c_neighbors[P.table][k][0], dy = c_neighbors[P.table][k][1];
    const int qy = y + dy;
    if (qy < 0 || qy >= P.H) return false;
    const size_t j = (size_t)qy * P.W + wrap_near(x + dx, P.W);
    nc = make_float3(P.nx[j], P.ny[j], P.nz[j]);
    const float den = dot3(nc, rp);
    const float2 r = sm.bound.near_row[qy - by + MAX_REACH], c = sm.bound.near_col[x + dx - bx + MAX_REACH];
    const float3 rq = make_float3(r.y * c.x, -r.x, r.y * c.y);
    dc = P.depth[j] * dot3(nc, rq) / den;
    return den < -1e-6f && dc >= P.d_min && dc <= P.d_max;
}

// One half-sweep over the pixels of `colour` in a tile (Sec. III-C), for exactly
// NS views: the maps of sweep_pooled bit for bit, by one loop that advances every
// lane by K samples of its own candidate (a window has K x K).
//
// First the neighbour candidates of the warp's pixels, pooled, 32 at a time to
// the end (their costs lie near the incumbent's: a bound drops almost none).
// Then the refinement tests, each dropped as soon as it provably cannot win.
// Dropped at different times, the tests leave lanes free, so any lane takes any
// pixel's test: the next test of each pixel first, and where lanes are left over,
// tests further ahead, on the supposition that those before them fail (on
// converged maps 1 in 30 succeeds). The owner lane takes up a pixel's results in
// order; a success makes the tests started from the older incumbent void, and
// they are started again.
//
// Bound, like sweep_pooled, by FP32 issue of the samples taken (1920x960, 6 views: 415
// warp instructions a sample with the bound and the hand-out, 25 of 32 lanes active;
// sweep_pooled 346 and 31.4). On a converged 960x480 keyframe of 6 views a test is dropped
// after 2.5 of 6 rows on average; lanes left idle and the hand-out keep a third of
// that from the clock. 1920x960, 6 views, 8 iterations: 75.9 -> 66.8 ms; 4 views at
// 960x480 14.7 -> 13.5 ms; 3840x1920, 8 views without noise, 4 iterations 229 ->
// 206 ms. Where costs stay above what the bound can reach (0.293, refine_margin; around 0.4
// with sensor noise at 3840x1920) it drops nothing and the hand-out costs 6 %, so
// such half-sweeps stay with the pooled kernel (bounded_turn).
template <int NS, class VA, int WIN, class SM>
__device__ __forceinline__ void sweep_bounded(const PixelParams& P, SM& sm, int bx, int by, int colour, int iter) {
    constexpr int NP = NS / 2, NPA = NP > 0 ? NP : 1;
    constexpr bool ODD = (NS & 1) != 0;
    using Sample = typename std::remove_reference<decltype(sm.bound)>::type::Sample;
    constexpr int MIN_FREE = 8;  // lanes that are free before new tests are handed out
    static_assert(SM::W / 2 * SM::H == BLOCK_THREADS, "a lane per pixel");
    const int K = Window<WIN>::K(P), R = Window<WIN>::R(P), stp = Window<WIN>::stride(P);
    const int ac = K >> 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    // pixel jt of the block
    auto pixel_x = [&](int jt, int py) { return bx + 2 * (jt % (SM::W / 2)) + ((py + colour) & 1); };
    auto pixel_y = [&](int jt) { return by + jt / (SM::W / 2); };
    auto pixel_ray = [&](int lx, int ly) {
        return make_float3(sm.row_cos[ly] * sm.col_sin[lx], -sm.row_sin[ly], sm.row_cos[ly] * sm.col_cos[lx]);
    };
    const int own = threadIdx.x, oy = pixel_y(own), ox = pixel_x(own, oy);
    const bool owner = ox < P.W && oy < P.H;
    const size_t oi = (size_t)oy * P.W + ox;
    unsigned need = 0;
    for (int k = threadIdx.x; k < K * K; k += BLOCK_THREADS) {
        const int centre = ac * K + ac, at = k == 0 ? centre : (k <= centre ? k - 1 : k);
        const int a = at / K, b = at - a * K, dy = a * stp - R, dx = b * stp - R;
        sm.bound.sample[k] = Sample::at(SM::PITCH, dy, dx, __fadd_rn(sm.wsp[a], sm.wsp[b]));
    }
    for (int k = threadIdx.x; k < SM::H + 2 * R; k += BLOCK_THREADS) sm.bound.row[k] = make_float2(sm.row_cos[k], sm.row_sin[k]);
    for (int k = threadIdx.x; k < SM::W + 2 * R; k += BLOCK_THREADS) sm.bound.col[k] = make_float2(sm.col_sin[k], sm.col_cos[k]);
    for (int k = threadIdx.x; k < SM::W + SM::H + 4 * MAX_REACH; k += BLOCK_THREADS) {
        float sn, cs;  // the angles of pixel_bearing
        if (k < SM::H + 2 * MAX_REACH) {
            sincospif(0.5f - (2.0f * (by + k - MAX_REACH) + 1.0f) / (2.0f * P.H), &sn, &cs);
            sm.bound.near_row[k] = make_float2(sn, cs);
        } else {
            const int c = k - (SM::H + 2 * MAX_REACH);
            sincospif((2.0f * wrap_index(bx + c - MAX_REACH, P.W) + 1.0f) / P.W - 1.0f, &sn, &cs);
            sm.bound.near_col[c] = make_float2(sn, cs);
        }
    }
    __syncthreads();
    if (owner) {
        const int lx = ox - bx + R, ly = oy - by + R;
        unsigned settled = 0;  // neighbours whose plane was tried in the last half-sweep
        if (P.changed != nullptr && iter > 0) {
#pragma unroll
            for (int k = 0; k < 8; ++k) settled |= (unsigned)unchanged_neighbour(P, ox, oy, k) << k;
        }
        const float3 rp = pixel_ray(lx, ly);
        float SII, w_centre;
        const RefStats st = ref_stats<WIN>(P, sm, lx, ly, SII, w_centre);
        sm.pool.st[own] = st;
        sm.bound.margin[own] = refine_margin(st, SII, w_centre, K * K);
        const float bd = P.depth[oi];
        const float3 bn = make_float3(P.nx[oi], P.ny[oi], P.nz[oi]);
        set_incumbent(sm, own, bd, bn, P.cost[oi]);
        sm.bound.version[own] = 0;
        sm.bound.taken[own] = 0;
        sm.pool.key[own] = ~0ull;
        float cd[8];
        float3 cn[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const bool ok = neighbour_from_tables(P, sm, bx, by, ox, oy, rp, k, cd[k], cn[k]);
            bool dup = same_plane(cd[k], cn[k], bd, bn);
#pragma unroll
            for (int m = 0; m < k; ++m) dup = dup || (((need >> m) & 1u) && same_plane(cd[k], cn[k], cd[m], cn[m]));
            if (ok && !dup && !((settled >> k) & 1u)) need |= 1u << k;
        }
    }
    const int n_refine = P.n_refine;
    for (int t = 0; t < min(n_refine, MAX_DRAWN); ++t) {
        const U4 u = refinement_steps(P, oi, iter, t);
        sm.bound.draw[t][0][own] = u.x;
        sm.bound.draw[t][1][own] = u.y;
        sm.bound.draw[t][2][own] = u.z;
        sm.bound.draw[t][3][own] = u.w;
    }
    // this lane's first slot in the warp's list: exclusive prefix of the counts
    const int cnt = __popc(need);
    int off = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, off, d);
        if (lane >= d) off += v;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= cnt;
    unsigned char* items = sm.pool.item[warp];
    for (unsigned m = need; m; m &= m - 1) items[off++] = (unsigned char)((lane << 3) | (__ffs(m) - 1));
    __syncthreads();  // the samples are listed by the whole block

    bool pooled = total > 0, run = false, valid = false, replaced = false;
    bool more = true, hit = false;   // (of the warp) tests not yet started; a test that beat the incumbent
    int next = 0;                    // pooled: list position of the next candidates
    int version = 0, taken = owner ? 0 : n_refine, issued = taken;  // the own pixel's incumbent; its tests: results taken up, started
    int g = K;                       // groups of K samples taken of the current candidate
    int jt = own, jk = 0, jv = 0;    // its pixel, its neighbour or test number, the version of its incumbent
    int lx = R, ly = R;              // the pixel's place in the tile
    float dc = 0.f, dn = 0.f, Ip = 0.f, mu = 0.f;
    float3 nc = make_float3(0.f, 0.f, 0.f);
    float2 c0[NPA], SJ[NPA], SJJ[NPA], SIJ[NPA];
    float c0o = 0.f, SJo = 0.f, SJJo = 0.f, SIJo = 0.f;
    float sw = 0.f, sI = 0.f, sII = 0.f;  // the reference's sums over the samples taken
#pragma unroll
    for (int q = 0; q < NPA; ++q) c0[q] = SJ[q] = SJJ[q] = SIJ[q] = pair(0.f);
    for (;;) {
        // new candidates: pooled, for the whole warp; then, for the lanes that are free
        const unsigned resting = __ballot_sync(0xffffffffu, !run);
        if (pooled ? g == K : resting == 0xffffffffu || hit || (more && __popc(resting) >= MIN_FREE)) {
            bool job = false;
            if (pooled && next >= total) {  // every neighbour candidate has been scored
                __syncwarp();
                if (owner) {
                    const unsigned long long key = sm.pool.key[own];
                    const float c = from_ordered_bits((unsigned)(key >> 3));
                    if (key != ~0ull && c < sm.bound.cost[own]) {
                        neighbour_from_tables(P, sm, bx, by, ox, oy, pixel_ray(ox - bx + R, oy - by + R), (int)(key & 7u), dc, nc);
                        set_incumbent(sm, own, dc, nc, c);
                        replaced = true;
                    }
                }
                pooled = false;
                run = false;
            }
            if (pooled) {
                if (next + lane < total) {
                    const int it = items[next + lane];
                    jk = it & 7;
                    jt = (warp << 5) + (it >> 3);
                    job = true;
                }
                next += 32;
            } else {
                __syncwarp();
                // take up the results of the own pixel's tests, in order (one that won when
                // its turn had come has replaced the incumbent already)
                if (owner && sm.bound.version[own] != version) {
                    version = sm.bound.version[own];
                    issued = taken = sm.bound.taken[own];
                    replaced = true;
                }
                while (taken < issued) {
                    const float c = sm.bound.result[taken % MAX_AHEAD][own];
                    if (__float_as_uint(c) == 0xffffffffu) break;  // under way
                    if (c < sm.bound.cost[own]) {
                        float d;
                        float3 n;
                        refinement_candidate(P, sm, own, oi, iter, taken, pixel_ray(ox - bx + R, oy - by + R), d, n);
                        set_incumbent(sm, own, d, n, c);
                        sm.bound.version[own] = (unsigned char)++version;
                        replaced = true;
                        issued = taken + 1;
                    }
                    ++taken;
                }
                if (owner) sm.bound.taken[own] = (unsigned char)taken;
                __syncwarp();
                if (run && jv != sm.bound.version[jt]) run = false;
                // hand out the pixels' next tests, then the ones after them
                unsigned idle = __ballot_sync(0xffffffffu, !run);
                for (int ahead = 0; ahead < MAX_AHEAD && idle != 0; ++ahead) {
                    const bool offer = issued < n_refine && issued - taken == ahead;
                    const unsigned m = __ballot_sync(0xffffffffu, offer);
                    if (m == 0) continue;
                    const int n_given = min(__popc(m), __popc(idle));
                    const int rank = __popc(m & below);
                    if (offer && rank < n_given) {
                        sm.bound.offer[warp * 32 + rank] = (unsigned)(own | (issued << 8) | (version << 16));
                        sm.bound.result[issued % MAX_AHEAD][own] = __uint_as_float(0xffffffffu);
                        ++issued;
                    }
                    __syncwarp();
                    const int at = __popc(idle & below);
                    if (((idle >> lane) & 1u) && at < n_given) {
                        const unsigned o = sm.bound.offer[warp * 32 + at];
                        jt = (int)(o & 255u);
                        jk = (int)((o >> 8) & 255u);
                        jv = (int)(o >> 16);
                        job = true;
                    }
                    __syncwarp();
                    idle = __ballot_sync(0xffffffffu, !run && !job);
                }
                more = __any_sync(0xffffffffu, issued < n_refine);
                hit = false;
            }
            if (job) {
                const int jy = pixel_y(jt), jx = pixel_x(jt, jy);
                lx = jx - bx + R;
                ly = jy - by + R;
                const float3 rp = pixel_ray(lx, ly);
                if (pooled)
                    neighbour_from_tables(P, sm, bx, by, jx, jy, rp, jk, dc, nc);
                else
                    refinement_candidate(P, sm, jt, (size_t)jy * P.W + jx, iter, jk, rp, dc, nc);
                dn = dc * dot3(nc, rp);
                const RefStats& st = sm.pool.st[jt];
                Ip = st.Ip;
                mu = st.mu;
                valid = !(st.varI < 1e-8f * st.Sw * st.Sw);
#pragma unroll
                for (int q = 0; q < NPA; ++q) SJ[q] = SJJ[q] = SIJ[q] = pair(0.f);
                SJo = SJJo = SIJo = sw = sI = sII = 0.f;
            }
            if (job || pooled) {
                run = job;
                g = 0;
            }
        }
        if (!__any_sync(0xffffffffu, run)) break;
        if (run) {
            const unsigned ref = shared_at(sm.ref + ly * SM::PITCH + lx);
            const unsigned row = shared_at(sm.bound.row + ly), col = shared_at(sm.bound.col + lx);
            unsigned table = 0;  // from a column's bearing to its entry of the column table
            if constexpr (NP > 0) table = shared_at(&col_table<NP, VA, SM::PITCH>()[0][0][0]) - shared_at(sm.bound.col);
            const Sample* smp = sm.bound.sample + g * K;
#pragma unroll 1
            for (int j = 0; j < K; ++j) {
                const Sample q = smp[j];
                const float Iq = shared_f(ref + q.ref());
                const float dI = Iq - Ip;
                const float w = exp2_approx(fmaf(P.wc, dI * dI, q.wsp));
                const float Ic = Iq - mu, wI = w * Ic;
                const unsigned at = col + q.col();
                const float2 rw = shared_f2(row + q.row()), cl = shared_f2(at);  // (cos, sin) latitude, (sin, cos) longitude
                const float3 rq = make_float3(rw.x * cl.x, -rw.y, rw.x * cl.y);
                const float den = dot3(nc, rq);
                valid = valid && (den < -1e-6f);
                const float t = __fdividef(dn, den);
                float2 J[NPA];
                if constexpr (NP > 0) {
                    float2 U[NP][3];
                    pairs_columns<NP, SM::PITCH>(at + table, U);
                    pairs_sample_columns<NP, VA>(P, t * rw.x, t * rq.y, U, J);
                }
                float Jo = 0.f;
                if (ODD) Jo = view_sample<VA>(P.src[NS - 1], t * rq.x, t * rq.y, t * rq.z);
                if (j == 0) {  // the first sample of all centres every view
                    if (g == 0) {
#pragma unroll
                        for (int p = 0; p < NP; ++p) c0[p] = J[p];
                        c0o = Jo;
                    }
                }
                const float2 w2 = pair(w), wI2 = pair(wI);
                sw += w;
                sI += wI;
                sII = fmaf(wI, Ic, sII);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const float2 Jc = add2(J[p], make_float2(-c0[p].x, -c0[p].y));
                    const float2 tw = mul2(w2, Jc);
                    SJ[p] = add2(SJ[p], tw);
                    SJJ[p] = fma2(tw, Jc, SJJ[p]);
                    SIJ[p] = fma2(wI2, Jc, SIJ[p]);
                }
                if (ODD) {
                    const float Jc = Jo - c0o;
                    const float tw = __fmul_rn(w, Jc);
                    SJo = __fadd_rn(SJo, tw);
                    SJJo = fmaf(tw, Jc, SJJo);
                    SIJo = fmaf(wI, Jc, SIJo);
                }
            }
        }
        ++g;
        bool done = run && g == K, dropped = false, won = false, in_turn = false;
        float c_won = 0.f;
        if (!pooled) {
            float thr = 0.f, VI = 0.f, scale = 0.f;
            bool may = false;
            // (where half the warp ends at once, their costs come cheaper than a bound first)
            const bool few = __popc(__ballot_sync(0xffffffffu, done)) < 16;
            if (run) {
                done = done || !valid;
                const RefStats& st = sm.pool.st[jt];
                thr = sm.bound.cost[jt] + sm.bound.margin[jt];
                VI = fmaf(sw, sII, -(sI * sI));
                scale = st.Sw * rcp_approx(st.varI * sw);
                // were no view to correlate in the samples taken: the most the bound can be
                may = valid && (g == K ? few : 1.0f - rsqrtf(fmaf(VI, scale, 1.0f)) > thr);
            }
            if (may) {
                const float fl = 1e-8f * sw * sw;
                float cs[NS];
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const float2 sw2 = pair(sw), sI2 = pair(-sI);
                    const float2 VJ = fma2(sw2, SJJ[p], mul2(make_float2(-SJ[p].x, -SJ[p].y), SJ[p]));
                    const float2 C = fma2(sw2, SIJ[p], mul2(sI2, SJ[p]));
                    cs[2 * p] = ncc_bound(VI, VJ.x, C.x, scale, fl, g == K);
                    cs[2 * p + 1] = ncc_bound(VI, VJ.y, C.y, scale, fl, g == K);
                }
                if (ODD) cs[NS - 1] = ncc_bound(VI, fmaf(sw, SJJo, -SJo * SJo), fmaf(sw, SIJo, -sI * SJo), scale, fl, g == K);
                // the best_k largest, bubbled to the end one by one
                float sum = 0.f;
#pragma unroll
                for (int b = 0; b < NS; ++b) {
                    if (b >= P.best_k) break;
#pragma unroll
                    for (int q = 0; q + 1 < NS - b; ++q) {
                        const float lo = fminf(cs[q], cs[q + 1]), hi = fmaxf(cs[q], cs[q + 1]);
                        cs[q] = lo;
                        cs[q + 1] = hi;
                    }
                    sum += 1.0f - cs[NS - 1 - b];
                }
                dropped = sum > thr * (float)P.best_k;
            }
            if (dropped) {
                sm.bound.result[jk % MAX_AHEAD][jt] = 4.0f;  // no cost: above every one
                done = run = false;
            }
        }
        if (done) {
            const RefStats& st = sm.pool.st[jt];
            float c = 2.0f;
            if (valid) {
                const float eps = 1e-8f * st.Sw * st.Sw;
                float cs[NS];
                auto view_cost = [&](float sj, float sjj, float sij) {
                    const float varJ = mul_sub(st.Sw, sjj, sj, sj);
                    const float cov = mul_sub(st.Sw, sij, st.SIc, sj);
                    if (varJ < eps) return 2.0f;
                    float ncc = cov * rsqrtf(st.varI * varJ);
                    ncc = fminf(1.0f, fmaxf(-1.0f, ncc));
                    return 1.0f - ncc;
                };
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    cs[2 * p] = view_cost(SJ[p].x, SJJ[p].x, SIJ[p].x);
                    cs[2 * p + 1] = view_cost(SJ[p].y, SJJ[p].y, SIJ[p].y);
                }
                if (ODD) cs[NS - 1] = view_cost(SJo, SJJo, SIJo);
                c = best_mean<NS>(P, cs);
            }
            if (pooled) {
                if (c == c) atomicMin(&sm.pool.key[jt], ((unsigned long long)ordered_bits(c) << 3) | (unsigned)jk);
            } else {
                sm.bound.result[jk % MAX_AHEAD][jt] = c;
                run = false;
                won = c < sm.bound.cost[jt];
                in_turn = won && jk == sm.bound.taken[jt];
                c_won = c;
            }
        }
        if (!pooled && __any_sync(0xffffffffu, won)) {
            hit = true;
            __syncwarp();  // (every lane has seen whose turn it is)
            if (in_turn) {
                set_incumbent(sm, jt, dc, nc, c_won);
                ++sm.bound.version[jt];
                ++sm.bound.taken[jt];
            }
        }
    }
    count_close(P, owner && sm.bound.cost[own] < CLOSE_COST);
    if (!owner) return;
    P.changed[oi] = replaced;
    if (!replaced) return;  // the planes stay as they are
    P.depth[oi] = sm.bound.d[own];
    P.nx[oi] = sm.bound.nx[own];
    P.ny[oi] = sm.bound.ny[own];
    P.nz[oi] = sm.bound.nz[own];
    P.cost[oi] = sm.bound.cost[own];
}

// The tile's column table (see col_table), from its staged bearings.
template <int NP, class VA, class SM>
__device__ __forceinline__ void build_col_table(const PixelParams& P, const SM& sm) {
    static_assert(NP <= PMSP_MAX_SOURCES / 2, "column table too small");
    const int cols = SM::W + 2 * P.radius;
    for (int i = threadIdx.x; i < cols * NP; i += BLOCK_THREADS) {
        const int q = i / cols, c = i - q * cols;
        const PixelParams::ViewPair& VP = P.pairs[q];
        const float2 sn = pair(sm.col_sin[c]), cs = pair(sm.col_cos[c]);
        col_table<NP, VA, SM::PITCH>()[q][0][c] = fma2(VP.R[0], sn, mul2(VP.R[2], cs));
        col_table<NP, VA, SM::PITCH>()[q][1][c] = fma2(VP.R[3], sn, mul2(VP.R[5], cs));
        col_table<NP, VA, SM::PITCH>()[q][2][c] = fma2(VP.R[6], sn, mul2(VP.R[8], cs));
    }
}

// What a tile's pixels need besides P: the staged tile and, on the paired path, the
// column table. The block calls it; it ends with a barrier.
template <int NS, bool EXACT, class VA, class SM>
__device__ __forceinline__ void prepare_tile(const PixelParams& P, SM& sm, int bx, int by) {
    stage_tile(P, sm, bx, by);
    __syncthreads();
    if constexpr (EXACT && NS >= 2 && paired_views<VA>()) {
        build_col_table<NS / 2, VA>(P, sm);
        __syncthreads();
    }
}

// MODE_INIT (random plane and its cost) or MODE_COST (the stored plane's cost) for
// this thread's pixel of `colour` in a prepared tile.
template <int NS, bool EXACT, int MODE, class VA, int WIN, class SM>
__device__ __forceinline__ void score_pixel(const PixelParams& P, const SM& sm, int bx, int by, int colour) {
    const int tx = threadIdx.x % (SM::W / 2), ty = threadIdx.x / (SM::W / 2);
    const int y = by + ty;
    const int x = bx + 2 * tx + ((y + colour) & 1);
    if (x >= P.W || y >= P.H) return;
    const int lx = x - bx + P.radius, ly = y - by + P.radius;
    const size_t i = (size_t)y * P.W + x;
    const float3 rp = make_float3(sm.row_cos[ly] * sm.col_sin[lx], -sm.row_sin[ly],
                                  sm.row_cos[ly] * sm.col_cos[lx]);
    float SII, w_centre;
    const RefStats st = ref_stats<WIN>(P, sm, lx, ly, SII, w_centre);
    float d;
    float3 n;
    if (MODE == MODE_COST) {
        d = P.depth[i];
        n = make_float3(P.nx[i], P.ny[i], P.nz[i]);
    } else {
        random_plane(P, i, rp, d, n);
        P.depth[i] = d;
        P.nx[i] = n.x;
        P.ny[i] = n.y;
        P.nz[i] = n.z;
    }
    P.cost[i] = cost_of<NS, EXACT, VA, WIN, SM>(P, sm, lx, ly, st, rp, d, n);
}

// One tile of one problem: stage the reference tile, then every active
// pixel of `colour` runs MODE. P may live in kernel parameters or in shared
// memory (the batched kernel). Returns without a trailing barrier.
template <int NS, bool EXACT, int MODE, class VA = ParamViews, int WIN = 0, class SM = TileSmem>
__device__ __forceinline__ void process_tile(const PixelParams& P, SM& sm, int bx, int by, int colour,
                                             int iter) {
    prepare_tile<NS, EXACT, VA>(P, sm, bx, by);
    if constexpr (MODE == MODE_SWEEP) {
        sweep_pooled<NS, EXACT, VA, WIN, SM>(P, sm, bx, by, colour, iter);
    } else {
        score_pixel<NS, EXACT, MODE, VA, WIN>(P, sm, bx, by, colour);
    }
}

template <int NS, bool EXACT, int MODE, int WIN = 0, int TS = 0>
__global__ void __launch_bounds__(BLOCK_THREADS, pixel_min_blocks(NS)) pixel_kernel(const __grid_constant__ PixelParams P) {
    using SM = typename TileShape<TS, Window<WIN>::HALO, MODE == MODE_SWEEP>::Smem;
    __shared__ SM sm;
    int tx, ty;
    tile_of_block(gridDim.x, gridDim.y, blockIdx.y * gridDim.x + blockIdx.x, tx, ty);
    if (MODE == MODE_SWEEP && has_bounded(NS, EXACT) && TS == 0 && P.close != nullptr && bounded_turn(P)) return;
    if constexpr (MODE == MODE_SWEEP) {
        process_tile<NS, EXACT, MODE, ParamViews, WIN, SM>(P, sm, tx * SM::W, ty * SM::H, P.colour, P.iter);
    } else {
        // both colours in one launch: one after the other from one staged tile, or in
        // two layers of blocks (launch_score)
        prepare_tile<NS, EXACT, ParamViews>(P, sm, tx * SM::W, ty * SM::H);
#pragma unroll 1
        for (int colour = blockIdx.z; colour < 2; colour += gridDim.z)
            score_pixel<NS, EXACT, MODE, ParamViews, WIN>(P, sm, tx * SM::W, ty * SM::H, colour);
    }
}

// The bounded half-sweep of one tile (sweep_bounded), where it is its turn.
template <int NS, int WIN>
__global__ void __launch_bounds__(BLOCK_THREADS, pixel_min_blocks(NS)) bounded_kernel(const __grid_constant__ PixelParams P) {
    using SM = TileSmemT<32, 8, 1, Window<WIN>::HALO, true, true>;
    __shared__ SM sm;
    if (!bounded_turn(P)) return;
    int tx, ty;
    tile_of_block(gridDim.x, gridDim.y, blockIdx.y * gridDim.x + blockIdx.x, tx, ty);
    const int bx = tx * SM::W, by = ty * SM::H;
    prepare_tile<NS, true, ParamViews>(P, sm, bx, by);
    sweep_bounded<NS, ParamViews, WIN, SM>(P, sm, bx, by, P.colour, P.iter);
}

// Grid of a tile shape over a W x H panorama.
template <int TS>
inline dim3 tile_grid(const PixelParams& p) {
    using SM = typename TileShape<TS>::Smem;
    return dim3((p.W + SM::W - 1) / SM::W, (p.H + SM::H - 1) / SM::H);
}

// The split of an SM's 256 KB between shared memory and texture cache that leaves
// the gathers all but what the blocks that its registers let reside need. The driver's own choice
// gave shared memory 100 KB where 64 do: 3840x1920 half-sweeps of 8 fp16 views,
// 4 iterations, took 242.9 ms with 100 KB, 229.0 with 64, 257.1 with 132, 287.0
// with 164 (1920x960, 6 uint8 views, 8 iterations: 76.4, 76.1, 76.9, 77.7). Set
// once per kernel and device; a failure leaves the driver's choice.
template <auto KERNEL>
inline void prefer_texture_cache() {
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64 || (done.load(std::memory_order_relaxed) >> dev) & 1) return;
    cudaFuncAttributes a;
    bool ok = cudaFuncGetAttributes(&a, KERNEL) == cudaSuccess;
    if (ok) {
        const int blocks = 65536 / (BLOCK_THREADS * ((a.numRegs + 7) / 8 * 8));
        const size_t need = (size_t)blocks * (a.sharedSizeBytes + 1024), most = 228 * 1024;  // 1 KB per block is the system's
        const int percent = (int)std::min<size_t>(100, (100 * need + most - 1) / most);
        ok = cudaFuncSetAttribute(KERNEL, cudaFuncAttributePreferredSharedMemoryCarveout, percent) == cudaSuccess;
    }
    if (!ok) cudaGetLastError();
    done.fetch_or(1ull << dev, std::memory_order_relaxed);
}

template <int NS, bool EXACT, int MODE, int WIN = 0, int TS = 0>
inline void launch_tiles(const PixelParams& p, cudaStream_t stream) {
    prefer_texture_cache<pixel_kernel<NS, EXACT, MODE, WIN, TS>>();
    pixel_kernel<NS, EXACT, MODE, WIN, TS><<<tile_grid<TS>(p), BLOCK_THREADS, 0, stream>>>(p);
}

// The window class of a problem: a fixed-window sweep instance where one exists.
__host__ __device__ inline int window_of(const PixelParams& p) {
    if (p.K == 6 && p.radius == 5 && p.stride == 2) return 1;
    if (p.K == 7 && p.radius == 3 && p.stride == 1) return 2;
    return 0;
}

// Initialisation or cost of every pixel, with the window fixed where a half-sweep's
// is. From 8 tiles an SM on a block scores both colours from one staged tile; where
// that leaves SMs idle, each colour gets its own blocks. 1920x960, 6 views, costs
// of given planes: 1.03 -> 0.94 ms.
template <int NS, bool EXACT, int MODE, int WIN>
inline void launch_score(const PixelParams& p, cudaStream_t stream) {
    prefer_texture_cache<pixel_kernel<NS, EXACT, MODE, WIN, 0>>();
    dim3 grid = tile_grid<0>(p);
    grid.z = (long long)grid.x * grid.y >= 8 * SM_COUNT ? 1 : 2;
    pixel_kernel<NS, EXACT, MODE, WIN, 0><<<grid, BLOCK_THREADS, 0, stream>>>(p);
}
template <int NS, bool EXACT, int MODE>
inline void launch_score(const PixelParams& p, cudaStream_t stream) {
    if constexpr (EXACT && NS >= 2) {
        const int win = window_of(p);
        if (win == 1) return launch_score<NS, EXACT, MODE, 1>(p, stream);
        if (win == 2) return launch_score<NS, EXACT, MODE, 2>(p, stream);
    }
    launch_score<NS, EXACT, MODE, 0>(p, stream);
}

// The bounded kernel's launch beside the pooled one's (see bounded_turn).
template <int NS, bool EXACT, int WIN>
inline void launch_bounded(const PixelParams& p, cudaStream_t stream) {
    if constexpr (has_bounded(NS, EXACT)) {
        if (p.close == nullptr || (p.iter == 0 && p.colour == 0)) return;
        prefer_texture_cache<bounded_kernel<NS, WIN>>();
        bounded_kernel<NS, WIN><<<tile_grid<0>(p), BLOCK_THREADS, 0, stream>>>(p);
    }
}

// The tile shape of a half-sweep: the one asked for, else 32x8 with as many lanes
// per pixel as its tiles, with those of the keyframes beside it, leave room for
// (tiles x lanes within 5/6 of the resident blocks). Whole runs, ms at 1, 2, 4 and 8
// lanes: 64x32 of 2 views (8 tiles) 1.59 1.08 0.83 0.72; 256x128 (128 tiles) of 2 views
// 1.66 1.22 1.18 1.39, of 6 views 3.47 2.83 3.12 3.59; 320x160 of 4 (200) 2.02 1.66 1.94
// 2.13; 384x192 (288) of 2 views 1.91 1.69 2.10 2.42, of 6 views 4.55 4.62 5.51 6.66;
// 512x256 of 2 (512) 2.63 2.81 3.19 3.96.
template <int NS>
inline int sweep_shape(const PixelParams& p) {
    if (p.tile != 0) return p.tile;
    const long long tiles = (long long)((p.W + TILE_W - 1) / TILE_W) * ((p.H + TILE_H - 1) / TILE_H) + p.crowd;
    const long long resident = (long long)SM_COUNT * pixel_min_blocks(NS);
    return 8 * tiles * 6 <= resident * 5 ? 5 : 4 * tiles * 6 <= resident * 5 ? 4 : 2 * tiles * 6 <= resident * 5 ? 3 : 0;
}

// A sweep in its tile shape.
template <int NS, bool EXACT, int WIN>
inline void launch_sweep_window(const PixelParams& p, cudaStream_t stream) {
    switch (sweep_shape<NS>(p)) {
        case 1: launch_tiles<NS, EXACT, MODE_SWEEP, WIN, WIN ? 1 : 0>(p, stream); break;
        case 2: launch_tiles<NS, EXACT, MODE_SWEEP, WIN, WIN ? 2 : 0>(p, stream); break;
        case 3: launch_tiles<NS, EXACT, MODE_SWEEP, WIN, 3>(p, stream); break;
        case 4: launch_tiles<NS, EXACT, MODE_SWEEP, WIN, 4>(p, stream); break;
        case 5: launch_tiles<NS, EXACT, MODE_SWEEP, WIN, 5>(p, stream); break;
        default: launch_tiles<NS, EXACT, MODE_SWEEP, WIN, 0>(p, stream); launch_bounded<NS, EXACT, WIN>(p, stream); break;
    }
}

// Half-sweeps with 2 or 4 threads per pixel: the views split over warps
// (pixel_split.cuh, PixelParams::tpp 2 or 4) or the patch samples split over
// adjacent lanes (pixel_lanes.cuh, tpp -2, -4 or -8).
template <int NS, bool EXACT>
cudaError_t launch_split_sweep(const PixelParams& p, cudaStream_t stream);
template <int NS, bool EXACT>
cudaError_t launch_lanes_sweep(const PixelParams& p, cudaStream_t stream);

template <int NS, bool EXACT>
cudaError_t launch_pixel_kernel_ns(const PixelParams& p, int mode, cudaStream_t stream) {
    switch (mode) {
        case MODE_COST: launch_score<NS, EXACT, MODE_COST>(p, stream); break;
        case MODE_INIT: launch_score<NS, EXACT, MODE_INIT>(p, stream); break;
        default:
            // views split over several warps per pixel (a tuning choice; same maps)
            if constexpr (EXACT && NS >= 2) {
                if (p.tpp > 1) return launch_split_sweep<NS, EXACT>(p, stream);
                if (p.tpp < -1) return launch_lanes_sweep<NS, EXACT>(p, stream);
            }
            // the half-sweep dominates the run time: fixed-window instances for the
            // paired path (exact view counts of at least 2), in three tile shapes
            if constexpr (EXACT && NS >= 2) {
                const int win = window_of(p);
                if (win == 1) {
                    launch_sweep_window<NS, EXACT, 1>(p, stream);
                    break;
                }
                if (win == 2) {
                    launch_sweep_window<NS, EXACT, 2>(p, stream);
                    break;
                }
            }
            launch_sweep_window<NS, EXACT, 0>(p, stream);
            break;
    }
    return cudaGetLastError();
}

}  // namespace pmsp
