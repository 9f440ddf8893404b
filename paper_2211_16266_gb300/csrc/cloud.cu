// Point kernels around the densification path: the View Filter on sparse
// points (paper Sec. III-A, Eq. 1), dense point-cloud fusion with duplicate
// erasure (Sec. III) and keyframe completeness (Sec. IV).
//
// View Filter: one thread per point computes the cosine of the parallax angle
//   between the rays to the two camera centres and tests it against the cosines
//   of the angle bounds; in-range points are counted with a warp ballot and one
//   atomic add per warp.
// Fusion: every valid pixel of every keyframe is lifted to a world point and
//   binned into a cubic voxel; an open-addressing hash table (linear probing,
//   64-bit packed voxel keys) keeps per voxel its smallest pixel (numbered through
//   the keyframes) by an atomic minimum. The kept pixels then set their bit in a
//   bitmap of all pixels, the bits are counted, and the marked points are written
//   in (keyframe, pixel) order, so the output does not depend on thread timing.
//   Bound by the atomics on the table: a wall at 2 m covers a 2 cm voxel with
//   about 10 pixels of a 1920x960 panorama, so a pixel whose left or upper
//   neighbour falls into the same voxel (a smaller index: it cannot be the voxel's
//   first) stays out, and the table is sized for a quarter of the pixels at first
//   (16 bytes a slot, key and pixel in one sector; 6 keyframes at 1920x960 take
//   64 MB, within L2, where two slots per pixel took 512 MB). The pixels left are
//   listed per tile, so that full warps wait for the table together. A table that
//   fills up is reported, with the candidates left, and the caller comes again with
//   one that has room for them. 6 keyframes
//   at 1920x960, 1 M voxels: 85 us insertion (was 198 over 6 launches), 33 us
//   marks, scan and points (was 280), against 10 us for its 64 MB of maps, points
//   and origins; the whole call with its count-only first pass 1.39 -> 0.45 ms.
// Completeness: one thread per point projects into a W x H panorama and sets
//   the nearest pixel's flag; a reduction counts the flags.
#include <algorithm>

#include "camera.cuh"
#include "common.cuh"

namespace pmsp {

namespace {

constexpr unsigned long long EMPTY = ~0ull;
constexpr int KEY_BITS = 21;
constexpr long long KEY_HALF = 1ll << (KEY_BITS - 1);

// World point of range d along the ray r of a pixel.
__device__ __forceinline__ float3 lift_along(const CloudView& V, float3 r, float d) {
    const float x = fmaf(d, r.x, -V.t[0]), y = fmaf(d, r.y, -V.t[1]), z = fmaf(d, r.z, -V.t[2]);
    // X = R^T (d r - t)
    return make_float3(fmaf(V.R[0], x, fmaf(V.R[3], y, V.R[6] * z)), fmaf(V.R[1], x, fmaf(V.R[4], y, V.R[7] * z)),
                       fmaf(V.R[2], x, fmaf(V.R[5], y, V.R[8] * z)));
}

// Packed voxel key (21 bits per axis, offset binary); false if out of range.
__device__ __forceinline__ bool voxel_key(float3 X, float inv_voxel, unsigned long long& key) {
    const float q[3] = {floorf(X.x * inv_voxel), floorf(X.y * inv_voxel), floorf(X.z * inv_voxel)};
    key = 0;
    unsigned part[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (!(q[a] >= -(float)KEY_HALF && q[a] < (float)KEY_HALF)) return false;
        part[a] = (unsigned)((int)q[a] + (int)KEY_HALF);
    }
    key = ((unsigned long long)part[0] << (2 * KEY_BITS)) | ((unsigned long long)part[1] << KEY_BITS) | part[2];
    return true;
}

__device__ __forceinline__ unsigned long long hash_slot(unsigned long long key, unsigned long long mask) {
    key ^= key >> 33;
    key *= 0xff51afd7ed558ccdull;
    key ^= key >> 33;
    key *= 0xc4ceb9fe1a85ec53ull;
    key ^= key >> 33;
    return key & mask;
}

constexpr int FT_W = 32, FT_H = 8, FT_V = 4;  // threads of a block, pixels of a thread (every eighth row of a 32 x 32 tile)
// Keyframe and tile of block b: the keyframes' tiles are numbered one after another.
__device__ __forceinline__ int fuse_view(const FuseArgs& A, int b) {
    int k = 0;
    while (k + 1 < A.n && b >= A.tile_base[k + 1]) ++k;
    return k;
}

__global__ void __launch_bounds__(FT_W * FT_H) fuse_insert_kernel(const __grid_constant__ FuseArgs A) {
    __shared__ float2 row[FT_H * FT_V], col[FT_W];  // (sin, cos) of latitude and longitude, as pixel_bearing
    __shared__ unsigned long long keys[FT_H * FT_V][FT_W];
    __shared__ unsigned short list[FT_H * FT_V * FT_W];
    __shared__ unsigned claimed, full, listed, missed;
    const int k = fuse_view(A, blockIdx.x), b = blockIdx.x - A.tile_base[k];
    const CloudView& V = A.views[k];
    const int tiles_x = (V.W + FT_W - 1) / FT_W;
    const int u0 = (b % tiles_x) * FT_W, v0 = (b / tiles_x) * FT_H * FT_V;
    const int u = u0 + threadIdx.x, tid = threadIdx.y * FT_W + threadIdx.x;
    float d[FT_V];
#pragma unroll
    for (int p = 0; p < FT_V; ++p) {
        const int v = v0 + threadIdx.y + p * FT_H;
        d[p] = u < V.W && v < V.H ? V.depth[v * V.W + u] : 0.f;
    }
    if (tid < FT_W + FT_H * FT_V) {
        float sn, cs;
        if (tid < FT_W) {
            sincospif((2.0f * (u0 + tid) + 1.0f) / V.W - 1.0f, &sn, &cs);
            col[tid] = make_float2(sn, cs);
        } else {
            sincospif(0.5f - (2.0f * (v0 + tid - FT_W) + 1.0f) / (2.0f * V.H), &sn, &cs);
            row[tid - FT_W] = make_float2(sn, cs);
        }
    } else if (tid == FT_W * FT_H - 1) {
        claimed = listed = missed = 0;
        full = *(volatile unsigned*)A.err & ERR_CAPACITY;  // the caller will come again: nothing more is worth doing
        const unsigned long long now = *(volatile unsigned long long*)A.count, voxels = (unsigned)now, tiles = now >> 32;
        if (!full && (voxels > A.most_voxels ||
                      (A.foresee && 2 * tiles >= gridDim.x && 5 * voxels * gridDim.x > 6 * A.most_voxels * tiles))) {
            full = 1;
            atomicOr(A.err, ERR_CAPACITY);
        }
    }
    __syncthreads();
    unsigned long long key[FT_V];
#pragma unroll
    for (int p = 0; p < FT_V; ++p) {
        key[p] = EMPTY;
        if (d[p] > 0.f) {
            const float2 r = row[threadIdx.y + p * FT_H], c = col[threadIdx.x];
            const float3 X = lift_along(V, make_float3(r.y * c.x, -r.x, r.y * c.y), d[p]);
            if (!voxel_key(X, A.inv_voxel, key[p])) {
                key[p] = EMPTY;
                atomicOr(A.err, ERR_RANGE);
            }
        }
        keys[threadIdx.y + p * FT_H][threadIdx.x] = key[p];
    }
    __syncthreads();
    // the tile's candidates in a list, so that the insertion runs with full warps
#pragma unroll
    for (int p = 0; p < FT_V; ++p) {
        const int y = threadIdx.y + p * FT_H;
        bool first = key[p] != EMPTY;
        if (first && threadIdx.x > 0) first = keys[y][threadIdx.x - 1] != key[p];
        if (first && y > 0) first = keys[y - 1][threadIdx.x] != key[p];
        const unsigned m = __ballot_sync(0xffffffffu, first);
        unsigned at = 0;
        if (threadIdx.x == 0 && m) at = atomicAdd(&listed, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << threadIdx.x) - 1u));
        if (first) list[at] = (unsigned short)(y * FT_W + threadIdx.x);
    }
    __syncthreads();
    if (full) {
        if (tid == 0 && listed) atomicAdd(A.left, (unsigned long long)listed);
        return;
    }
    unsigned won = 0;
    for (int c = tid; c < (int)listed; c += FT_W * FT_H) {
        const int y = list[c] / FT_W, x = list[c] % FT_W;
        const unsigned long long mine = keys[y][x];
        unsigned long long s = hash_slot(mine, A.mask), probe = 0;
        for (; probe < A.most_probes; ++probe) {  // bounded: at most one pass over the table
            FuseSlot* t = A.table + s;
            unsigned long long seen = *(volatile unsigned long long*)&t->key;
            if (seen == EMPTY) {
                seen = atomicCAS(&t->key, EMPTY, mine);
                won += seen == EMPTY;
            }
            if (seen == EMPTY || seen == mine) {
                atomicMin(&t->pixel, (unsigned)(A.base[k] + (v0 + y) * V.W + u0 + x));
                break;
            }
            s = (s + 1) & A.mask;
        }
        if (probe == A.most_probes) {
            atomicOr(A.err, ERR_CAPACITY);
            atomicAdd(&missed, 1u);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) won += __shfl_xor_sync(0xffffffffu, won, o);
    if (threadIdx.x == 0 && won) atomicAdd(&claimed, won);
    __syncthreads();
    if (tid == 0) {
        atomicAdd(A.count, (1ull << 32) | claimed);
        if (missed) atomicAdd(A.left, (unsigned long long)missed);
    }
}

// Sets the bit of every slot's pixel.
__global__ void __launch_bounds__(256) fuse_mark_kernel(const __grid_constant__ FuseArgs A) {
    if (*A.err & ERR_CAPACITY) return;  // the caller will come again
    for (unsigned long long s = (unsigned long long)blockIdx.x * 256 + threadIdx.x; s <= A.mask; s += (unsigned long long)gridDim.x * 256) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(A.table + s);
        if (t.x == EMPTY) continue;
        const unsigned p = (unsigned)t.y;
        atomicOr(A.bits + (p >> 5), 1u << (p & 31));
    }
}

constexpr int SCAN_BLOCK = 256;  // bitmap words (32 pixels each) of a block of the two passes below
constexpr int FEW_GROUPS = 8;    // up to so many blocks the writing pass counts for itself

__device__ __forceinline__ unsigned block_sum(unsigned x, unsigned* warp_sums) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = x;
    __syncthreads();
    unsigned s = 0;
    for (int w = 0; w < SCAN_BLOCK / 32; ++w) s += warp_sums[w];
    __syncthreads();
    return s;
}

__global__ void __launch_bounds__(SCAN_BLOCK) fuse_count_kernel(const __grid_constant__ FuseArgs A) {
    __shared__ unsigned ws[SCAN_BLOCK / 32];
    const int w = blockIdx.x * SCAN_BLOCK + threadIdx.x;
    const unsigned s = block_sum(w < A.n_words ? __popc(A.bits[w]) : 0, ws);
    if (threadIdx.x == 0) A.sums[blockIdx.x] = s;
}

// The groups' sums to the marks before each group, by one block.
__global__ void __launch_bounds__(1024) fuse_scan_kernel(unsigned* sums, int groups) {
    __shared__ unsigned ws[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned carry = 0;
    for (int c = 0; c < groups; c += 1024) {
        const int q = c + threadIdx.x;
        const unsigned x = q < groups ? sums[q] : 0;
        unsigned incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) ws[warp] = incl;
        __syncthreads();
        unsigned before = carry;
        for (int w = 0; w < warp; ++w) before += ws[w];
        if (q < groups) sums[q] = before + incl - x;
        for (int w = 0; w < 32; ++w) carry += ws[w];
        __syncthreads();
    }
}

// Writes the marked points of a group of 256 words, a thread per point: its word
// by bisection of the marks before each, its bit within the word by halving.
// (A lane per pixel instead kept 3 of 32 lanes busy: 53 us for what takes 12.)
// A group's points go to gridDim.y blocks: one block each left small inputs to a
// few SMs. Up to FEW_GROUPS groups the marks before a group are counted here, which
// saves two launches. Calls with room for every point: 64x32 110 -> 102 us, 2 of 256x128
// 133 -> 108, 1 of 1920x960 at 1.39M voxels 192 -> 181.
__global__ void __launch_bounds__(SCAN_BLOCK) fuse_write_kernel(const __grid_constant__ FuseArgs A) {
    __shared__ unsigned ws[SCAN_BLOCK / 32], words[SCAN_BLOCK], before[SCAN_BLOCK];
    if (*A.err & ERR_CAPACITY) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int w0 = blockIdx.x * SCAN_BLOCK;
    const unsigned own = w0 + threadIdx.x < A.n_words ? A.bits[w0 + threadIdx.x] : 0;
    unsigned incl = __popc(own);
    const unsigned mine = incl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    unsigned ahead = 0, total = 0;
    for (int w = 0; w < SCAN_BLOCK / 32; ++w) {
        if (w < warp) ahead += ws[w];
        total += ws[w];
    }
    words[threadIdx.x] = own;
    before[threadIdx.x] = ahead + incl - mine;
    __syncthreads();
    long long start;
    if (gridDim.x > FEW_GROUPS) {
        start = A.sums[blockIdx.x];
    } else {  // the groups before this one are counted here
        unsigned x = 0;
        for (int w = threadIdx.x; w < w0; w += SCAN_BLOCK) x += __popc(A.bits[w]);
        start = block_sum(x, ws);
    }
    for (unsigned q = blockIdx.y * SCAN_BLOCK + threadIdx.x; q < total && start + q < A.cap; q += gridDim.y * SCAN_BLOCK) {
        int w = 0;
#pragma unroll
        for (int h = SCAN_BLOCK / 2; h > 0; h >>= 1)
            if (before[w + h] <= q) w += h;  // the last word with at most q marks before it has the mark
        unsigned bits = words[w], n = q - before[w];
        int bit = 0;
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) {
            const unsigned c = __popc(bits & ((1u << h) - 1u));
            if (n >= c) {
                n -= c;
                bits >>= h;
                bit += h;
            }
        }
        const long long g = ((long long)(w0 + w) << 5) + bit;  // pixel, numbered through the keyframes
        int k = 0;
        while (k + 1 < A.n && g >= A.base[k + 1]) ++k;
        const CloudView& V = A.views[k];
        const int i = (int)(g - A.base[k]);
        const float3 X = lift_along(V, pixel_bearing(i % V.W, i / V.W, V.W, V.H), V.depth[i]);
        float* o = A.points + 3 * (start + q);
        o[0] = X.x;
        o[1] = X.y;
        o[2] = X.z;
        if (A.src) A.src[start + q] = (long long)(((unsigned long long)k << 32) | (unsigned)i);
    }
}

__global__ void completeness_kernel(const __grid_constant__ CompletenessArgs A) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    const float* p = A.points + 3 * i;
    const float X = p[0], Y = p[1], Z = p[2];
    const float y0 = fmaf(A.R[0], X, fmaf(A.R[1], Y, fmaf(A.R[2], Z, A.t[0])));
    const float y1 = fmaf(A.R[3], X, fmaf(A.R[4], Y, fmaf(A.R[5], Z, A.t[1])));
    const float y2 = fmaf(A.R[6], X, fmaf(A.R[7], Y, fmaf(A.R[8], Z, A.t[2])));
    if (y0 == 0.f && y1 == 0.f && y2 == 0.f) return;  // at the camera centre: no direction
    float uc, vc;
    project_dir_fast(y0, y1, y2, A.su, A.ou, A.sv, A.ov, uc, vc);
    int u = (int)floorf(uc + 0.5f) % A.W;
    if (u < 0) u += A.W;
    int v = (int)floorf(vc + 0.5f);
    v = v < 0 ? 0 : (v > A.H - 1 ? A.H - 1 : v);
    A.hit[(size_t)v * A.W + u] = 1;
}

__global__ void count_hits_kernel(const unsigned char* hit, long long n, unsigned long long* count) {
    unsigned c = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        c += hit[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, (unsigned long long)c);
}

__global__ void view_filter_kernel(const __grid_constant__ ViewFilterArgs A) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool ok = false;
    if (i < A.n) {
        const float* p = A.points + 3 * i;
        const float ax = A.ca[0] - p[0], ay = A.ca[1] - p[1], az = A.ca[2] - p[2];
        const float bx = A.cb[0] - p[0], by = A.cb[1] - p[1], bz = A.cb[2] - p[2];
        const float la = fmaf(ax, ax, fmaf(ay, ay, az * az)), lb = fmaf(bx, bx, fmaf(by, by, bz * bz));
        if (la > 0.f && lb > 0.f) {
            const float c = fmaf(ax, bx, fmaf(ay, by, az * bz)) / sqrtf(la * lb);
            ok = c >= A.cos_max && c <= A.cos_min;  // theta in [min, max] <=> cos in [cos max, cos min]
        }
        if (A.flags) A.flags[i] = ok;
    }
    const unsigned votes = __ballot_sync(0xffffffffu, ok);
    if ((threadIdx.x & 31) == 0 && votes) atomicAdd(A.count, (unsigned long long)__popc(votes));
}

}  // namespace

int fuse_tiles(int W, int H) { return ((W + FT_W - 1) / FT_W) * ((H + FT_H * FT_V - 1) / (FT_H * FT_V)); }

cudaError_t launch_fuse(const FuseArgs& a, cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(a.table, 0xff, (a.mask + 1) * sizeof(FuseSlot), stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(a.count, 0, 3 * sizeof(unsigned long long), stream);  // and the words after it
    if (e != cudaSuccess) return e;
    fuse_insert_kernel<<<a.tile_base[a.n], dim3(FT_W, FT_H), 0, stream>>>(a);
    if (a.cap > 0) {  // else the count is all that is asked for
        e = cudaMemsetAsync(a.bits, 0, (size_t)a.n_words * sizeof(unsigned), stream);
        if (e != cudaSuccess) return e;
        const int blocks = (a.n_words + SCAN_BLOCK - 1) / SCAN_BLOCK;
        fuse_mark_kernel<<<(unsigned)std::min<unsigned long long>((a.mask + 256) / 256, 8192), 256, 0, stream>>>(a);
        if (blocks > FEW_GROUPS) {
            fuse_count_kernel<<<blocks, SCAN_BLOCK, 0, stream>>>(a);
            fuse_scan_kernel<<<1, 1024, 0, stream>>>(a.sums, blocks);
        }
        const int split = std::min(std::max(8 * SM_COUNT / blocks, 1), 32);  // 32: a thread for every pixel of a group
        fuse_write_kernel<<<dim3(blocks, split), SCAN_BLOCK, 0, stream>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_completeness(const CompletenessArgs& a, unsigned long long* count, cudaStream_t stream) {
    const size_t px = (size_t)a.W * a.H;
    cudaError_t e = cudaMemsetAsync(a.hit, 0, px, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, sizeof *count, stream);
    if (e != cudaSuccess) return e;
    if (a.n > 0) completeness_kernel<<<(unsigned)((a.n + 255) / 256), 256, 0, stream>>>(a);
    count_hits_kernel<<<(unsigned)std::min<size_t>((px + 255) / 256, 4096), 256, 0, stream>>>(a.hit, (long long)px,
                                                                                          count);
    return cudaGetLastError();
}

cudaError_t launch_view_filter(const ViewFilterArgs& a, cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(a.count, 0, sizeof *a.count, stream);
    if (e != cudaSuccess) return e;
    if (a.n > 0) view_filter_kernel<<<(unsigned)((a.n + 255) / 256), 256, 0, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace pmsp
