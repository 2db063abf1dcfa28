// Shared device helpers for the GSta kernels (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gsta.h"

namespace gs {

constexpr int kRow = 64;    // floats per parameter row (59 used)
constexpr int kSplat = 12;  // floats per projected splat record
constexpr int kG2d = 12;    // floats per raster-gradient row (9 used)
constexpr unsigned kFull = 0xffffffffu;

// Kernel-argument copy of gs_camera plus derived constants.
struct DevCam {
    int W, H, tile, tiles_x, tiles_y;
    float fx, fy, cx, cy;
    float R[9], t[3], campos[3];
    float znear, dilation;
    float bg[3];
    float limx, limy;  // 1.3 x tan(half field of view), the Jacobian clamp
};

inline bool tile_ok(int t) { return t == 8 || t == 16 || t == 32; }

inline bool camera_ok(const gs_camera *c) {
    if (!c) return false;
    if (c->width <= 0 || c->height <= 0 || c->width > 16384 || c->height > 16384) return false;
    if (!tile_ok(c->tile)) return false;
    if (!(c->fx > 0.f) || !(c->fy > 0.f)) return false;
    if (!(c->znear >= 0.f) || !(c->dilation >= 0.f)) return false;
    return true;
}

__host__ __device__ inline DevCam make_cam(const gs_camera *c) {
    DevCam d;
    d.W = c->width;
    d.H = c->height;
    d.tile = c->tile;
    d.tiles_x = (c->width + c->tile - 1) / c->tile;
    d.tiles_y = (c->height + c->tile - 1) / c->tile;
    d.fx = c->fx; d.fy = c->fy; d.cx = c->cx; d.cy = c->cy;
    for (int i = 0; i < 9; ++i) d.R[i] = c->R[i];
    for (int i = 0; i < 3; ++i) { d.t[i] = c->t[i]; d.campos[i] = c->campos[i]; d.bg[i] = c->bg[i]; }
    d.znear = c->znear;
    d.dilation = c->dilation;
    d.limx = 1.3f * 0.5f * (float)c->width / c->fx;
    d.limy = 1.3f * 0.5f * (float)c->height / c->fy;
    return d;
}

inline cudaStream_t as_stream(gs_stream_t s) { return reinterpret_cast<cudaStream_t>(s); }

// Adds k to the library-wide count of kernel launches (gs_launch_count).
void note_launches(int k);

inline int launch_status() { return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA; }

// Whether a launch or another runtime call was accepted; a refusal is taken off
// the runtime's record of the last error, since the caller returns it.
inline bool accepted(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
}

// Two float32 values in one 64-bit register pair, and the packed FP32
// instructions of sm_100 and later (add/sub/mul/fma .rn .f32x2): each half is
// rounded exactly as the scalar __fadd_rn / __fsub_rn / __fmul_rn / __fmaf_rn
// of the same operands, and one instruction issues both.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void f2_unpack(f32x2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ f32x2 f2_sub(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Programmatic dependent launch: a kernel started by launch_chained may be
// scheduled while the kernel before it in the stream is still finishing, so
// that its launch overlaps that kernel's last blocks. It must call
// wait_prior_grid() before anything else: griddepcontrol.wait returns once
// the grids it depends on have completed and their memory operations are
// visible (at once when it was launched without a dependency).
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained_smem(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                       Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, Args &&...args) {
    return launch_chained_smem(kernel, grid, block, 0, s, static_cast<Args &&>(args)...);
}

inline unsigned grid_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// Tile rectangle of a splat, decided in float32 with explicitly rounded
// operations: x0 = floor((mx - r) / tile), x1 = floor((mx + r) / tile),
// clipped to the grid. Writes the half-open rectangle; returns the count.
__device__ __forceinline__ int tile_rect(float mx, float my, int r, int tile, int tx, int ty, int &x0, int &y0,
                                         int &x1, int &y1) {
    float inv = 1.0f / (float)tile;  // exact: tile is a power of two
    float fr = (float)r;
    float fx0 = floorf(__fmul_rn(__fsub_rn(mx, fr), inv));
    float fx1 = floorf(__fmul_rn(__fadd_rn(mx, fr), inv));
    float fy0 = floorf(__fmul_rn(__fsub_rn(my, fr), inv));
    float fy1 = floorf(__fmul_rn(__fadd_rn(my, fr), inv));
    fx0 = fmaxf(fx0, 0.0f);
    fy0 = fmaxf(fy0, 0.0f);
    fx1 = fminf(fx1, (float)(tx - 1));
    fy1 = fminf(fy1, (float)(ty - 1));
    if (fx0 > fx1 || fy0 > fy1) {
        x0 = y0 = x1 = y1 = 0;
        return 0;
    }
    x0 = (int)fx0;
    y0 = (int)fy0;
    x1 = (int)fx1 + 1;
    y1 = (int)fy1 + 1;
    return (x1 - x0) * (y1 - y0);
}

// Opacity from its parameter under the sigmoid activation; one definition
// for the projection and for the switch to the absolute-value activation,
// which must reproduce it bit for bit.
__device__ __forceinline__ float opacity_sigmoid(float x) { return 1.f / (1.f + expf(-x)); }

// Exponent of the 2-D Gaussian at offset (dx, dy), -0.5 (a dx^2 + c dy^2) -
// b dx dy, as a quadratic in dy whose coefficients depend on dx only:
// power = (c2 dy + c1) dy + c0 with c2 = -c/2, c1 = -b dx, c0 = -a dx^2 / 2.
// A thread's pixels share a column, so per splat it forms the row once and
// pays two fused multiply-adds per pixel. Every kernel rounds it the same
// way (explicit intrinsics), so forward and backward take identical skip
// decisions.
struct SplatRow {
    float c0, c1, c2;
};

__device__ __forceinline__ SplatRow splat_row(float dx, float a, float b, float c) {
    SplatRow r;
    r.c0 = __fmul_rn(__fmul_rn(-0.5f, a), __fmul_rn(dx, dx));
    r.c1 = __fmul_rn(-b, dx);
    r.c2 = __fmul_rn(-0.5f, c);
    return r;
}

__device__ __forceinline__ float splat_power(const SplatRow &r, float dy) {
    return __fmaf_rn(__fmaf_rn(r.c2, dy, r.c1), dy, r.c0);
}

// 2^x. Results below the normal range flush to zero; the composited alphas
// are compared with 1/255, so nothing downstream sees the difference, and the
// instruction needs none of the scaling that keeps subnormal results.
__device__ __forceinline__ float ex2_ftz(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 1 / x of an x in [0.01, 1] (within one unit in the last place, as the
// division by it was; no scaling for extreme operands).
__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

constexpr float kLog2e = 1.44269504088896341f;  // exp(x) = 2^(x log2 e)

// exp(power), the one formula of every kernel that decides whether a splat is
// blended (the rasteriser's packed steps take the product for two pixels at once).
__device__ __forceinline__ float splat_falloff(float power) { return ex2_ftz(__fmul_rn(power, kLog2e)); }

template <int N>
struct IntC {  // a compile-time integer passed as an argument
    static constexpr int value = N;
};

constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kAlphaMax = 0.99f;
constexpr float kTMin = 1e-4f;

// Block-wide exclusive scan of one int per thread (blockDim.x <= 1024, a
// multiple of 32). Returns the exclusive prefix; *total gets the block sum.
// `warp_sums` must hold 32 ints of shared memory.
__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int *total) {
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < nwarps ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;  // inclusive prefix over warps
    }
    __syncthreads();
    int before = warp > 0 ? warp_sums[warp - 1] : 0;
    *total = warp_sums[nwarps - 1];
    __syncthreads();
    return before + x - v;
}

// The order in which a rasteriser's blocks take the tiles. Longest list first:
// the blocks that start last are then the short ones, and no SM waits for one
// long tile that started late (in ascending tiles the SMs were busy for 64-90% of
// the rasteriser's time). The sort leaves the order by list length at the front of
// its workspace, marked with the grid it is for; a training step's backward
// takes them by the depth that the forward's walk reached. 1M Gaussians, 1237 x
// 822, 8-pixel tiles: forward 136 -> 123 us, backward 355 -> 296 (nothing frozen)
// and 167 -> 137 us (95% frozen); by list length 320 and 144. 120K at 800 x 800,
// 16-pixel tiles, half frozen: 44 -> 37 and 82 -> 75 us.
struct TileOrder {
    const uint32_t *order;  // [tiles]; NULL: ascending tiles
    const uint2 *stamp;     // read and compared with key where the caller vouches for nothing; NULL: order is good
    uint2 key;
};

// Fewer tiles than this start all at once, whatever their order (three blocks
// of 16 x 16 pixels on each of 152 SMs).
constexpr int kOrderMinTiles = 456;

__host__ __device__ inline uint2 tile_order_key(int tiles_x, int tiles_y, int tile) {
    return make_uint2((uint32_t)tiles_x | ((uint32_t)tiles_y << 16), 0x67530000u | (uint32_t)tile);
}

// The tile of this block (each lane of a warp calls it). The reduction hands
// the compiler a value that is the same in every lane: with the plain load what is
// derived from the tile takes vector registers and the backward 12% more time.
__device__ __forceinline__ int ordered_tile(const TileOrder &o) {
    if (!o.order) return (int)blockIdx.x;
    uint32_t t = o.order[blockIdx.x];
    if (o.stamp) {
        const uint2 s = *o.stamp;
        if (s.x != o.key.x || s.y != o.key.y) t = blockIdx.x;
    }
    return (int)__reduce_min_sync(kFull, min(t, gridDim.x - 1));
}

// What the sort keeps at the front of its workspace, whatever the other sizes.
struct SortFront {
    uint2 *stamp;
    uint32_t *order;       // [tiles] by list length
    int32_t *depth;        // [tiles] zeroed by the sort: the list position the forward's walk reaches
    uint32_t *order_deep;  // [tiles] by depth
    uint32_t *hist, *next;  // [kLenBuckets] zeroed by the sort: tiles per bucket of depth, places given out
    size_t bytes;
};

constexpr int kLenBuckets = 256;

inline SortFront sort_front(void *ws, int64_t tiles) {
    char *p = static_cast<char *>(ws);
    const size_t each = ((size_t)tiles * 4 + 255) & ~size_t(255);
    return SortFront{reinterpret_cast<uint2 *>(p), reinterpret_cast<uint32_t *>(p + 256),
                     reinterpret_cast<int32_t *>(p + 256 + each), reinterpret_cast<uint32_t *>(p + 256 + 2 * each),
                     reinterpret_cast<uint32_t *>(p + 256 + 3 * each),
                     reinterpret_cast<uint32_t *>(p + 256 + 3 * each) + kLenBuckets,
                     256 + 3 * each + 8 * kLenBuckets};
}

// Bucket of a list length, eight to an octave.
__device__ __forceinline__ int length_bucket(uint32_t len) {
    return len ? min(kLenBuckets - 1, 1 + (int)((__float_as_uint((float)len) - 0x3f800000u) >> 20)) : 0;
}

// Adds one to bin[b] for every lane whose `in` is set and returns its place
// among them; equal bins of a warp take one addition.
__device__ __forceinline__ uint32_t take_place(uint32_t *bin, int b, bool in) {
    const unsigned same = __match_any_sync(kFull, in ? b : -1);
    const int lane = threadIdx.x & 31, leader = __ffs((int)same) - 1;
    uint32_t at = 0;
    if (in && lane == leader) at = atomicAdd(bin + b, (uint32_t)__popc(same));
    at = __shfl_sync(kFull, at, leader);
    return at + (uint32_t)__popc(same & ((1u << lane) - 1u));
}

// A counting sort of the tiles by bucket, longest first, by blocks of 256 threads
// with Q tiles per thread each; the first kernel counts them, a later one gives
// out the places.
template <int Q, class Len>
__device__ __forceinline__ void count_buckets(int block, int tiles, Len len, uint32_t *bins /* shared [kLenBuckets] */,
                                              uint32_t *hist) {
    bins[threadIdx.x] = 0u;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int t = (block * Q + q) * kLenBuckets + (int)threadIdx.x;
        take_place(bins, t < tiles ? length_bucket(len(t)) : -1, t < tiles);
    }
    __syncthreads();
    if (bins[threadIdx.x]) atomicAdd(hist + threadIdx.x, bins[threadIdx.x]);
    __syncthreads();
}

template <int Q, class Len, class Put>
__device__ __forceinline__ void place_buckets(int block, int tiles, Len len, Put put, const uint32_t *hist,
                                              uint32_t *next, uint32_t *s /* shared [3 * kLenBuckets + 32] */) {
    uint32_t *start = s, *mine = s + kLenBuckets, *base = s + 2 * kLenBuckets;
    const int b0 = kLenBuckets - 1 - (int)threadIdx.x;
    int b[Q], all;
    uint32_t at[Q];
    mine[threadIdx.x] = 0u;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int t = (block * Q + q) * kLenBuckets + (int)threadIdx.x;
        b[q] = t < tiles ? length_bucket(len(t)) : -1;
    }
    start[b0] = (uint32_t)block_exclusive_scan((int)hist[b0], reinterpret_cast<int *>(s + 3 * kLenBuckets), &all);
#pragma unroll
    for (int q = 0; q < Q; ++q) at[q] = take_place(mine, b[q], b[q] >= 0);
    __syncthreads();
    if (mine[threadIdx.x]) base[threadIdx.x] = start[threadIdx.x] + atomicAdd(next + threadIdx.x, mine[threadIdx.x]);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q)
        if (b[q] >= 0) put((block * Q + q) * kLenBuckets + (int)threadIdx.x, base[b[q]] + at[q]);
    __syncthreads();
}

}  // namespace gs
