// Training loss L = (1 - lambda) L1 + lambda (1 - SSIM) and dL/dimage
// (Sec. 3.1, Eq. 3), and the PSNR of Eq. 7's early-stop check (Sec. 3.2.2).
//
// SSIM uses the 11x11 Gaussian window (sigma 1.5) as two 1-D passes in
// shared memory (Sec. 3.3, "Accelerated SSIM loss calculation"): one kernel
// builds the five window moments of a 32x32 tile plus its 5-pixel halo and
// emits the SSIM map's three partial-derivative maps (two of them as one array
// of pairs); a second kernel runs the same separable window over those maps
// (the window is symmetric, so it is its own adjoint) and combines them with
// the L1 term into dL/dimage. Block partial sums are reduced in a fixed order,
// so the loss is deterministic.
#include "common.cuh"

namespace gs {

__device__ uint32_t g_loss_flags;

namespace {

constexpr int kT = 32;            // output tile edge
constexpr int kR = 5;             // window radius
constexpr int kE = kT + 2 * kR;   // tile edge with halo
constexpr int kLossThreads = 256;
constexpr int kLoadRows = kLossThreads / kE;  // haloed rows loaded per round (6; threads 252-255 idle)

struct Win {
    float w[11];
};

// Each pass gives a thread kV = 4 consecutive outputs, so that it reads the
// kV + 10 inputs of their windows once from shared memory instead of
// 11 per output. Horizontal items: (4 columns, row of the haloed tile), a warp
// on 32 rows; vertical items: (column, 4 rows), one per thread, a warp on 32
// columns.
//
// Quantities that share a weight go in pairs through the packed FP32
// instructions -- (x, y) and (x^2, y^2) with x y beside them in the forward,
// the first two maps with the third in the backward -- and lie interleaved in
// shared memory, so that a load brings a ready pair and no instruction is
// spent on packing. Every rounded operation is the scalar one's. Row strides
// of the arrays are 4 words times an odd number: 16-byte accesses of eight
// consecutive rows meet all 32 banks. The loss is reduced from the forward's
// partial sums by the backward's first block, so that the forward counts no
// blocks, fences nothing and no counter has to be cleared before it.
//
// Bound by instruction issue (66-71%) and, at its four blocks per SM, by the
// two barriers between the passes. 3 x 822 x 1237: 68.4 us with scalar passes, a
// counted last block and a cleared counter; 61.8 us with packed passes; 50.0 us
// with the reduction in the backward; 48.5 us with the backward's pixels loaded ahead
// of its last windows.
constexpr int kV = 4;
constexpr int kSeg = kT / kV;              // 8 segments per row / column
constexpr int kHItems = kE * kSeg;         // 336 horizontal items
constexpr int kH2 = kT + 2;                // pairs per row of the horizontal sums (68 words)
constexpr int kH1 = kT + 4;                // words per row of the third one (36)
constexpr int kE1 = kE + 2;                // words per row of a haloed single map (44); pairs need no padding (84)
static_assert(kT * kSeg == kLossThreads, "one vertical item per thread");

// Window sums of kV outputs from kV + 10 inputs, N packed quantities and one
// scalar: in(q, pairs, scalar) gives input q.
template <int N, class In>
__device__ __forceinline__ void window(const Win &win, In in, f32x2 (&p)[N][kV], float (&s)[kV]) {
#pragma unroll
    for (int v = 0; v < kV; ++v) {
#pragma unroll
        for (int k = 0; k < N; ++k) p[k][v] = f2_pack(0.f, 0.f);
        s[v] = 0.f;
    }
#pragma unroll
    for (int q = 0; q < kV + 10; ++q) {
        f32x2 x[N];
        float z;
        in(q, x, z);
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            const int t = q - v;  // tap of input q in output v's window
            if (t >= 0 && t < 11) {
                const float w = win.w[t];
                const f32x2 w2 = f2_pack(w, w);
#pragma unroll
                for (int k = 0; k < N; ++k) p[k][v] = f2_fma(w2, x[k], p[k][v]);
                s[v] = __fmaf_rn(w, z, s[v]);
            }
        }
    }
}

// The loss from the forward's per-block partial sums (L1 sum, SSIM sum), by the
// backward's first block: every thread sums a fixed stride of them in double,
// then a fixed-shape tree.
__device__ void loss_from_parts(const float2 *part, int nparts, int64_t N, float lambda, float *loss,
                                double *scratch /* shared, 2 * kLossThreads */) {
    double *r1 = scratch, *r2 = scratch + kLossThreads;
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < nparts; k += kLossThreads) {
        const float2 v = part[k];
        a += (double)v.x;
        b += (double)v.y;
    }
    r1[threadIdx.x] = a;
    r2[threadIdx.x] = b;
    __syncthreads();
    for (int w = kLossThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            r1[threadIdx.x] += r1[threadIdx.x + w];
            r2[threadIdx.x] += r2[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double L = (1.0 - lambda) * r1[0] / (double)N + lambda * (1.0 - r2[0] / (double)N);
        const float Lf = (float)L;
        if (!isfinite(Lf)) atomicOr(&g_loss_flags, GS_FLAG_NONFINITE);
        *loss = Lf;
    }
}

// Inside a training step the first blocks of the two kernels also make the order in
// which the rasteriser's backward takes the tiles: by the depth their walk
// reached in the forward, longest first, 256 tiles per block (one block for all
// of 16K tiles took 40 us longer than the kernel's others).
struct DepthOrder {
    int tiles;  // 0: none
    const int32_t *depth;
    uint32_t *order, *hist, *next;

    __device__ int block() const { return (int)((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x); }
    __device__ bool mine() const { return block() < (tiles + kLenBuckets - 1) / kLenBuckets; }
};
static_assert(kLossThreads == kLenBuckets, "a bucket per thread");

__global__ void __launch_bounds__(kLossThreads) k_ssim_fwd(const float *__restrict__ img,
                                                          const float *__restrict__ gt, int H, int W, Win win,
                                                          f32x2 *__restrict__ mapAB, float *__restrict__ mapC,
                                                          float2 *__restrict__ part, DepthOrder deep) {
    __shared__ __align__(16) f32x2 sxy[kE][kE];
    __shared__ __align__(16) f32x2 h[2][kE][kH2];
    __shared__ __align__(16) float hxy[kE][kH1];
    __shared__ float red[2][kLossThreads / 32];
    wait_prior_grid();
    if (deep.mine())
        count_buckets<1>(deep.block(), deep.tiles, [&](int t) { return (uint32_t)deep.depth[t]; },
                         reinterpret_cast<uint32_t *>(&hxy[0][0]), deep.hist);
    const int ch = blockIdx.z;
    const int64_t HW = (int64_t)H * W;
    const float *x = img + ch * HW, *y = gt + ch * HW;
    const int oy = blockIdx.y * kT - kR, ox = blockIdx.x * kT - kR;
    {   // thread t loads column t % kE of rows t / kE, + kLoadRows, ...: all its loads in flight together
        const int c = (int)threadIdx.x % kE, r0 = (int)threadIdx.x / kE;
        const int gx = ox + c;
        const bool col_in = gx >= 0 && gx < W;
        if (r0 < kLoadRows) {
#pragma unroll
            for (int r = r0; r < kE; r += kLoadRows) {
                const int gy = oy + r;
                const bool in = col_in && gy >= 0 && gy < H;
                const int64_t o = (int64_t)gy * W + gx;
                sxy[r][c] = f2_pack(in ? __ldg(x + o) : 0.f, in ? __ldg(y + o) : 0.f);
            }
        }
    }
    __syncthreads();
    // horizontal: window sums of (x, y), (x^2, y^2), x y along the rows
    for (int it = threadIdx.x; it < kHItems; it += kLossThreads) {
        const int r = it % kE, c0 = (it / kE) * kV;
        f32x2 in2[kV + 10];
#pragma unroll
        for (int q = 0; q < kV + 10; q += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&sxy[r][c0 + q]);
            in2[q] = v.x;
            in2[q + 1] = v.y;
        }
        f32x2 p[2][kV];
        float s[kV];
        window<2>(win, [&](int q, f32x2 (&o)[2], float &z) {
            float xv, yv;
            f2_unpack(in2[q], xv, yv);
            o[0] = in2[q];
            o[1] = f2_mul(in2[q], in2[q]);
            z = xv * yv;
        }, p, s);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
            for (int v = 0; v < kV; v += 2)
                *reinterpret_cast<ulonglong2 *>(&h[k][r][c0 + v]) = make_ulonglong2(p[k][v], p[k][v + 1]);
        }
        *reinterpret_cast<float4 *>(&hxy[r][c0]) = make_float4(s[0], s[1], s[2], s[3]);
    }
    __syncthreads();
    // vertical, then the SSIM map and its partial derivatives
    const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
    float l1 = 0.f, ss = 0.f;
    {
        const int c = threadIdx.x % kT, r0 = (threadIdx.x / kT) * kV;
        f32x2 p[2][kV];
        float xy[kV];
        window<2>(win, [&](int q, f32x2 (&o)[2], float &z) {
            o[0] = h[0][r0 + q][c];
            o[1] = h[1][r0 + q][c];
            z = hxy[r0 + q][c];
        }, p, xy);
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            const int r = r0 + v;
            const int gy = blockIdx.y * kT + r, gx = blockIdx.x * kT + c;
            if (gy >= H || gx >= W) continue;
            float mx, my, xx, yy, xc, yc;
            f2_unpack(p[0][v], mx, my);
            f2_unpack(p[1][v], xx, yy);
            f2_unpack(sxy[r + kR][c + kR], xc, yc);
            const float vx = xx - mx * mx, vy = yy - my * my, cxy = xy[v] - mx * my;
            const float n1 = 2.f * mx * my + C1, n2 = 2.f * cxy + C2;
            const float d1 = mx * mx + my * my + C1, d2 = vx + vy + C2;
            // d1 >= C1 and d2 >= C2 (up to rounding of the variances): the map
            // and its partials are formed without dividing by n1 or n2, which
            // may be zero (m / n2 = n1 / (d1 d2), m / n1 = n2 / (d1 d2))
            const float rd1 = __fdividef(1.f, d1), rd2 = __fdividef(1.f, d2);  // d1, d2 in [1e-4, 3]
            const float qd = rd1 * rd2;
            const float m_n1 = n2 * qd, m_n2 = n1 * qd;
            const float m = n1 * m_n1;
            ss += m;
            l1 += fabsf(xc - yc);
            // partials of the map value w.r.t. the window means of x, x^2 and x*y
            const int64_t o = ch * HW + (int64_t)gy * W + gx;
            mapAB[o] = f2_pack(2.f * my * (m_n1 - m_n2) + 2.f * mx * m * (rd2 - rd1), -m * rd2);
            mapC[o] = 2.f * m_n2;
        }
    }
    // block sums
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        l1 += __shfl_xor_sync(kFull, l1, o);
        ss += __shfl_xor_sync(kFull, ss, o);
    }
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = l1; red[1][threadIdx.x >> 5] = ss; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float a = 0.f, b = 0.f;
        for (int w = 0; w < kLossThreads / 32; ++w) { a += red[0][w]; b += red[1][w]; }
        int64_t blk = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        part[blk] = make_float2(a, b);
    }
}

__global__ void __launch_bounds__(kLossThreads, 5) k_ssim_bwd(const float *__restrict__ img,
                                                          const float *__restrict__ gt, int H, int W, Win win,
                                                          float lambda, const f32x2 *__restrict__ mapAB,
                                                          const float *__restrict__ mapC,
                                                          const float2 *__restrict__ part, float *__restrict__ loss,
                                                          float *__restrict__ dl, DepthOrder deep) {
    __shared__ __align__(16) f32x2 sab[kE][kE];
    __shared__ __align__(16) float sc[kE][kE1];
    __shared__ __align__(16) f32x2 h[kE][kH2];  // also the first block's reduction scratch
    __shared__ __align__(16) float hc[kE][kH1];
    static_assert(sizeof(h) >= 2 * kLossThreads * sizeof(double), "scratch fits");
    wait_prior_grid();
    const int ch = blockIdx.z;
    const int64_t HW = (int64_t)H * W;
    if (deep.mine())
        place_buckets<1>(deep.block(), deep.tiles, [&](int t) { return (uint32_t)deep.depth[t]; },
                         [&](int t, uint32_t at) { deep.order[at] = (uint32_t)t; }, deep.hist, deep.next,
                         reinterpret_cast<uint32_t *>(&hc[0][0]));
    if (blockIdx.x + blockIdx.y + blockIdx.z == 0)  // h is written again behind the next barrier
        loss_from_parts(part, (int)(gridDim.x * gridDim.y * gridDim.z), 3 * HW, lambda, loss,
                        reinterpret_cast<double *>(&h[0][0]));
    const int oy = blockIdx.y * kT - kR, ox = blockIdx.x * kT - kR;
    const f32x2 *ab = mapAB + ch * HW;
    const float *c = mapC + ch * HW;
    {
        const int q = (int)threadIdx.x % kE, r0 = (int)threadIdx.x / kE;
        const int gx = ox + q;
        const bool col_in = gx >= 0 && gx < W;
        if (r0 < kLoadRows) {
#pragma unroll
            for (int r = r0; r < kE; r += kLoadRows) {
                const int gy = oy + r;
                const bool in = col_in && gy >= 0 && gy < H;
                const int64_t o = (int64_t)gy * W + gx;
                sab[r][q] = in ? __ldg(ab + o) : 0ull;
                sc[r][q] = in ? __ldg(c + o) : 0.f;
            }
        }
    }
    __syncthreads();
    for (int it = threadIdx.x; it < kHItems; it += kLossThreads) {
        const int r = it % kE, c0 = (it / kE) * kV;
        f32x2 p[1][kV], in2[kV + 10];
        float s[kV], in1[kV + 12];
#pragma unroll
        for (int q = 0; q < kV + 10; q += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&sab[r][c0 + q]);
            in2[q] = v.x;
            in2[q + 1] = v.y;
        }
#pragma unroll
        for (int q = 0; q < kV + 10; q += 4) {  // the last two words are the row's padding
            const float4 v = *reinterpret_cast<const float4 *>(&sc[r][c0 + q]);
            in1[q] = v.x; in1[q + 1] = v.y; in1[q + 2] = v.z; in1[q + 3] = v.w;
        }
        window<1>(win, [&](int q, f32x2 (&o)[1], float &z) { o[0] = in2[q]; z = in1[q]; }, p, s);
#pragma unroll
        for (int v = 0; v < kV; v += 2)
            *reinterpret_cast<ulonglong2 *>(&h[r][c0 + v]) = make_ulonglong2(p[0][v], p[0][v + 1]);
        *reinterpret_cast<float4 *>(&hc[r][c0]) = make_float4(s[0], s[1], s[2], s[3]);
    }
    __syncthreads();
    const float invN = 1.f / (3.f * (float)HW);
    const int cc = threadIdx.x % kT, r0 = (threadIdx.x / kT) * kV;
    const int gx = blockIdx.x * kT + cc, gy0 = blockIdx.y * kT + r0;
    float xv[kV], yv[kV];  // on their way while the windows are summed
#pragma unroll
    for (int v = 0; v < kV; ++v) {
        const bool in = gx < W && gy0 + v < H;
        const int64_t o = ch * HW + (int64_t)(gy0 + v) * W + gx;
        xv[v] = in ? __ldg(img + o) : 0.f;
        yv[v] = in ? __ldg(gt + o) : 0.f;
    }
    f32x2 p[1][kV];
    float s0[kV], s1[kV], s2[kV];
    window<1>(win, [&](int q, f32x2 (&o)[1], float &z) { o[0] = h[r0 + q][cc]; z = hc[r0 + q][cc]; }, p, s2);
#pragma unroll
    for (int v = 0; v < kV; ++v) f2_unpack(p[0][v], s0[v], s1[v]);
#pragma unroll
    for (int v = 0; v < kV; ++v) {
        if (gx >= W || gy0 + v >= H) continue;
        const float d = xv[v] - yv[v];
        const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
        const float dssim = s0[v] + 2.f * xv[v] * s1[v] + yv[v] * s2[v];
        const float g = ((1.f - lambda) * sg - lambda * dssim) * invN;
        if (!isfinite(g)) atomicOr(&g_loss_flags, GS_FLAG_NONFINITE);
        dl[ch * HW + (int64_t)(gy0 + v) * W + gx] = g;
    }
}

// ---- PSNR ----
constexpr int kPsnrThreads = 256;
constexpr int kPsnrBlocks = 64;  // partial sums per image

__global__ void __launch_bounds__(kPsnrThreads) k_psnr_partial(const float *__restrict__ img,
                                                              const float *__restrict__ gt, int64_t N,
                                                              float *__restrict__ part) {
    __shared__ float red[kPsnrThreads / 32];
    const int s = blockIdx.y;
    const float *x = img + s * N, *y = gt + s * N;
    float acc = 0.f;
    for (int64_t k = (int64_t)blockIdx.x * kPsnrThreads + threadIdx.x; k < N; k += (int64_t)kPsnrBlocks * kPsnrThreads) {
        float v = fminf(fmaxf(__ldg(x + k), 0.f), 1.f) - __ldg(y + k);
        acc += v * v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float a = 0.f;
        for (int w = 0; w < kPsnrThreads / 32; ++w) a += red[w];
        part[(int64_t)s * kPsnrBlocks + blockIdx.x] = a;
    }
}

__global__ void k_psnr_final(const float *__restrict__ part, int64_t N, float *__restrict__ psnr) {
    const int s = blockIdx.x;
    if (threadIdx.x != 0) return;
    double se = 0.0;
    for (int b = 0; b < kPsnrBlocks; ++b) se += (double)part[(int64_t)s * kPsnrBlocks + b];
    double mse = se / (double)N;
    if (mse < 1e-10) mse = 1e-10;
    psnr[s] = (float)(10.0 * log10(1.0 / mse));
}

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

struct LossGrid {
    dim3 grid;
    int nparts;
};

inline LossGrid loss_grid(int H, int W) {
    LossGrid g;
    g.grid = dim3((unsigned)((W + kT - 1) / kT), (unsigned)((H + kT - 1) / kT), 3);
    g.nparts = (int)(g.grid.x * g.grid.y * g.grid.z);
    return g;
}

Win make_window() {
    Win w;
    double g[11], s = 0.0;
    for (int i = 0; i < 11; ++i) {
        g[i] = exp(-(double)((i - 5) * (i - 5)) / (2.0 * 1.5 * 1.5));
        s += g[i];
    }
    for (int i = 0; i < 11; ++i) w.w[i] = (float)(g[i] / s);
    return w;
}

}  // namespace

uint32_t take_loss_flags() {
    uint32_t f = 0, z = 0;
    cudaMemcpyFromSymbol(&f, g_loss_flags, sizeof(f));
    cudaMemcpyToSymbol(g_loss_flags, &z, sizeof(z));
    return f;
}

}  // namespace gs

using namespace gs;

extern "C" size_t gs_loss_workspace_bytes(int32_t H, int32_t W) {
    if (H <= 0 || W <= 0) return 0;
    size_t maps = 3 * (size_t)3 * H * W * sizeof(float);
    return align256(maps) + align256(sizeof(float2) * (size_t)loss_grid(H, W).nparts) + 256;
}

namespace gs {
int loss_ordering(const float *image, const float *gt, int32_t H, int32_t W, float lambda, void *ws, size_t ws_bytes,
                  float *loss_dev, float *dl_dimage, int tiles, const SortFront &front, gs_stream_t stream) {
    if (H <= 0 || W <= 0 || H > 16384 || W > 16384 || !(lambda >= 0.f && lambda <= 1.f)) return GS_ERR_INVALID_ARG;
    if (!image || !gt || !ws || !loss_dev || !dl_dimage) return GS_ERR_INVALID_ARG;
    if (ws_bytes < gs_loss_workspace_bytes(H, W) || (reinterpret_cast<uintptr_t>(ws) & 255)) return GS_ERR_INVALID_ARG;
    cudaStream_t s = as_stream(stream);
    const int64_t HW = (int64_t)H * W;
    f32x2 *mapAB = static_cast<f32x2 *>(ws);
    float *mapC = reinterpret_cast<float *>(mapAB + 3 * HW);
    float2 *part = reinterpret_cast<float2 *>(static_cast<char *>(ws) + align256(9 * (size_t)HW * sizeof(float)));
    LossGrid g = loss_grid(H, W);
    Win win = make_window();
    // 256 tiles of 64 pixels or more and 3 x 1024 pixels a block: there are enough of them
    const DepthOrder deep{tiles, front.depth, front.order_deep, front.hist, front.next};
    launch_chained(k_ssim_fwd, g.grid, kLossThreads, s, image, gt, H, W, win, mapAB, mapC, part, deep);
    launch_chained(k_ssim_bwd, g.grid, kLossThreads, s, image, gt, H, W, win, lambda, mapAB, mapC, part, loss_dev,
                   dl_dimage, deep);
    note_launches(2);
    return launch_status();
}
}  // namespace gs

extern "C" int gs_loss(const float *image, const float *gt, int32_t H, int32_t W, float lambda, void *ws,
                       size_t ws_bytes, float *loss_dev, float *dl_dimage, gs_stream_t stream) {
    return loss_ordering(image, gt, H, W, lambda, ws, ws_bytes, loss_dev, dl_dimage, 0, SortFront{}, stream);
}

extern "C" size_t gs_psnr_workspace_bytes(int32_t S, int32_t H, int32_t W) {
    (void)H; (void)W;
    if (S <= 0) return 0;
    return align256(sizeof(float) * (size_t)S * kPsnrBlocks);
}

extern "C" int gs_psnr(const float *images, const float *gts, int32_t S, int32_t H, int32_t W, void *ws,
                       size_t ws_bytes, float *psnr_dev, gs_stream_t stream) {
    if (S < 0 || H <= 0 || W <= 0) return GS_ERR_INVALID_ARG;
    if (S == 0) return GS_OK;
    if (!images || !gts || !ws || !psnr_dev || ws_bytes < gs_psnr_workspace_bytes(S, H, W)) return GS_ERR_INVALID_ARG;
    cudaStream_t s = as_stream(stream);
    const int64_t N = 3 * (int64_t)H * W;
    float *part = static_cast<float *>(ws);
    k_psnr_partial<<<dim3(kPsnrBlocks, (unsigned)S), kPsnrThreads, 0, s>>>(images, gts, N, part);
    k_psnr_final<<<(unsigned)S, 32, 0, s>>>(part, N, psnr_dev);
    note_launches(2);
    return launch_status();
}
