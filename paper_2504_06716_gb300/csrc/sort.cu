// Per-tile depth order of splats (Sec. 3.1: colours are blended "in a sorted
// order").
//
// The result equals a stable sort of the 64-bit keys (tile << 32 | depth
// bits) generated in Gaussian order, but no (Gaussian, tile) entry is ever
// sorted:
//   1. compact the visible Gaussians (ascending index) and LSD-radix-sort
//      them by the bits of their float32 depth above the view's smallest (3
//      passes of 9 bits, or 4 of 8 where the depths span more, over the
//      visible Gaussians only, one launch each; stable, so equal depths keep
//      index order);
//   2. in that depth order, emit one entry per super-tile (8 x 8 tiles) a
//      Gaussian's tile rectangle meets -- about one per Gaussian -- and
//      stable-sort those few entries by super-tile id (1-2 radix passes);
//   3. split each super-tile's depth-ordered list into chunks of 256; per
//      chunk, every entry's 64-bit mask of the tiles that list it (see the
//      tile membership rule below) and one warp ballot
//      per tile give the entry's rank among the chunk's entries of that tile;
//      a scan over the chunks of a super-tile and one over the tile counts
//      give every tile's start (the ranges) and every entry's final place,
//      written once: in depth order, then index order, inside each tile.
// All counts live on the device; nothing waits on the host.
#include "common.cuh"

namespace gs {

__device__ uint32_t g_sort_flags;

namespace {

constexpr int kMaxRadixBits = 9;                       // digits of up to 9 bits (512 buckets) per pass
constexpr int kMaxRadix = 1 << kMaxRadixBits;
constexpr int kScanBlock = 1024;                       // elements per scan block

// Contiguous chunks of a device-side count that the blocks of a pass own, one
// per SM of the chip, none under kMinChunk (then the last blocks have none).
constexpr int kSortGrid = 152;
constexpr int kMinChunk = 2048;

__host__ __device__ inline uint32_t chunk_len(uint32_t n) {
    const uint32_t c = (n + kSortGrid - 1) / kSortGrid;
    return c <= (uint32_t)kMinChunk ? (uint32_t)kMinChunk : (c + 255u) & ~255u;
}

// Rows of a pass's histogram that a count of at most n can use.
inline int64_t chunk_rows(int64_t n) {
    const int64_t r = (n + kMinChunk - 1) / kMinChunk;
    return r < 1 ? 1 : (r < kSortGrid ? r : kSortGrid);
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

template <typename T>
__device__ __forceinline__ T block_scan_excl(T v, T *warp_sums, T *total) {
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nwarps ? warp_sums[lane] : T(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;
    }
    __syncthreads();
    T before = warp > 0 ? warp_sums[warp - 1] : T(0);
    *total = warp_sums[nwarps - 1];
    __syncthreads();
    return before + x - v;
}

__device__ __forceinline__ bool splat_visible(const float *splats, int64_t i) {
    return __float_as_int(__ldg(splats + i * kSplat + 11)) > 0;
}

// Sum of this block's kScanBlock values of v, and the sum before element i of
// part[0 .. nb) with the whole (every thread gets all).
template <typename T>
struct PartSum {
    T before, total;
};

template <typename T>
__device__ __forceinline__ PartSum<T> part_sum(const T *__restrict__ part, int nb, int i, T *warp_sums) {
    T b = 0, t = 0;
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const T v = part[j];
        t += v;
        b += j < i ? v : T(0);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        b += __shfl_xor_sync(kFull, b, o);
        t += __shfl_xor_sync(kFull, t, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) {
        warp_sums[warp] = b;
        warp_sums[32 + warp] = t;
    }
    __syncthreads();
    PartSum<T> r{T(0), T(0)};
    for (int w = 0; w < nw; ++w) {
        r.before += warp_sums[w];
        r.total += warp_sums[32 + w];
    }
    __syncthreads();
    return r;
}

// ---- stage 1a: compaction of visible Gaussians ----
// Five small blocks per SM, each over one contiguous range of the Gaussians, so
// that the next kernel's blocks can sum the counts in front of their own range
// and no scan runs between the two. Five fit at the emitting kernels' 48
// registers: one wave, each block with the same share (eight per SM, in a second
// wave of a few: the emitting kernels 25.5 + 27.8 us against 24.5 + 21.3 at 1M
// Gaussians, 12.9 + 12.1 against 10.9 + 10.8 at 250K).
constexpr int kVisBlock = 256;
constexpr int kVisGrid = 5 * kSortGrid;

__host__ __device__ inline int64_t vis_range(int64_t n) {
    const int64_t r = (n + kVisGrid - 1) / kVisGrid;
    return (r + kVisBlock - 1) / kVisBlock * kVisBlock;
}

// What the visible Gaussians' depths span: the depth keys are float32 bits
// less the smallest, so that views whose depths lie within a factor of about
// 16 sort on at most 27 bits, three passes of 9 instead of four of 8.
struct DepthSpan {
    uint32_t lowest, bits;
};

// The digit of launch k (of 4) of the depth sort; bits 0: the launch does
// nothing. With three passes it is the first launch that is left out, so that
// the order ends in the same buffer.
__host__ __device__ inline int depth_first(uint32_t bits) { return bits <= 27 ? 1 : 0; }

inline unsigned vis_blocks(int64_t n) { return (unsigned)((n + vis_range(n) - 1) / vis_range(n)); }

// The same for a count known on the device only, at most n: as many blocks as
// any such count may use.
inline unsigned entry_blocks(int64_t n) {
    const int64_t b = (n + kVisBlock - 1) / kVisBlock;
    return (unsigned)(b < kVisGrid ? b : kVisGrid);
}

// What the first kernel zeroes for the rest of the sort.
struct ZeroSpans {
    uint32_t *p[3];
    int64_t n[3];
};

// Per block: its visible Gaussians, and the least and largest depth bits
// among them (part [3][kVisGrid]).
__global__ void __launch_bounds__(kVisBlock) k_count_visible(const float *__restrict__ splats, int64_t n,
                                                            uint32_t *__restrict__ part, ZeroSpans z,
                                                            unsigned long long *__restrict__ total_exact,
                                                            uint2 *__restrict__ stamp) {
    __shared__ uint32_t s_c[kVisBlock / 32], s_lo[kVisBlock / 32], s_hi[kVisBlock / 32];
    wait_prior_grid();
    const int64_t range = vis_range(n), lo = (int64_t)blockIdx.x * range, hi = lo + range < n ? lo + range : n;
    const int64_t t = (int64_t)blockIdx.x * kVisBlock + threadIdx.x, all = (int64_t)gridDim.x * kVisBlock;
#pragma unroll
    for (int k = 0; k < 3; ++k)
        for (int64_t i = t; i < z.n[k]; i += all) z.p[k][i] = 0u;
    if (t == 0) {
        *total_exact = 0ull;
        *stamp = make_uint2(0u, 0u);  // an earlier sort's tile order is good no more; order_tiles marks this one's
    }
    uint32_t c = 0u, kl = 0xffffffffu, kh = 0u;
#pragma unroll 4
    for (int64_t i = lo + threadIdx.x; i < hi; i += kVisBlock) {
        const uint32_t key = __float_as_uint(__ldg(splats + i * kSplat + 9));
        if (splat_visible(splats, i)) {
            ++c;
            kl = min(kl, key);
            kh = max(kh, key);
        }
    }
    c = __reduce_add_sync(kFull, c);
    kl = __reduce_min_sync(kFull, kl);
    kh = __reduce_max_sync(kFull, kh);
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { s_c[warp] = c; s_lo[warp] = kl; s_hi[warp] = kh; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kVisBlock / 32; ++w) {
            c += s_c[w];
            kl = min(kl, s_lo[w]);
            kh = max(kh, s_hi[w]);
        }
        part[blockIdx.x] = c;
        part[kVisGrid + blockIdx.x] = kl;
        part[2 * kVisGrid + blockIdx.x] = kh;
    }
}

// ---- LSD radix pass, one launch ----
// The number of keys lives on the device; block b owns the keys of chunk b
// (chunk_len). hist [kSortGrid][kMaxRadix] holds every chunk's digit counts:
// they were added up by whoever wrote the keys (the kernel before the first
// pass, or the pass before), key by key with atomics that nobody waits for, at
// the chunk each key went to. So a pass needs no histogram and no scan launch
// of its own: a block sums the rows of the chunks in front of its own (at most
// 152 x 256 words, read by all 1024 threads) for where its digits begin.
//
// Inside the block every warp owns a contiguous piece of the chunk: it counts
// its digits in a row of its own, one scan over the warps per digit turns the
// rows into positions, and the warp then goes through its keys in order,
// ranking each 32 with a match. The keys of a piece (up to 256 at a time) are
// loaded together before anything waits. Two block barriers in all, whatever
// the chunk's length; the order is stable.
//
// Bound by L2: the rows of counts (156 KB per block on 8 bits), the scattered
// 8-byte words and the atomics (about 2.5 cycles per SM each). The three
// launches it replaces (histograms, a scan per digit, a scatter of 1024 keys
// per block with four barriers per 256) took 20 us a pass and four passes at
// 551K keys; this takes 13 to 16 us and three passes (five passes with the
// super-tiles' one: 102 -> 68 us). Putting a chunk in order in shared memory
// first, to write runs, made it 72 us.
constexpr int kRadixThreads = 1024;
constexpr int kRadixWarps = kRadixThreads / 32;

// Where a one-pass sort by super-tile id leaves each super-tile's entries:
// its digit's range of the output. Given (chunk_base non-null), block 0 of
// the pass writes the chunk plan from the digit totals: chunk_base [ns + 1]
// (exclusive scan of ceil(len / chunk)) and chunk_rec (per chunk: its
// super-tile, first entry, the segment's end and the super-tile's first
// chunk).
struct SegPlan {
    uint32_t *chunk_base;
    uint4 *chunk_rec;
    int ns, chunk;
};

// The digit a pass sorts by, and its histogram rows.
struct Digit {
    uint32_t *hist;
    int shift, bits;
};

// The digit of launch k of the depth sort, from the span of the keys (bits 0:
// nothing to do). hist: row blocks of the four launches, `stride` words apart.
__device__ __forceinline__ Digit depth_digit(uint32_t *hist, size_t stride, uint32_t bits, int k) {
    const int first = depth_first(bits), passes = 4 - first;
    if (k < first || k > 3) return Digit{nullptr, 0, 0};
    const int per = max(1, ((int)bits + passes - 1) / passes);
    return Digit{hist + (size_t)k * stride, (k - first) * per, per};
}

// A key that goes to `pos` of n, counted for the pass that sorts by d next.
__device__ __forceinline__ void count_next(const Digit &d, uint32_t key, uint32_t pos, uint32_t chunk) {
    const uint32_t v = (key >> d.shift) & ((1u << d.bits) - 1u);
    atomicAdd(d.hist + (size_t)(pos / chunk) * kMaxRadix + v, 1u);
}

// With span given, launch k of the depth sort (cur.hist the histograms of all
// four, next unused, stride their distance); else the digits cur and next.
//
// A key and its value travel as one 8-byte word (one scattered store instead
// of two); the last pass writes the values (vout) and, if asked, the keys
// (kout) by themselves instead.
__global__ void __launch_bounds__(kRadixThreads) k_radix_pass(const uint2 *__restrict__ in, uint2 *__restrict__ out,
                                                              uint32_t *__restrict__ kout, uint32_t *__restrict__ vout,
                                                              const uint32_t *__restrict__ count, Digit cur, Digit next,
                                                              const DepthSpan *__restrict__ span, int k, size_t stride,
                                                              SegPlan sp) {
    extern __shared__ uint32_t s_cnt[];  // [warps][radix]
    __shared__ uint4 s_sum[2][kRadixThreads];  // [row group][four digits]
    __shared__ uint32_t ws[32];
    constexpr int kRounds = 8;
    wait_prior_grid();
    const uint32_t n = *count, len = chunk_len(n);
    const uint32_t lo = (uint32_t)blockIdx.x * len;  // below 2^32: 152 chunks hold at most 2^31 + 152 * 256
    if (span) {
        uint32_t *hist = cur.hist;
        const uint32_t bits = span->bits;
        cur = depth_digit(hist, stride, bits, k);
        next = depth_digit(hist, stride, bits, k + 1);
        if (!cur.hist) return;
    }
    const bool plan = sp.chunk_base && blockIdx.x == 0;
    if (lo >= n && !plan) return;
    const int radix = 1 << cur.bits, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint32_t mask = (uint32_t)radix - 1u;
    const uint32_t piece = len / kRadixWarps;
    const uint32_t b0 = lo + warp * piece, b1 = lo < n ? min(n, b0 + piece) : b0;
    uint2 kv[kRounds];
    auto load = [&](uint32_t i0) {
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            const uint32_t i = i0 + 32 * r + lane;
            kv[r] = i < b1 ? in[i] : make_uint2(0u, 0u);
        }
    };
    load(b0);
    for (int e = t; e < kRadixWarps * radix; e += kRadixThreads) s_cnt[e] = 0u;
    // rows in front of this chunk's, and all rows, four digits per thread and
    // every load in flight (a row's words past the radix are zero)
    const int used = (int)((n + len - 1) / len), quads = max(1, radix / 4), parts = kRadixThreads / quads;
    uint4 below4 = make_uint4(0u, 0u, 0u, 0u), total4 = below4;
    {
        const uint4 *h4 = reinterpret_cast<const uint4 *>(cur.hist) + (t & (quads - 1));
#pragma unroll 20
        for (int r = t / quads; r < used; r += parts) {
            const uint4 v = h4[(size_t)r * (kMaxRadix / 4)];
            total4.x += v.x; total4.y += v.y; total4.z += v.z; total4.w += v.w;
            if (r < (int)blockIdx.x) { below4.x += v.x; below4.y += v.y; below4.z += v.z; below4.w += v.w; }
        }
    }
    s_sum[0][t] = below4;
    s_sum[1][t] = total4;
    __syncthreads();
    uint32_t *row = s_cnt + warp * radix;
    for (uint32_t i0 = b0; i0 < b1; i0 += 32 * kRounds) {  // this warp's piece, counted
        if (i0 != b0) load(i0);
#pragma unroll
        for (int r = 0; r < kRounds; ++r)
            if (i0 + 32 * r + lane < b1) atomicAdd(row + ((kv[r].x >> cur.shift) & mask), 1u);
    }
    // per digit (threads below radix): totals, their exclusive scan, this chunk's start
    uint32_t below = 0u, total = 0u;
    if (t < radix) {
        const uint32_t *sb = reinterpret_cast<const uint32_t *>(s_sum[0]), *st = reinterpret_cast<const uint32_t *>(s_sum[1]);
#pragma unroll 8
        for (int q = 0; q < parts; ++q) {
            below += sb[t + q * 4 * quads];
            total += st[t + q * 4 * quads];
        }
    }
    uint32_t all;
    const uint32_t dbase = block_scan_excl<uint32_t>(total, ws, &all);  // its barriers also order the counts
    if (plan) {
        const uint32_t nc = t < sp.ns ? (total + (uint32_t)sp.chunk - 1u) / (uint32_t)sp.chunk : 0u;
        uint32_t nctot;
        const uint32_t cb = block_scan_excl<uint32_t>(nc, ws, &nctot);
        if (t < sp.ns) {
            sp.chunk_base[t] = cb;
            for (uint32_t c = 0; c < nc; ++c)
                sp.chunk_rec[cb + c] =
                    make_uint4((uint32_t)t, dbase + c * (uint32_t)sp.chunk, dbase + total, cb);
        }
        if (t == 0) sp.chunk_base[sp.ns] = nctot;
        if (lo >= n) return;
    }
    if (t < radix) {
        uint32_t c = dbase + below;
#pragma unroll 8
        for (int w = 0; w < kRadixWarps; ++w) {
            const uint32_t x = s_cnt[w * radix + t];
            s_cnt[w * radix + t] = c;
            c += x;
        }
    }
    __syncthreads();
    const unsigned lt = lanemask_lt();
    const bool held = piece <= 32 * kRounds;  // the registers still hold the whole piece
    for (uint32_t i0 = b0; i0 < b1; i0 += 32 * kRounds) {
        if (!held) load(i0);
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            if (i0 + 32 * r >= b1) break;  // uniform
            const bool valid = i0 + 32 * r + lane < b1;
            const uint32_t key = kv[r].x;
            const uint32_t d = valid ? (key >> cur.shift) & mask : 0xffffu;
            const unsigned peers = __match_any_sync(kFull, d);
            uint32_t pos = 0u;
            if (valid) pos = row[d] + __popc(peers & lt);
            __syncwarp();
            if (valid && !(peers & lt)) row[d] += (uint32_t)__popc(peers);
            __syncwarp();
            if (valid) {
                if (vout) {
                    if (kout) kout[pos] = key;
                    vout[pos] = kv[r].y;
                } else {
                    out[pos] = kv[r];
                    count_next(next, key, pos, len);
                }
            }
        }
    }
}

// All passes of the depth sort in one launch, by one block, for at most
// kSmallSort Gaussians: every pass is bound by launch latency there (10 chunks or
// fewer), and the keys fit in shared memory. Digits of up to 8 bits; every warp
// holds its piece in registers while the pass writes the keys' new places, so
// one buffer is enough. The whole sort at 600x400, against the passes of many
// blocks: 1000 Gaussians 35 us against 44, 4000 42 against 51, 6000 47 against 52,
// 8192 even; more do not fit the registers of a block.
constexpr int kSmallSort = 8192;
constexpr int kSmallBits = 8, kSmallRadix = 1 << kSmallBits;
constexpr size_t kSmallShared = kSmallSort * sizeof(uint2) + kRadixWarps * kSmallRadix * sizeof(uint32_t);

__global__ void __launch_bounds__(kRadixThreads) k_depth_small(const uint2 *kv0, const uint2 *kv1, uint32_t *order,
                                                               const uint32_t *__restrict__ count,
                                                               const DepthSpan *__restrict__ span) {
    extern __shared__ __align__(16) uint2 s_kv[];
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_kv + kSmallSort);  // [warps][radix]
    __shared__ uint32_t s_base[kSmallRadix];
    __shared__ uint32_t ws[32];
    constexpr int kRounds = kSmallSort / kRadixThreads;
    wait_prior_grid();
    const uint32_t n = *count;
    const int bits = (int)span->bits, passes = (bits + kSmallBits - 1) / kSmallBits;
    const int per = passes ? (bits + passes - 1) / passes : 0;
    const uint32_t mask = (1u << per) - 1u;
    const uint2 *in = depth_first((uint32_t)bits) ? kv1 : kv0;  // where k_emit_visible left them
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint32_t piece = (n + kRadixThreads - 1) / kRadixThreads * 32;
    const uint32_t b0 = warp * piece, b1 = min(n, b0 + piece);
    uint32_t *row = s_cnt + warp * kSmallRadix;
    const unsigned lt = lanemask_lt();
    uint2 kv[kRounds];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const uint32_t i = b0 + 32 * r + lane;
        kv[r] = i < b1 ? in[i] : make_uint2(0u, 0u);
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = p * per;
        if (p) {
#pragma unroll
            for (int r = 0; r < kRounds; ++r)
                if (b0 + 32 * r + lane < b1) kv[r] = s_kv[b0 + 32 * r + lane];
        }
        for (int e = t; e < kRadixWarps * kSmallRadix; e += kRadixThreads) s_cnt[e] = 0u;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRounds; ++r)
            if (b0 + 32 * r + lane < b1) atomicAdd(row + ((kv[r].x >> shift) & mask), 1u);
        __syncthreads();
        uint32_t total = 0u, all;
        if (t < kSmallRadix) {
#pragma unroll 8
            for (int w = 0; w < kRadixWarps; ++w) {
                const uint32_t x = s_cnt[w * kSmallRadix + t];
                s_cnt[w * kSmallRadix + t] = total;
                total += x;
            }
        }
        const uint32_t base = block_scan_excl<uint32_t>(total, ws, &all);
        if (t < kSmallRadix) s_base[t] = base;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            if (b0 + 32 * r >= b1) break;  // uniform
            const bool valid = b0 + 32 * r + lane < b1;
            const uint32_t d = valid ? (kv[r].x >> shift) & mask : 0xffffu;
            const unsigned peers = __match_any_sync(kFull, d);
            uint32_t pos = 0u;
            if (valid) pos = s_base[d] + row[d] + __popc(peers & lt);
            __syncwarp();
            if (valid && !(peers & lt)) row[d] += (uint32_t)__popc(peers);
            __syncwarp();
            if (valid) s_kv[pos] = kv[r];
        }
        __syncthreads();
    }
    __syncthreads();  // the input, whose place `order` shares, has been read
    if (passes) {
        for (uint32_t i = t; i < n; i += kRadixThreads) order[i] = s_kv[i].y;
    } else {  // equal depths: by index, as they come
#pragma unroll
        for (int r = 0; r < kRounds; ++r)
            if (b0 + 32 * r + lane < b1) order[b0 + 32 * r + lane] = kv[r].y;
    }
}

// Blocks of 256 threads the device holds at once (grids of the loops above).
int64_t resident_blocks() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (int64_t)(sms > 0 ? sms : 152) * 8;
}

__global__ void k_zero_u32(uint32_t *__restrict__ p, int64_t n) {
    wait_prior_grid();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = 0u;
}

// ---- stage 2: super-tile entries in depth order ----
constexpr int kSuper = 8;       // a super-tile is kSuper x kSuper tiles (64 = one bit each)
constexpr int kChunk = 256;     // super-tile list entries per chunk (one per thread)

__device__ __forceinline__ int splat_rect(const float *splats, uint32_t g, const DevCam &cam, int &x0, int &y0,
                                          int &x1, int &y1) {
    const float *r = splats + (int64_t)g * kSplat;
    int rad = __float_as_int(__ldg(r + 10));
    if (rad <= 0) { x0 = y0 = x1 = y1 = 0; return 0; }
    return tile_rect(__ldg(r), __ldg(r + 1), rad, cam.tile, cam.tiles_x, cam.tiles_y, x0, y0, x1, y1);
}

__device__ __forceinline__ int super_rect(int x0, int y0, int x1, int y1, int &sx0, int &sy0, int &sx1, int &sy1) {
    sx0 = x0 / kSuper; sy0 = y0 / kSuper;
    sx1 = (x1 - 1) / kSuper + 1; sy1 = (y1 - 1) / kSuper + 1;
    return (sx1 - sx0) * (sy1 - sy0);
}

// ---- tile membership ----
// A tile of a splat's 3-sigma rectangle lists the splat only if the box of its
// pixel centres [X, X + T - 1] x [Y, Y + T - 1] holds a point where the
// conic's quadratic form q = a dx^2 + 2 b dx dy + c dy^2 is at most
// tau + 1e-3 (1 + tau), tau = 2 ln(255 o): elsewhere alpha = o exp(-q/2) is
// below the 1/255 floor of Eq. 2 at every pixel of the tile, so leaving the
// splat out changes no image and no gradient. A splat with 255 o < 1 is
// listed nowhere. Decided in single precision, every operation rounded
// (explicit intrinsics, no contraction); the 1e-3 relative margin makes the
// lists a superset of the tiles that hold a pixel centre with alpha >= 1/255
// exactly, so float32 rounding never drops a contribution.

// ln x for x >= 1: x = m 2^e, m in [1, 2); ln m = 2 atanh(s), s = (m-1)/(m+1),
// by the series 2 s (1 + s^2/3 + ... + s^14/15).
__device__ __forceinline__ float ln_f32(float x) {
    const uint32_t b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xffu) - 127;
    const float m = __uint_as_float((b & 0x007fffffu) | 0x3f800000u);
    const float s = __fdiv_rn(__fsub_rn(m, 1.f), __fadd_rn(m, 1.f));
    const float s2 = __fmul_rn(s, s);
    float p = 0.0666666667f;
    p = __fadd_rn(__fmul_rn(p, s2), 0.0769230769f);
    p = __fadd_rn(__fmul_rn(p, s2), 0.0909090909f);
    p = __fadd_rn(__fmul_rn(p, s2), 0.111111111f);
    p = __fadd_rn(__fmul_rn(p, s2), 0.142857143f);
    p = __fadd_rn(__fmul_rn(p, s2), 0.2f);
    p = __fadd_rn(__fmul_rn(p, s2), 0.333333333f);
    p = __fadd_rn(__fmul_rn(p, s2), 1.f);
    return __fadd_rn(__fmul_rn((float)e, 0.693147181f), __fmul_rn(__fmul_rn(2.f, s), p));
}

// The bound on q with its margin; negative when the splat is listed nowhere.
__device__ __forceinline__ float tile_tau(float opacity) {
    const float x = __fmul_rn(255.f, opacity);
    if (!(x >= 1.f)) return -1.f;
    const float tau = __fmul_rn(2.f, ln_f32(x));
    return __fadd_rn(tau, __fmul_rn(1e-3f, __fadd_rn(1.f, tau)));
}

__device__ __forceinline__ float quad_f32(float a, float b, float c, float dx, float dy) {
    return __fadd_rn(__fadd_rn(__fmul_rn(__fmul_rn(a, dx), dx), __fmul_rn(__fmul_rn(__fmul_rn(2.f, b), dx), dy)),
                     __fmul_rn(__fmul_rn(c, dy), dy));
}

struct SplatShape {
    float mx, my, a, b, c, tau, bc, ba;  // bc = b / c, ba = b / a
};

__device__ __forceinline__ SplatShape splat_shape(const float *splats, uint32_t g) {
    const float4 *r = reinterpret_cast<const float4 *>(splats + (int64_t)g * kSplat);
    const float4 p0 = __ldg(r), p1 = __ldg(r + 1);
    SplatShape sh;
    sh.mx = p0.x; sh.my = p0.y; sh.a = p0.z; sh.b = p0.w; sh.c = p1.x;
    sh.tau = tile_tau(p1.y);
    sh.bc = __fdiv_rn(sh.b, sh.c);
    sh.ba = __fdiv_rn(sh.b, sh.a);
    return sh;
}

// Whether tile (x, y) lists the splat: the box minimum of q is 0 when the mean
// lies inside, else the least of the four edges' clamped one-dimensional
// minima (on x = X at y = my - (b/c)(X - mx), on y = Y at x = mx - (b/a)(Y - my)).
__device__ __forceinline__ bool tile_hit(const SplatShape &sh, int tile, int x, int y) {
    if (sh.tau < 0.f) return false;
    const float x0 = (float)(x * tile), x1 = (float)(x * tile + tile - 1);
    const float y0 = (float)(y * tile), y1 = (float)(y * tile + tile - 1);
    if (sh.mx >= x0 && sh.mx <= x1 && sh.my >= y0 && sh.my <= y1) return true;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float ex = k ? x1 : x0, ey = k ? y1 : y0;
        const float dx = __fsub_rn(ex, sh.mx);
        const float yo = __fsub_rn(sh.my, __fmul_rn(sh.bc, dx));
        const float yy = yo < y0 ? y0 : (yo > y1 ? y1 : yo);
        if (quad_f32(sh.a, sh.b, sh.c, dx, __fsub_rn(yy, sh.my)) <= sh.tau) return true;
        const float dy = __fsub_rn(ey, sh.my);
        const float xo = __fsub_rn(sh.mx, __fmul_rn(sh.ba, dy));
        const float xx = xo < x0 ? x0 : (xo > x1 ? x1 : xo);
        if (quad_f32(sh.a, sh.b, sh.c, __fsub_rn(xx, sh.mx), dy) <= sh.tau) return true;
    }
    return false;
}

// tile_hit by the edges that face the mean alone: for a mean outside the box the
// least q over the box lies on one of them, so the other edges can pass only
// where rounding decides. `none` is a bound above tau beyond which it cannot:
// 1.01 tau for kappa <= 1e4 (as in cand_rect: q is off by at most 0.24%, the
// clamped minimiser's own rounding by less), infinite for worse conics; q
// between tau and `none` goes through all four edges. The same decision as
// tile_hit, in two evaluations of q instead of four.
__device__ __forceinline__ bool tile_hit_facing(const SplatShape &sh, float none, int tile, int x, int y) {
    const float x0 = (float)(x * tile), x1 = (float)(x * tile + tile - 1);
    const float y0 = (float)(y * tile), y1 = (float)(y * tile + tile - 1);
    const bool out_x = !(sh.mx >= x0 && sh.mx <= x1), out_y = !(sh.my >= y0 && sh.my <= y1);
    if (sh.tau < 0.f) return false;
    if (!out_x && !out_y) return true;
    const float dx = __fsub_rn(sh.mx > x1 ? x1 : x0, sh.mx);
    const float yo = __fsub_rn(sh.my, __fmul_rn(sh.bc, dx));
    const float yy = yo < y0 ? y0 : (yo > y1 ? y1 : yo);
    const float q1 = quad_f32(sh.a, sh.b, sh.c, dx, __fsub_rn(yy, sh.my));
    const float dy = __fsub_rn(sh.my > y1 ? y1 : y0, sh.my);
    const float xo = __fsub_rn(sh.mx, __fmul_rn(sh.ba, dy));
    const float xx = xo < x0 ? x0 : (xo > x1 ? x1 : xo);
    const float q2 = quad_f32(sh.a, sh.b, sh.c, __fsub_rn(xx, sh.mx), dy);
    // a non-facing edge's q is one of the four as well: a pass is a pass
    if (q1 <= sh.tau || q2 <= sh.tau) return true;
    const float q = out_x ? (out_y ? fminf(q1, q2) : q1) : q2;
    if (q > none) return false;
    return tile_hit(sh, tile, x, y);
}

// The tiles a splat may be listed in: its 3-sigma rectangle, narrowed to the
// bounding box of the ellipse q <= tau when that box is provably wide
// enough. tile_hit evaluates q = a dx^2 + 2 b dx dy + c dy^2 (float32) only
// at points of a tile's pixel-centre box, and min over dy of q is
// dx^2 det / c (det = a c - b^2), so q > tau wherever |dx| >= sqrt(tau c /
// det). The rounding error of q is at most 4 u kappa q (u = 2^-24) with
// kappa = (a + |b| + c)(a + c) / det >= (|a| dx^2 + 2 |b dx dy| + c dy^2) / q,
// and det carries a relative error of about 2 u kappa; for kappa <= 1e4 both
// stay below 0.3%, well inside the 4% that the factor 1.02 on the box's half
// widths leaves (plus a pixel). Ill-conditioned conics keep the rectangle.
// So every tile dropped here fails tile_hit: the lists are unchanged. `cull`,
// when given, takes the bound of tile_hit_facing and the constants of row_span.
struct CullExtra {
    float none;     // bound of tile_hit_facing (infinite: none)
    float det, hx;  // row_span: determinant of the conic, half width of the ellipse (0: not for row_span)
};

__device__ __forceinline__ int cand_rect(const float *splats, uint32_t g, const DevCam &cam, float tau, int &x0,
                                         int &y0, int &x1, int &y1, CullExtra *cull = nullptr) {
    if (cull) *cull = CullExtra{__int_as_float(0x7f800000), 0.f, 0.f};  // no bounds for ill-conditioned conics
    if (!splat_rect(splats, g, cam, x0, y0, x1, y1)) return 0;
    const float *r = splats + (int64_t)g * kSplat;
    const float mx = __ldg(r), my = __ldg(r + 1), a = __ldg(r + 2), b = __ldg(r + 3), c = __ldg(r + 4);
    const float det = a * c - b * b;
    if (!(tau >= 0.f) || !(det > 0.f) || !(a > 0.f) || !(c > 0.f)) return 1;
    const float kappa = (a + fabsf(b) + c) * (a + c) / det;
    if (!(kappa <= 1e4f)) return 1;
    const float hx0 = sqrtf(tau * c / det), hx = hx0 * 1.02f + 1.f;
    if (cull) {
        cull->none = 1.01f * tau;
        if (kappa <= 1e3f && a <= 4.f && c <= 4.f && tau <= 1e3f && fabsf(mx) <= 32768.f && fabsf(my) <= 32768.f) {
            cull->det = det;
            cull->hx = hx0;
        }
    }
    const float hy = sqrtf(tau * a / det) * 1.02f + 1.f;
    const float inv = 1.f / (float)cam.tile;  // exact: a power of two
    x0 = max(x0, (int)floorf((mx - hx) * inv));
    x1 = min(x1, (int)floorf((mx + hx) * inv) + 1);
    y0 = max(y0, (int)floorf((my - hy) * inv));
    y1 = min(y1, (int)floorf((my + hy) * inv) + 1);
    if (x0 >= x1 || y0 >= y1) {
        x0 = y0 = x1 = y1 = 0;
        return 0;
    }
    return 1;
}

// The tiles of one row of tiles, pixel rows y0 .. y1, that list a splat, as two
// spans of tile columns counted from pixel column xo: [lo, hi] outside of which
// none does, and [sure_lo, sure_hi] all of which do (either may be empty, hi <
// lo). What lies between them is for tile_hit to decide. The region q <= L inside
// the row is convex, so the columns it reaches are an interval: its right end lies
// at the ellipse's rightmost point, dy = -(b/c) hx, or on the row's edge nearest
// to it, where dx = (-b dy + sqrt(a L - det dy^2)) / a, and so on the left; no real
// root means the row is missed.
//
// For the splats it takes (kappa <= 1000, a, c <= 4: cand_rect) tile_hit's q is off
// by 6 u kappa = 0.036%, its minimiser by half a unit in the last place of the
// position (5e-4 pixels at 16384), worth c (5e-4)^2 = 1e-6, and det here by 2 u
// kappa = 0.012%. The levels tau (1 +- 0.0007) +- 1.5e-6 enclose all of that, and by
// what is left the rounding of the columns in units of the ellipse; 0.002 pixels
// cover it in units of the position.
struct RowSpan {
    int lo, hi, sure_lo, sure_hi;
};

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ RowSpan row_span(const SplatShape &sh, float det, float hx, int tile, int xo, int y) {
    const float y0 = __fsub_rn((float)(y * tile), sh.my), y1 = __fsub_rn((float)(y * tile + tile - 1), sh.my);
    const float dyr = -sh.bc * hx;
    const float dr = fminf(fmaxf(dyr, y0), y1), dl = fminf(fmaxf(-dyr, y0), y1);
    const float at = sh.a * sh.tau, qr = det * dr * dr, ql = det * dl * dl;
    const float hi = fmaf(1.5e-6f, sh.a, 1.0007f * at), lo = fmaf(-1.5e-6f, sh.a, 0.9993f * at);
    const float r_hi = hi - qr, l_hi = hi - ql, r_lo = lo - qr, l_lo = lo - ql;
    if (r_hi < 0.f || l_hi < 0.f) return RowSpan{0, -1, 0, -1};
    const float ia = __fdividef(1.f, sh.a), inv = 1.f / (float)tile;  // exact: a power of two
    const float o = __fsub_rn(sh.mx, (float)xo), left = o - (float)(tile - 1);
    const float cr = -sh.b * dr, cl = -sh.b * dl;
    RowSpan s;
    s.hi = (int)floorf((o + fmaf(cr + sqrt_approx(r_hi), ia, 0.002f)) * inv);
    s.lo = (int)ceilf((left + fmaf(cl - sqrt_approx(l_hi), ia, -0.002f)) * inv);
    s.sure_lo = 0;
    s.sure_hi = -1;
    if (r_lo >= 0.f && l_lo >= 0.f) {
        s.sure_hi = (int)floorf((o + fmaf(cr + sqrt_approx(r_lo), ia, -0.002f)) * inv);
        s.sure_lo = (int)ceilf((left + fmaf(cl - sqrt_approx(l_lo), ia, 0.002f)) * inv);
    }
    return s;
}

// Columns lo .. hi of a row as bits, those inside [x0, x1).
__device__ __forceinline__ uint32_t span_bits(int lo, int hi, int x0, int x1) {
    lo = max(lo, x0);
    hi = min(hi, x1 - 1);
    return hi < lo ? 0u : (2u << hi) - (1u << lo);
}

// The tile tests' constants and the candidate rectangle of a visible
// Gaussian, computed once per sort (k_emit_visible) and read by the
// depth-ordered passes and the chunk kernels: cull[2 g] = (tau, b / c, b / a,
// the bound of tile_hit_facing), cull[2 g + 1] = (x0 | y0 << 16, x1 | y1 << 16, det, hx), the rectangle as
// integers (empty when no tile can list the splat, 255 o < 1), det and hx for row_span.
__device__ __forceinline__ void write_cull(const float *splats, uint32_t g, const DevCam &cam, float4 *cull) {
    const SplatShape sh = splat_shape(splats, g);
    int x0 = 0, y0 = 0, x1 = 0, y1 = 0;
    CullExtra ex{0.f, 0.f, 0.f};
    if (!(sh.tau >= 0.f) || !cand_rect(splats, g, cam, sh.tau, x0, y0, x1, y1, &ex)) x0 = y0 = x1 = y1 = 0;
    cull[2 * (int64_t)g] = make_float4(sh.tau, sh.bc, sh.ba, ex.none);
    reinterpret_cast<uint4 *>(cull)[2 * (int64_t)g + 1] =
        make_uint4((uint32_t)x0 | ((uint32_t)y0 << 16), (uint32_t)x1 | ((uint32_t)y1 << 16), __float_as_uint(ex.det),
                   __float_as_uint(ex.hx));
}

// Tile coordinates are below 2^16 (images of at most 16384 pixels a side).
__device__ __forceinline__ bool unpack_rect(const uint4 &r, int &x0, int &y0, int &x1, int &y1) {
    x0 = (int)(r.x & 0xffffu);
    y0 = (int)(r.x >> 16);
    x1 = (int)(r.y & 0xffffu);
    y1 = (int)(r.y >> 16);
    return x0 < x1 && y0 < y1;
}

__device__ __forceinline__ bool cull_rect(const float4 *cull, uint32_t g, int &x0, int &y0, int &x1, int &y1) {
    return unpack_rect(__ldg(reinterpret_cast<const uint4 *>(cull) + 2 * (int64_t)g + 1), x0, y0, x1, y1);
}

// The items a block takes at once: warp w has consecutive ones, up to four
// rounds of 32 of them (fewer when the block's range is short, so that every
// warp has some), a thread's loads in flight together, and one barrier orders
// the warps.
constexpr int kVisRounds = 4;

__device__ __forceinline__ int vis_rounds(int64_t range) {
    return range >= kVisRounds * kVisBlock ? kVisRounds : (int)((range + kVisBlock - 1) / kVisBlock);
}

// Exclusive sum over the block's warps of v (one value per warp) and the
// block's total; double-buffered by `turn`, one barrier.
__device__ __forceinline__ PartSum<uint32_t> warps_before(uint32_t v, uint32_t (*buf)[kVisBlock / 32], int turn) {
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) buf[turn & 1][warp] = v;
    __syncthreads();
    PartSum<uint32_t> r{0u, 0u};
#pragma unroll
    for (int w = 0; w < kVisBlock / 32; ++w) {
        const uint32_t x = buf[turn & 1][w];
        r.before += w < warp ? x : 0u;
        r.total += x;
    }
    return r;
}

// The depth keys and indices of the visible Gaussians, ascending index, their
// cull records, and the first radix pass's digit counts.
__global__ void __launch_bounds__(kVisBlock, 5) k_emit_visible(const float *__restrict__ splats, int64_t n,
                                                           const uint32_t *__restrict__ part, DevCam cam,
                                                           uint2 *__restrict__ kv0, uint2 *__restrict__ kv1,
                                                           float4 *__restrict__ cull, uint32_t *__restrict__ n_vis,
                                                           DepthSpan *__restrict__ span, uint32_t *__restrict__ hist,
                                                           size_t stride) {
    __shared__ uint32_t ps[64];
    __shared__ uint32_t buf[2][kVisBlock / 32];
    __shared__ uint32_t s_lo, s_hi;
    wait_prior_grid();
    if (threadIdx.x == 0) { s_lo = 0xffffffffu; s_hi = 0u; }
    uint32_t kl = 0xffffffffu, kh = 0u;
    for (int j = threadIdx.x; j < (int)gridDim.x; j += kVisBlock) {
        kl = min(kl, part[kVisGrid + j]);
        kh = max(kh, part[2 * kVisGrid + j]);
    }
    kl = __reduce_min_sync(kFull, kl);
    kh = __reduce_max_sync(kFull, kh);
    const PartSum<uint32_t> sum = part_sum<uint32_t>(part, (int)gridDim.x, (int)blockIdx.x, ps);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&s_lo, kl);
        atomicMax(&s_hi, kh);
    }
    __syncthreads();
    const uint32_t lowest = s_lo, bits = sum.total ? 32u - (uint32_t)__clz(s_hi - lowest) : 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *n_vis = sum.total;
        span->lowest = lowest;
        span->bits = bits;
    }
    const int first = depth_first(bits);
    const Digit dig = depth_digit(hist, stride, bits, first);
    uint2 *kv = first ? kv1 : kv0;
    const uint32_t chunk = chunk_len(sum.total);
    uint32_t at = sum.before;
    const int64_t range = vis_range(n), lo = (int64_t)blockIdx.x * range, hi = lo + range < n ? lo + range : n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    const int rounds = vis_rounds(range);
    int turn = 0;
    for (int64_t base = lo; base < hi; base += (int64_t)rounds * kVisBlock, ++turn) {
        const int64_t i0 = base + warp * 32 * rounds + lane;
        unsigned seen[kVisRounds];
        uint32_t mine = 0u;
#pragma unroll
        for (int r = 0; r < kVisRounds; ++r)
            seen[r] = r < rounds && i0 + 32 * r < hi && splat_visible(splats, i0 + 32 * r);
#pragma unroll
        for (int r = 0; r < kVisRounds; ++r) {
            seen[r] = __ballot_sync(kFull, seen[r] != 0u);
            mine += (uint32_t)__popc(seen[r]);
        }
        const PartSum<uint32_t> w = warps_before(mine, buf, turn);
        uint32_t pos0 = at + w.before;
        at += w.total;
#pragma unroll
        for (int r = 0; r < kVisRounds; ++r) {
            if ((seen[r] >> lane) & 1u) {
                const uint32_t pos = pos0 + (uint32_t)__popc(seen[r] & lt), i = (uint32_t)(i0 + 32 * r);
                const uint32_t key = __float_as_uint(__ldg(splats + (int64_t)i * kSplat + 9)) - lowest;
                kv[pos] = make_uint2(key, i);
                count_next(dig, key, pos, chunk);
                write_cull(splats, i, cam, cull);
            }
            pos0 += (uint32_t)__popc(seen[r]);
        }
    }
}

// Per block of depth-ordered Gaussians: its super-tile entries (part_s).
// Only splats some tile can list (255 o >= 1) get entries.
__device__ __forceinline__ unsigned long long super_entries(const float4 *cull, uint32_t g, int &sx0, int &sy0,
                                                            int &sx1, int &sy1) {
    int x0, y0, x1, y1;
    if (!cull_rect(cull, g, x0, y0, x1, y1)) return 0ull;
    return (unsigned long long)super_rect(x0, y0, x1, y1, sx0, sy0, sx1, sy1);
}

// Range of the depth-ordered Gaussians a block of the two kernels below owns.
__device__ __forceinline__ void entry_range(uint32_t n_vis, int64_t &lo, int64_t &hi) {
    const int64_t range = vis_range((int64_t)n_vis);
    lo = (int64_t)blockIdx.x * range;
    hi = lo + range < (int64_t)n_vis ? lo + range : (int64_t)n_vis;
}

__global__ void __launch_bounds__(kVisBlock) k_count_entries(const float4 *__restrict__ cull,
                                                             const uint32_t *__restrict__ order,
                                                             const uint32_t *__restrict__ n_vis,
                                                             unsigned long long *__restrict__ part_s) {
    wait_prior_grid();
    __shared__ unsigned long long ws[32];
    int64_t lo, hi;
    entry_range(*n_vis, lo, hi);
    unsigned long long c = 0ull;
#pragma unroll 4
    for (int64_t k = lo + threadIdx.x; k < hi; k += kVisBlock) {
        int sx0, sy0, sx1, sy1;
        c += super_entries(cull, order[k], sx0, sy0, sx1, sy1);
    }
    unsigned long long tot;
    block_scan_excl<unsigned long long>(c, ws, &tot);
    if (threadIdx.x == 0) part_s[blockIdx.x] = tot;
}

// Only when the super-tile entries alone overflowed the capacity (then the
// tile counts miss the dropped ones): P counted splat by splat, tile by tile.
// The tiles that list splat g, counted one by one.
__device__ __forceinline__ unsigned long long exact_tiles(const float *splats, uint32_t g, const DevCam &cam) {
    int x0, y0, x1, y1;
    const SplatShape sh = splat_shape(splats, g);
    if (sh.tau < 0.f || !cand_rect(splats, g, cam, sh.tau, x0, y0, x1, y1)) return 0ull;
    unsigned long long m = 0ull;
    for (int y = y0; y < y1; ++y)
        for (int x = x0; x < x1; ++x) m += tile_hit(sh, cam.tile, x, y) ? 1ull : 0ull;
    return m;
}

// A warp's sum of v added to *total (every lane of the warp calls it).
__device__ __forceinline__ void warp_add_total(unsigned long long v, unsigned long long *total) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(total, v);
}

// count_dev = P, the number of entries: the sum of the tile counts, or the
// exact count above when the super-tile entries overflowed.
__global__ void k_finish_count(const unsigned long long *__restrict__ total_t,
                               const unsigned long long *__restrict__ total_s,
                               const unsigned long long *__restrict__ total_exact, int64_t capacity,
                               int64_t *__restrict__ count_dev) {
    wait_prior_grid();
    const unsigned long long P = *total_s > (unsigned long long)capacity ? *total_exact : *total_t;
    *count_dev = (int64_t)P;
    if (P > (unsigned long long)capacity) atomicOr(&g_sort_flags, GS_FLAG_CAPACITY);
}

// The super-tile entries in depth order, clipped to the capacity (*sclip of
// them kept, of *total_s), and the first super-tile pass's digit counts.
__global__ void __launch_bounds__(kVisBlock, 5) k_emit_super(const float *__restrict__ splats,
                                                          const float4 *__restrict__ cull,
                                                          const uint32_t *__restrict__ order,
                                                          const uint32_t *__restrict__ n_vis, DevCam cam,
                                                          int supers_x, const unsigned long long *__restrict__ part_s,
                                                          unsigned long long *__restrict__ total_s,
                                                          uint32_t *__restrict__ sclip, int64_t capacity,
                                                          uint2 *__restrict__ entries,
                                                          uint32_t *__restrict__ skeys, uint32_t *__restrict__ svals,
                                                          unsigned long long *__restrict__ total_exact, Digit first) {
    __shared__ unsigned long long ps[64];
    __shared__ uint32_t buf[2][kVisBlock / 32];
    wait_prior_grid();
    const unsigned long long cap = (unsigned long long)capacity;
    const PartSum<unsigned long long> sum =
        part_sum<unsigned long long>(part_s, (int)gridDim.x, (int)blockIdx.x, ps);
    const uint32_t kept = (uint32_t)(sum.total > cap ? cap : sum.total);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *total_s = sum.total;
        *sclip = kept;
        if (sum.total > cap) atomicOr(&g_sort_flags, GS_FLAG_CAPACITY);
    }
    const uint32_t chunk = chunk_len(kept);
    unsigned long long at = sum.before;
    int64_t lo, hi;
    entry_range(*n_vis, lo, hi);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rounds = vis_rounds(hi - lo);
    int turn = 0;
    for (int64_t base = lo; base < hi; base += (int64_t)rounds * kVisBlock, ++turn) {
        const int64_t k0 = base + warp * 32 * rounds + lane;
        uint32_t g[kVisRounds], c[kVisRounds], before[kVisRounds], mine = 0u;
#pragma unroll
        for (int r = 0; r < kVisRounds; ++r)
            g[r] = r < rounds && k0 + 32 * r < hi ? order[k0 + 32 * r] : 0xffffffffu;
        int sx0, sy0, sx1, sy1;
#pragma unroll
        for (int r = 0; r < kVisRounds; ++r)
            c[r] = g[r] != 0xffffffffu ? (uint32_t)super_entries(cull, g[r], sx0, sy0, sx1, sy1) : 0u;
#pragma unroll
        for (int r = 0; r < kVisRounds; ++r) {  // at most 1024 x 65536 entries in a batch: 32 bits
            uint32_t x = c[r];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, x, o);
                if (lane >= o) x += y;
            }
            before[r] = mine + x - c[r];
            mine += __shfl_sync(kFull, x, 31);
        }
        const PartSum<uint32_t> w = warps_before(mine, buf, turn);
        const unsigned long long off0 = at + w.before;
        at += w.total;
        if (sum.total > cap) {  // the super-tile entries overflowed: P counted tile by tile
            unsigned long long m = 0ull;
            for (int r = 0; r < kVisRounds; ++r) m += c[r] ? exact_tiles(splats, g[r], cam) : 0ull;
            warp_add_total(m, total_exact);
        }
#pragma unroll
        for (int r = 0; r < kVisRounds; ++r) {
            if (c[r] == 0u) continue;
            unsigned long long off = off0 + before[r];
            super_entries(cull, g[r], sx0, sy0, sx1, sy1);
            for (int y = sy0; y < sy1; ++y)
                for (int x = sx0; x < sx1; ++x, ++off) {
                    if (off >= cap) break;
                    const uint32_t key = (uint32_t)(y * supers_x + x);
                    if (first.hist) {
                        entries[off] = make_uint2(key, g[r]);
                        count_next(first, key, (uint32_t)off, chunk);
                    } else {  // one super-tile: already in order
                        skeys[off] = key;
                        svals[off] = g[r];
                    }
                }
        }
    }
}

// Segments of the super-tile-sorted list: seg_lo / seg_hi [ns] (zero for an
// empty super-tile; both arrays zeroed before).
__global__ void __launch_bounds__(256) k_seg_mark(const uint32_t *__restrict__ skeys,
                                                 const uint32_t *__restrict__ count, uint32_t *__restrict__ seg_lo,
                                                 uint32_t *__restrict__ seg_hi) {
    wait_prior_grid();
    const uint32_t n = *count;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = skeys[e];
        if (e == 0 || skeys[e - 1] != k) seg_lo[k] = (uint32_t)e;
        if (e == (int64_t)n - 1 || skeys[e + 1] != k) seg_hi[k] = (uint32_t)(e + 1);
    }
}

// One block: chunk bases, chunk_base [ns + 1] (exclusive scan of
// ceil(len / kChunk)), and the record of every chunk, chunk_rec [chunks] (as
// the one-pass radix writes them).
__global__ void __launch_bounds__(1024) k_super_plan(const uint32_t *__restrict__ seg_lo,
                                                     const uint32_t *__restrict__ seg_hi, int ns,
                                                     uint32_t *__restrict__ chunk_base,
                                                     uint4 *__restrict__ chunk_rec) {
    wait_prior_grid();
    __shared__ uint32_t ws[32];
    uint32_t carry = 0;
    for (int base = 0; base < ns; base += 1024) {
        const int j = base + threadIdx.x;
        const uint32_t nc = j < ns ? (seg_hi[j] - seg_lo[j] + kChunk - 1) / kChunk : 0u;
        uint32_t tot;
        const uint32_t ex = block_scan_excl<uint32_t>(nc, ws, &tot);
        if (j < ns) {
            chunk_base[j] = carry + ex;
            for (uint32_t c = 0; c < nc; ++c)
                chunk_rec[carry + ex + c] = make_uint4((uint32_t)j, seg_lo[j] + c * kChunk, seg_hi[j], carry + ex);
        }
        carry += tot;
    }
    if (threadIdx.x == 0) chunk_base[ns] = carry;
}

// Shared part of the chunk kernels for chunk c: this thread's entry and the
// mask of the tiles of the super-tile that list it.
struct ChunkCtx {
    int s, sx, sy;
    uint32_t first;  // the super-tile's first chunk
    uint32_t g;
    unsigned long long mask;
};

// Scratch of the tile tests (shared memory, one slot per thread): hit masks
// as eight rows of tiles, a byte each; the entry's shape and the bounds of
// tile_hit_facing and row_span; its candidate rectangle packed as lx0 | ly0 << 3 |
// w << 6 | first row << 10; per warp the bits of the first rows (256 of them at
// most) and the entries that have any.
struct TestScratch {
    uint32_t *hit;     // [2 * kChunk]
    float4 *shape;     // [3 * kChunk]
    uint32_t *rect;    // [kChunk]
    uint32_t *starts;  // [kChunk / 32][8]
    uint8_t *owner;    // [kChunk]
};

// With masks_in NULL the masks are computed by the tile test (and stored to
// masks_out when given); else they are read.
__device__ __forceinline__ void chunk_load(ChunkCtx &cx, uint32_t c, const float *__restrict__ splats,
                                           const float4 *__restrict__ cull,
                                           const uint32_t *__restrict__ svals,
                                           const uint4 *__restrict__ chunk_rec, int supers_x,
                                           const DevCam &cam, const TestScratch &sc,
                                           const unsigned long long *__restrict__ masks_in,
                                           unsigned long long *__restrict__ masks_out) {
    __syncthreads();  // the previous chunk's shared data is no longer read
    const uint4 cr = chunk_rec[c];
    cx.s = (int)cr.x;
    cx.first = cr.w;
    cx.sx = cx.s % supers_x;
    cx.sy = cx.s / supers_x;
    const uint32_t e = cr.y + threadIdx.x;
    const bool valid = e < cr.z;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cx.mask = 0ull;
    cx.g = valid ? svals[e] : 0u;
    if (masks_in) {
        if (valid) cx.mask = masks_in[e];
        return;
    }
    // candidate tiles: the entry's rectangle inside this super-tile, w x h
    // tiles from (lx0, ly0) in the super-tile's own tile coordinates
    int lx0 = 0, ly0 = 0, w = 0, h = 0;
    if (valid) {  // every listed entry's splat has tau >= 0 and a candidate rectangle
        const float *r = splats + (int64_t)cx.g * kSplat;
        const float4 p0 = __ldg(reinterpret_cast<const float4 *>(r));
        const float4 c0 = __ldg(cull + 2 * (int64_t)cx.g);
        const uint4 c1 = __ldg(reinterpret_cast<const uint4 *>(cull) + 2 * (int64_t)cx.g + 1);
        sc.shape[3 * threadIdx.x] = p0;
        sc.shape[3 * threadIdx.x + 1] = make_float4(__ldg(r + 4), c0.x, c0.y, c0.z);
        sc.shape[3 * threadIdx.x + 2] = make_float4(c0.w, __uint_as_float(c1.z), __uint_as_float(c1.w), 0.f);
        int x0, y0, x1, y1;
        if (unpack_rect(c1, x0, y0, x1, y1)) {
            lx0 = max(x0 - cx.sx * kSuper, 0);
            ly0 = max(y0 - cx.sy * kSuper, 0);
            w = max(min(x1 - cx.sx * kSuper, kSuper) - lx0, 0);
            h = max(min(y1 - cx.sy * kSuper, kSuper) - ly0, 0);
        }
    }
    const int cnt = w > 0 ? h : 0;
    sc.hit[2 * threadIdx.x] = 0u;
    sc.hit[2 * threadIdx.x + 1] = 0u;
    uint32_t *starts = sc.starts + warp * 8;
    uint8_t *owner = sc.owner + warp * 32;
    if (lane < 8) starts[lane] = 0u;
    // the warp's (entry, row of tiles) pairs, spread evenly over its lanes
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const int excl = incl - cnt, total = __shfl_sync(kFull, incl, 31);
    const unsigned some = __ballot_sync(kFull, cnt > 0);
    __syncwarp();
    if (cnt) {
        sc.rect[threadIdx.x] = (uint32_t)(lx0 | (ly0 << 3) | (w << 6)) | ((uint32_t)excl << 10);
        owner[__popc(some & lanemask_lt())] = (uint8_t)lane;
        atomicOr(starts + (excl >> 5), 1u << (excl & 31));
    }
    __syncwarp();
    int passed = -1;  // entries that begin before this round, less one
    for (int base = 0; base < total; base += 32) {
        // row j belongs to the last entry that begins at or before it
        const int j = base + lane;
        const uint32_t word = starts[base >> 5];
        const int i = owner[min(31, passed + __popc(word & (kFull >> (31 - lane))))];
        passed += __popc(word);
        if (j < total) {
            const int o = warp * 32 + i;
            const uint32_t pk = sc.rect[o];
            const int ly = (int)((pk >> 3) & 7u) + j - (int)(pk >> 10);
            const int ox0 = (int)(pk & 7u), ox1 = ox0 + (int)((pk >> 6) & 15u);
            const float4 s0 = sc.shape[3 * o], s1 = sc.shape[3 * o + 1], s2 = sc.shape[3 * o + 2];
            SplatShape os;
            os.mx = s0.x; os.my = s0.y; os.a = s0.z; os.b = s0.w;
            os.c = s1.x; os.tau = s1.y; os.bc = s1.z; os.ba = s1.w;
            uint32_t hit = 0u, open = span_bits(ox0, ox1 - 1, ox0, ox1);
            if (s2.z > 0.f) {
                const RowSpan sp = row_span(os, s2.y, s2.z, cam.tile, cx.sx * kSuper * cam.tile, cx.sy * kSuper + ly);
                hit = span_bits(sp.sure_lo, sp.sure_hi, ox0, ox1);
                open = span_bits(sp.lo, sp.hi, ox0, ox1) & ~hit;
            }
            for (; open; open &= open - 1u) {
                const int x = __ffs((int)open) - 1;
                if (tile_hit_facing(os, s2.x, cam.tile, cx.sx * kSuper + x, cx.sy * kSuper + ly)) hit |= 1u << x;
            }
            reinterpret_cast<uint8_t *>(sc.hit)[8 * o + ly] = (uint8_t)hit;
        }
    }
    __syncwarp();
    cx.mask = ((unsigned long long)sc.hit[2 * threadIdx.x + 1] << 32) | sc.hit[2 * threadIdx.x];
    if (valid && masks_out) masks_out[e] = cx.mask;
}

// 32 x 32 bit-matrix transpose across a warp: lane i holds row i (bit j =
// M[i][j]); on return lane j holds column j (bit i = M[i][j]) -- for every
// slot j at once what __ballot_sync of bit j would give. Swaps the
// off-diagonal blocks of 16, 8, 4, 2 and 1 bits.
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x, int lane) {
    const uint32_t m16 = 0x0000FFFFu, m8 = 0x00FF00FFu, m4 = 0x0F0F0F0Fu, m2 = 0x33333333u, m1 = 0x55555555u;
#define GS_TSTEP(S, M)                                                                  \
    {                                                                                   \
        const uint32_t p = __shfl_xor_sync(kFull, x, S);                                \
        x = (lane & S) ? ((x & ~(M)) | ((p >> S) & (M))) : ((x & (M)) | ((p & (M)) << S)); \
    }
    GS_TSTEP(16, m16)
    GS_TSTEP(8, m8)
    GS_TSTEP(4, m4)
    GS_TSTEP(2, m2)
    GS_TSTEP(1, m1)
#undef GS_TSTEP
    return x;
}

// Global tile id of slot t of super-tile (sx, sy).
__device__ __forceinline__ int slot_tile(int t, int sx, int sy, int tiles_x) {
    return (sy * kSuper + (t >> 3)) * tiles_x + sx * kSuper + (t & 7);
}

// Bound by instruction issue and the latency of the records' gather. About 12
// candidate tiles per entry in 3.5 rows: a lane takes a row, whose listed tiles are
// a span found at once (row_span), and only the tiles at an uncertain end go
// through the test. 1M Gaussians, 931K entries: 66 us with the four-edge test of
// every tile, 61 with two edges and the owner found by a population count, 42 by
// rows (22M instead of 40M instructions); 3M Gaussians 117 -> 88 us.
__global__ void __launch_bounds__(kChunk, 5) k_chunk_counts(const float *__restrict__ splats,
                                                        const float4 *__restrict__ cull,
                                                        const uint32_t *__restrict__ svals,
                                                        const uint32_t *__restrict__ chunk_base,
                                                        const uint4 *__restrict__ chunk_rec, int ns,
                                                        int supers_x, DevCam cam, uint32_t *__restrict__ counts,
                                                        uint32_t *__restrict__ tile_count,
                                                        unsigned long long *__restrict__ masks) {
    wait_prior_grid();
    __shared__ uint32_t hit_mask[2 * kChunk];  // per entry, low and high halves
    __shared__ float4 shape[3 * kChunk];
    __shared__ uint32_t rect[kChunk];
    __shared__ uint32_t starts[kChunk / 32][8];
    __shared__ uint8_t owner[kChunk];
    __shared__ uint32_t cnt[kChunk / 32][64];  // per warp and slot: the warp's entries that the slot's tile lists
    const TestScratch sc{hit_mask, shape, rect, &starts[0][0], owner};
    const uint32_t nc = chunk_base[ns];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
        ChunkCtx cx;
        chunk_load(cx, c, splats, cull, svals, chunk_rec, supers_x, cam, sc, nullptr, masks);
        cnt[warp][lane] = (uint32_t)__popc(warp_transpose32((uint32_t)cx.mask, lane));
        cnt[warp][lane + 32] = (uint32_t)__popc(warp_transpose32((uint32_t)(cx.mask >> 32), lane));
        __syncthreads();
        if (threadIdx.x < 64) {
            const int t = threadIdx.x;
            uint32_t n = 0u;
#pragma unroll
            for (int w = 0; w < kChunk / 32; ++w) n += cnt[w][t];
            counts[(int64_t)c * 64 + t] = n;
            if (n) atomicAdd(tile_count + slot_tile(t, cx.sx, cx.sy, cam.tiles_x), n);
        }
    }
}

// Tile starts (exclusive scan of the tile counts over tile ids) and the
// ranges, clipped to the capacity: each block scans its own 1024 tiles from
// the sum of those in front, taken from the tile counts themselves while the
// grid is small (up to kDirectTiles blocks; 24 words per thread at most) and
// from per-block sums (k_tile_sums, one launch more) for larger ones. The last
// block also sets count_dev = P, the sum of the tile counts, or the exact
// count when the super-tile entries overflowed (and the capacity flag if P
// exceeds it).
constexpr int kDirectTiles = 24;

__global__ void __launch_bounds__(kScanBlock) k_tile_sums(const uint32_t *__restrict__ tile_count, int64_t tiles,
                                                         unsigned long long *__restrict__ part) {
    wait_prior_grid();
    __shared__ unsigned long long ws[32];
    const int64_t j = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
    unsigned long long tot;
    block_scan_excl<unsigned long long>(j < tiles ? tile_count[j] : 0ull, ws, &tot);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanBlock) k_tile_starts(const uint32_t *__restrict__ tile_count, int64_t tiles,
                                                           const unsigned long long *__restrict__ part,
                                                           int64_t capacity,
                                                           const unsigned long long *__restrict__ total_s,
                                                           const unsigned long long *__restrict__ total_exact,
                                                           unsigned long long *__restrict__ tile_start,
                                                           uint32_t *__restrict__ ranges,
                                                           int64_t *__restrict__ count_dev,
                                                           uint32_t *__restrict__ len_hist) {
    __shared__ unsigned long long ws[32];
    __shared__ unsigned long long ps[64];
    __shared__ uint32_t bins[kLenBuckets];
    if (threadIdx.x < kLenBuckets) bins[threadIdx.x] = 0u;
    wait_prior_grid();
    const int64_t first = (int64_t)blockIdx.x * kScanBlock, j = first + threadIdx.x;
    const unsigned long long n = j < tiles ? tile_count[j] : 0ull;
    if (len_hist) {  // tiles per length bucket, for the order that k_expand's first blocks make
        __syncthreads();
        take_place(bins, length_bucket((uint32_t)n), j < tiles);
        __syncthreads();
        if (threadIdx.x < kLenBuckets && bins[threadIdx.x]) atomicAdd(len_hist + threadIdx.x, bins[threadIdx.x]);
    }
    unsigned long long before;
    if (part) {
        before = part_sum<unsigned long long>(part, (int)gridDim.x, (int)blockIdx.x, ps).before;
    } else {
        unsigned long long b = 0ull;
#pragma unroll 8
        for (int64_t q = threadIdx.x; q < first; q += kScanBlock) b += tile_count[q];
        block_scan_excl<unsigned long long>(b, ws, &before);
    }
    unsigned long long tot;
    const unsigned long long st = before + block_scan_excl<unsigned long long>(n, ws, &tot);
    const unsigned long long cap = (unsigned long long)capacity;
    if (j < tiles) {
        const unsigned long long en = st + n;
        tile_start[j] = st;
        // an empty tile has the range (0, 0)
        ranges[2 * j] = n ? (uint32_t)(st < cap ? st : cap) : 0u;
        ranges[2 * j + 1] = n ? (uint32_t)(en < cap ? en : cap) : 0u;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        const unsigned long long P = *total_s > cap ? *total_exact : before + tot;
        *count_dev = (int64_t)P;
        if (P > cap) atomicOr(&g_sort_flags, GS_FLAG_CAPACITY);
    }
}

// What k_expand's first blocks turn into the tiles' order by list length: a
// counting sort, the buckets from k_tile_starts, kOrderTiles tiles per block.
constexpr int kOrderTiles = 4 * kChunk;
struct OrderPlan {
    int blocks;  // 0: no order is made
    const uint32_t *count, *hist;
    uint32_t *next;
    SortFront front;
    int tiles;
    uint2 key;
};

__device__ __forceinline__ void order_tiles(const OrderPlan &o, uint32_t *s /* 3 * kLenBuckets + 32 */) {
    static_assert(kChunk == kLenBuckets, "a bucket per thread");
    place_buckets<kOrderTiles / kChunk>(
        (int)blockIdx.x, o.tiles, [&](int t) { return o.count[t]; },
        [&](int t, uint32_t at) {
            o.front.order[at] = (uint32_t)t;
            o.front.depth[t] = 0;
        },
        o.hist, o.next, s);
    if (blockIdx.x == 0) {
        o.front.hist[threadIdx.x] = o.front.next[threadIdx.x] = 0u;
        if (threadIdx.x == 0) *o.front.stamp = o.key;
    }
}

// Bound by instruction issue; a slot's place and its lanes are one 8-byte word
// in shared memory and positions have 32 bits (40 -> 30 us at 931K entries,
// 4.8M places).
__global__ void __launch_bounds__(kChunk) k_expand(const float *__restrict__ splats, const uint32_t *__restrict__ svals,
                                                  const uint32_t *__restrict__ chunk_base,
                                                  const uint4 *__restrict__ chunk_rec, int ns, int supers_x,
                                                  DevCam cam, const uint32_t *__restrict__ counts,
                                                  const unsigned long long *__restrict__ tile_start, int64_t capacity,
                                                  const unsigned long long *__restrict__ masks,
                                                  uint32_t *__restrict__ vals, OrderPlan plan) {
    wait_prior_grid();
    constexpr int kW = kChunk / 32;
    // per (warp, slot): where the warp's entries of the slot's tile start in the
    // final list (clipped to the capacity), and the lanes whose entry it lists
    __shared__ uint2 place[kW][64];
    __shared__ uint32_t before[kChunk / 64][64];         // partial sums of earlier chunks' counts
    if ((int)blockIdx.x < plan.blocks) {
        order_tiles(plan, reinterpret_cast<uint32_t *>(&place[0][0]));
        return;
    }
    const uint32_t nc = chunk_base[ns], cap = (uint32_t)capacity;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    for (uint32_t c = blockIdx.x - plan.blocks; c < nc; c += gridDim.x - plan.blocks) {
        ChunkCtx cx;
        chunk_load(cx, c, splats, nullptr, svals, chunk_rec, supers_x, cam, TestScratch{}, masks, nullptr);
        const uint32_t lo = (uint32_t)cx.mask, hi = (uint32_t)(cx.mask >> 32);
        place[warp][lane].y = warp_transpose32(lo, lane);
        place[warp][lane + 32].y = warp_transpose32(hi, lane);
        {   // entries of each slot in the super-tile's earlier chunks: 4 threads per slot,
            // four independent sums so that the loads overlap
            constexpr int kQ = kChunk / 64;
            const int t = threadIdx.x & 63, q = threadIdx.x >> 6;
            uint32_t n0 = 0u, n1 = 0u, n2 = 0u, n3 = 0u;
            uint32_t c2 = cx.first + q;
            for (; c2 + 3 * kQ < c; c2 += 4 * kQ) {
                n0 += counts[(int64_t)c2 * 64 + t];
                n1 += counts[(int64_t)(c2 + kQ) * 64 + t];
                n2 += counts[(int64_t)(c2 + 2 * kQ) * 64 + t];
                n3 += counts[(int64_t)(c2 + 3 * kQ) * 64 + t];
            }
            for (; c2 < c; c2 += kQ) n0 += counts[(int64_t)c2 * 64 + t];
            before[q][t] = (n0 + n1) + (n2 + n3);
        }
        __syncthreads();
        if (threadIdx.x < 64) {
            const int t = threadIdx.x;
            const bool inside = cx.sx * kSuper + (t & 7) < cam.tiles_x && cx.sy * kSuper + (t >> 3) < cam.tiles_y;
            unsigned long long run = 0ull;
            if (inside) {
                run = tile_start[slot_tile(t, cx.sx, cx.sy, cam.tiles_x)];
#pragma unroll
                for (int q = 0; q < kChunk / 64; ++q) run += before[q][t];
            }
            uint32_t at = (uint32_t)(run < (unsigned long long)cap ? run : (unsigned long long)cap);
#pragma unroll
            for (int w = 0; w < kW; ++w) {  // below 2^31 + 256 + ...: 32 bits hold it
                place[w][t].x = at;
                at += (uint32_t)__popc(place[w][t].y);
            }
        }
        __syncthreads();
        // An entry's position in tile t's list: the warp's start there plus the
        // lanes before it that tile t lists. Written slot by slot over the
        // slots some lane has (a warp's entries of one tile go to consecutive
        // words) or, when that takes more rounds, each lane over its own slots.
        const unsigned any_lo = __reduce_or_sync(kFull, lo), any_hi = __reduce_or_sync(kFull, hi);
        const int by_slot = __popc(any_lo) + __popc(any_hi);
        const bool by_lane = (int)__reduce_max_sync(kFull, (unsigned)__popcll(cx.mask)) < by_slot;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t mine = half ? hi : lo;
            for (uint32_t u = by_lane ? mine : (half ? any_hi : any_lo); u; u &= u - 1u) {
                const int t = __ffs((int)u) - 1;
                if ((mine >> t) & 1u) {
                    const uint2 p = place[warp][32 * half + t];
                    const uint32_t pos = p.x + (uint32_t)__popc(p.y & lt);
                    if (pos < cap) vals[pos] = cx.g;
                }
            }
        }
    }
}

// ---- workspace ----
struct SortWs {
    uint2 *kv[2];                 // visible Gaussians: (depth key, index)
    uint32_t *order;              // [n] their indices in depth order
    uint2 *entries[2];            // super-tile entries: (super-tile, index); the second shares the masks' place
    uint32_t *skeys, *svals;      // in super-tile order
    uint32_t *hist_d, *hist_s;    // digit counts of the depth and super-tile passes (hist_of)
    uint32_t *part32;
    unsigned long long *part_s, *total_s, *total_t, *total_exact;
    unsigned long long *masks;                 // [capacity] tile mask of each super-tile entry
    unsigned long long *tile_part;             // [tile blocks]
    float4 *cull;                              // [2 n] cull record of each visible Gaussian
    uint32_t *n_vis, *sclip;
    DepthSpan *span;
    uint32_t *seg_lo, *seg_hi, *chunk_base;    // [ns], [ns], [ns + 1]
    uint32_t *tile_count;                      // [tiles]
    uint32_t *len_hist, *len_next;             // [kLenBuckets] tiles per length bucket, places given out
    SortFront front;
    unsigned long long *tile_start;            // [tiles]
    uint32_t *chunk_counts;                    // [max chunks][64]
    uint4 *chunk_rec;                          // [max chunks]
    size_t bytes;
};

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

inline int64_t max_chunks(int64_t cap, int64_t ns) { return (cap + kChunk - 1) / kChunk + ns + 1; }

constexpr int kDepthPasses = 4, kSuperPasses = 2;  // super-tile ids take at most 16 bits

// Digit counts of pass p of a sort whose count is at most n.
inline uint32_t *hist_of(uint32_t *base, int64_t n, int p) { return base + (size_t)p * chunk_rows(n) * kMaxRadix; }

inline SortWs sort_layout(char *base, int64_t n, int64_t cap, int64_t tiles, int64_t ns) {
    SortWs w;
    size_t off = 0;
    auto take = [&](size_t bytes) -> char * {
        char *p = base ? base + off : nullptr;
        off += align256(bytes);
        return p;
    };
    w.front = sort_front(base, tiles);  // first: found by the rasteriser from the grid alone
    take(w.front.bytes);
    for (int k = 0; k < 2; ++k) w.kv[k] = (uint2 *)take(8 * (size_t)n);
    w.order = (uint32_t *)w.kv[0];  // written by the pass that reads kv[1]
    w.entries[0] = (uint2 *)take(8 * (size_t)cap);
    w.svals = (uint32_t *)take(4 * (size_t)cap);
    w.skeys = (uint32_t *)w.entries[0];  // kept only by two passes (the second reads entries[1]) or none
    w.hist_d = (uint32_t *)take(4 * (size_t)kDepthPasses * kMaxRadix * (size_t)chunk_rows(n));
    w.hist_s = (uint32_t *)take(4 * (size_t)kSuperPasses * kMaxRadix * (size_t)chunk_rows(cap));
    w.part32 = (uint32_t *)take(4 * 3 * (size_t)kVisGrid);
    w.part_s = (unsigned long long *)take(8 * (size_t)kVisGrid);
    w.total_s = (unsigned long long *)take(8);
    w.total_t = (unsigned long long *)take(8);
    w.total_exact = (unsigned long long *)take(8);
    w.masks = (unsigned long long *)take(8 * (size_t)cap);
    w.entries[1] = (uint2 *)w.masks;  // the masks are made after the sort
    w.cull = (float4 *)take(32 * (size_t)n);
    w.n_vis = (uint32_t *)take(4);
    w.span = (DepthSpan *)take(sizeof(DepthSpan));
    w.sclip = (uint32_t *)take(4);
    // zeroed together before each sort: segment bounds, tile counts, length buckets
    w.seg_lo = (uint32_t *)take(4 * (size_t)(2 * ns + tiles + 2 * kLenBuckets));
    w.seg_hi = w.seg_lo ? w.seg_lo + ns : nullptr;
    w.tile_count = w.seg_lo ? w.seg_lo + 2 * ns : nullptr;
    w.len_hist = w.seg_lo ? w.tile_count + tiles : nullptr;
    w.len_next = w.seg_lo ? w.len_hist + kLenBuckets : nullptr;
    w.chunk_base = (uint32_t *)take(4 * (size_t)(ns + 1));
    w.chunk_rec = (uint4 *)take(16 * (size_t)max_chunks(cap, ns));
    w.tile_part = (unsigned long long *)take(8 * (size_t)((tiles + kScanBlock - 1) / kScanBlock));
    w.tile_start = (unsigned long long *)take(8 * (size_t)tiles);
    w.chunk_counts = (uint32_t *)take(4 * 64 * (size_t)max_chunks(cap, ns));
    w.bytes = off;
    return w;
}

struct SuperGrid {
    int supers_x, supers_y;
    int64_t tiles, ns;
};

inline SuperGrid super_grid(int32_t width, int32_t height, int32_t tile) {
    SuperGrid g;
    const int tx = (width + tile - 1) / tile, ty = (height + tile - 1) / tile;
    g.supers_x = (tx + kSuper - 1) / kSuper;
    g.supers_y = (ty + kSuper - 1) / kSuper;
    g.tiles = (int64_t)tx * ty;
    g.ns = (int64_t)g.supers_x * g.supers_y;
    return g;
}

// The digits of a sort on `total_bits` low bits: 8 bits each, or one pass of up
// to kMaxRadixBits when that suffices.
inline int radix_passes(int total_bits) {
    return total_bits <= 0 ? 0 : (total_bits <= kMaxRadixBits ? 1 : (total_bits + 7) / 8);
}

inline Digit radix_digit(uint32_t *hist, int64_t bound, int total_bits, int p) {
    const int npass = radix_passes(total_bits);
    if (p >= npass) return Digit{nullptr, 0, 0};
    const int per = (total_bits + npass - 1) / npass, shift = p * per;
    return Digit{hist_of(hist, bound, p), shift, per < total_bits - shift ? per : total_bits - shift};
}

// Lets the two kernels that need more than 48 KB of shared memory be launched
// with the most they ever take. The limit belongs to the function on the
// device, not to a launch: it is the same in every call and never lowered, so
// that another thread's sort, or a captured launch replayed later, finds it.
bool allow_shared() {
    constexpr size_t radix_most = (sizeof(uint32_t) * (size_t)kRadixWarps) << kMaxRadixBits;  // 64 KB
    const auto most = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return accepted(cudaFuncSetAttribute(k_radix_pass, most, (int)radix_most)) &&
           accepted(cudaFuncSetAttribute(k_depth_small, most, (int)kSmallShared));
}

// A radix pass over a count of at most `bound`, on a digit of at most `bits`.
template <typename... Args>
cudaError_t launch_radix(int bits, int64_t bound, cudaStream_t s, Args &&...args) {
    const size_t smem = (sizeof(uint32_t) * (size_t)kRadixWarps) << bits;  // at most allow_shared's
    return launch_chained_smem(k_radix_pass, (unsigned)chunk_rows(bound), kRadixThreads, smem, s,
                               static_cast<Args &&>(args)...);
}

int ceil_log2(int64_t x) {
    int b = 0;
    while ((int64_t(1) << b) < x) ++b;
    return b;
}

}  // namespace

uint32_t take_sort_flags() {
    uint32_t f = 0, z = 0;
    cudaMemcpyFromSymbol(&f, g_sort_flags, sizeof(f));
    cudaMemcpyToSymbol(g_sort_flags, &z, sizeof(z));
    return f;
}

}  // namespace gs

using namespace gs;

extern "C" size_t gs_sort_workspace_bytes(int64_t n, int64_t capacity, int32_t width, int32_t height, int32_t tile) {
    if (n < 0 || capacity < 0 || width <= 0 || height <= 0 || !tile_ok(tile)) return 0;
    const SuperGrid sg = super_grid(width, height, tile);
    return sort_layout(nullptr, n, capacity, sg.tiles, sg.ns).bytes;
}

extern "C" int gs_sort(const float *splats, int64_t n, const gs_camera *cam, void *ws, size_t ws_bytes,
                       int64_t capacity, uint32_t *vals, uint32_t *ranges, int64_t *count_dev, gs_stream_t stream) {
    if (n < 0 || n > INT32_MAX || capacity < 0 || capacity > INT32_MAX || !camera_ok(cam)) return GS_ERR_INVALID_ARG;
    if (!ranges || !count_dev || (n > 0 && !splats) || (capacity > 0 && !vals)) return GS_ERR_INVALID_ARG;
    const SuperGrid sg = super_grid(cam->width, cam->height, cam->tile);
    SortWs w = sort_layout(static_cast<char *>(ws), n, capacity, sg.tiles, sg.ns);
    if (!ws || ws_bytes < w.bytes) return GS_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(ws) & 255) return GS_ERR_INVALID_ARG;
    cudaStream_t s = as_stream(stream);
    DevCam dc = make_cam(cam);
    const int64_t tiles = sg.tiles;
    const int ns = (int)sg.ns;

    if (n == 0 || capacity == 0) {
        k_zero_u32<<<grid_for(2 * tiles, 256), 256, 0, s>>>(ranges, 2 * tiles);
        note_launches(1);
        if (n == 0) {
            if (!accepted(cudaMemsetAsync(count_dev, 0, sizeof(int64_t), s)) ||
                !accepted(cudaMemsetAsync(w.front.stamp, 0, sizeof(uint2), s)))  // no order either
                return GS_ERR_CUDA;
            return launch_status();
        }
    }
    const int sbits = ceil_log2(sg.ns), npass = radix_passes(sbits);
    // A launch that is refused ends the call: the kernels behind it would read as
    // counts and indices whatever lies in the place of its output.
    if (!allow_shared()) return GS_ERR_CUDA;
    // stage 1: visible Gaussians by depth (the first kernel also zeroes the
    // segment bounds, tile counts, digit counts and exact count)
    const ZeroSpans z{{w.seg_lo, w.hist_d, w.hist_s},
                      {2 * sg.ns + tiles + 2 * kLenBuckets, kDepthPasses * kMaxRadix * chunk_rows(n),
                       capacity ? npass * kMaxRadix * chunk_rows(capacity) : 0}};
    const unsigned vgrid = vis_blocks(n), egrid = entry_blocks(n);
    const size_t hstride = (size_t)chunk_rows(n) * kMaxRadix;
    if (!accepted(launch_chained(k_count_visible, vgrid, kVisBlock, s, splats, n, w.part32, z, w.total_exact,
                                 w.front.stamp)))
        return GS_ERR_CUDA;
    if (!accepted(launch_chained(k_emit_visible, vgrid, kVisBlock, s, splats, n, w.part32, dc, w.kv[0], w.kv[1],
                                 w.cull, w.n_vis, w.span, w.hist_d, hstride)))
        return GS_ERR_CUDA;
    if (n <= kSmallSort) {
        if (!accepted(launch_chained_smem(k_depth_small, 1, kRadixThreads, kSmallShared, s, w.kv[0], w.kv[1], w.order,
                                          w.n_vis, w.span)))
            return GS_ERR_CUDA;
        note_launches(3);
    } else {
        for (int k = 0; k < kDepthPasses; ++k)
            if (!accepted(launch_radix(kMaxRadixBits, n, s, w.kv[k & 1], w.kv[1 - (k & 1)],
                                       static_cast<uint32_t *>(nullptr), k == 3 ? w.order : nullptr, w.n_vis,
                                       Digit{w.hist_d, 0, 0}, Digit{nullptr, 0, 0}, w.span, k, hstride, SegPlan{})))
                return GS_ERR_CUDA;
        note_launches(2 + kDepthPasses);
    }
    const uint32_t *order = w.order;
    // stage 2: super-tile entries in depth order, stable-sorted by super-tile
    if (!accepted(launch_chained(k_count_entries, egrid, kVisBlock, s, w.cull, order, w.n_vis, w.part_s)))
        return GS_ERR_CUDA;
    note_launches(1);
    if (!accepted(launch_chained(k_emit_super, egrid, kVisBlock, s, splats, w.cull, order, w.n_vis, dc, sg.supers_x,
                                 w.part_s, w.total_s, w.sclip, capacity, w.entries[0], w.skeys, w.svals, w.total_exact,
                                 capacity ? radix_digit(w.hist_s, capacity, sbits, 0) : Digit{nullptr, 0, 0})))
        return GS_ERR_CUDA;
    note_launches(1);
    if (capacity == 0) {
        cudaMemsetAsync(w.total_t, 0, sizeof(unsigned long long), s);
        if (!accepted(launch_chained(k_finish_count, 1, 1, s, w.total_t, w.total_s, w.total_exact, capacity,
                                     count_dev)))
            return GS_ERR_CUDA;
        note_launches(1);
        return launch_status();
    }
    // One pass (up to 512 super-tiles): its digit ranges are the segments, written
    // by the pass itself. Two: the second leaves the keys, which mark them.
    for (int p = 0; p < npass; ++p) {
        const bool last = p == npass - 1;
        const Digit dg = radix_digit(w.hist_s, capacity, sbits, p);
        if (!accepted(launch_radix(dg.bits, capacity, s, w.entries[p], w.entries[1],
                                   last && npass == 2 ? w.skeys : nullptr, last ? w.svals : nullptr, w.sclip, dg,
                                   radix_digit(w.hist_s, capacity, sbits, p + 1), static_cast<DepthSpan *>(nullptr), 0,
                                   size_t(0), npass == 1 ? SegPlan{w.chunk_base, w.chunk_rec, ns, kChunk} : SegPlan{})))
            return GS_ERR_CUDA;
        note_launches(1);
    }
    // stage 3: per-tile lists
    const int64_t chunks = max_chunks(capacity, sg.ns), resident = resident_blocks();
    const unsigned cgrid = (unsigned)(chunks < resident ? chunks : resident);
    if (npass != 1) {
        if (!accepted(launch_chained(k_seg_mark, (unsigned)resident, 256, s, w.skeys, w.sclip, w.seg_lo, w.seg_hi)))
            return GS_ERR_CUDA;
        if (!accepted(launch_chained(k_super_plan, 1, 1024, s, w.seg_lo, w.seg_hi, ns, w.chunk_base, w.chunk_rec)))
            return GS_ERR_CUDA;
        note_launches(2);
    }
    if (!accepted(launch_chained(k_chunk_counts, cgrid, kChunk, s, splats, w.cull, w.svals, w.chunk_base, w.chunk_rec,
                                 ns, sg.supers_x, dc, w.chunk_counts, w.tile_count, w.masks)))
        return GS_ERR_CUDA;
    OrderPlan plan{};
    if (tiles >= kOrderMinTiles)
        plan = OrderPlan{(int)((tiles + kOrderTiles - 1) / kOrderTiles), w.tile_count, w.len_hist, w.len_next, w.front,
                         (int)tiles, tile_order_key(dc.tiles_x, dc.tiles_y, dc.tile)};
    const int tb = (int)((tiles + kScanBlock - 1) / kScanBlock);
    const bool direct = tb <= kDirectTiles;
    if (!direct) {
        if (!accepted(launch_chained(k_tile_sums, tb, kScanBlock, s, w.tile_count, tiles, w.tile_part)))
            return GS_ERR_CUDA;
        note_launches(1);
    }
    if (!accepted(launch_chained(k_tile_starts, tb, kScanBlock, s, w.tile_count, tiles,
                                 direct ? nullptr : w.tile_part, capacity, w.total_s, w.total_exact, w.tile_start,
                                 ranges, count_dev, plan.blocks ? w.len_hist : nullptr)))
        return GS_ERR_CUDA;
    if (!accepted(launch_chained(k_expand, cgrid + plan.blocks, kChunk, s, splats, w.svals, w.chunk_base, w.chunk_rec,
                                 ns, sg.supers_x, dc, w.chunk_counts, w.tile_start, capacity, w.masks, vals, plan)))
        return GS_ERR_CUDA;
    note_launches(3);  // chunk counts, tile starts, lists
    return launch_status();
}
