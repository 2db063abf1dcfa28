// Tile rasteriser: front-to-back alpha compositing (Sec. 3.1, Eq. 2) and its
// backward (Sec. 3.2.4), which skips the gradient work of frozen Gaussians.
//
// One CTA per screen tile; the tile's sorted splat list is staged through
// shared memory, so every thread reads each splat as a shared-memory
// broadcast. No tensor cores: the work is a per-pixel exponential and a
// handful of FMAs.
//
// The backward walks each list back to front and recovers the transmittance
// in front of every splat from the value the forward left over, so no
// per-pixel list is stored. A warp's pixels see the same splat at the same
// time; its nine gradient terms are summed with a recursive-halving warp
// reduction and added to the splat's row in global memory.
#include "common.cuh"

static_assert(sizeof(gs_camera) == 112, "gs_camera layout");
static_assert(sizeof(gs_raster_job) == 184, "gs_raster_job layout");

namespace gs {
namespace {


// ---- warps of a tile ----
// A tile is cut into blocks of 8 x 4 PPT pixels, one per warp: lane l owns the
// pixels (l % 8, l / 8 + 4 k), k < PPT, of its warp's block. Every warp walks
// the tile's list by itself, 32 entries at a time, and keeps of them only the
// splats that can reach its own block (block_hit); where the block is the
// tile (8-pixel tiles, two pixels per thread) the list is already that
// selection. So a tile of 16 or 32 pixels pays per 8-pixel block what 8-pixel
// tiles pay, and no warp waits for another.
//
// With an even number of pixels per thread the pixels go in pairs through the
// packed FP32 instructions (f2_*); the code is written once over a value type
// V (f32x2 or float) with the same rounded operations, so every shape gives
// the same bits.
__device__ __forceinline__ float v_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ f32x2 v_sub(f32x2 a, f32x2 b) { return f2_sub(a, b); }
__device__ __forceinline__ float v_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ f32x2 v_mul(f32x2 a, f32x2 b) { return f2_mul(a, b); }
__device__ __forceinline__ float v_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ f32x2 v_fma(f32x2 a, f32x2 b, f32x2 c) { return f2_fma(a, b, c); }
__device__ __forceinline__ void v_get(float v, float (&o)[1]) { o[0] = v; }
__device__ __forceinline__ void v_get(f32x2 v, float (&o)[2]) { f2_unpack(v, o[0], o[1]); }
__device__ __forceinline__ void v_set(float &v, const float (&o)[1]) { v = o[0]; }
__device__ __forceinline__ void v_set(f32x2 &v, const float (&o)[2]) { v = f2_pack(o[0], o[1]); }
__device__ __forceinline__ float v_lo(float v) { return v; }
__device__ __forceinline__ float v_lo(f32x2 v) {
    float a, b;
    f2_unpack(v, a, b);
    return a;
}
template <class V>
__device__ __forceinline__ V v_dup(float x);
template <>
__device__ __forceinline__ float v_dup<float>(float x) { return x; }
template <>
__device__ __forceinline__ f32x2 v_dup<f32x2>(float x) { return f2_pack(x, x); }

template <int PPT>
struct Lanes {
    static constexpr int L = PPT % 2 == 0 ? 2 : 1;  // pixels per value
    static constexpr int NP = PPT / L;              // values per thread
};
template <int L>
struct ValueOf { typedef float T; };
template <>
struct ValueOf<2> { typedef f32x2 T; };

template <class V>
struct alignas(16) V4 {
    V x, y, z, w;
};

constexpr int kStage = 32;  // list entries a warp stages at once, one per lane

// The staged splats of one warp, every value duplicated into the halves of V:
// a = (mean_x, mean_y, -conic_a / 2, -conic_b), b = (-conic_c / 2, opacity,
// red, green) and blue -- the halves and signs formed once per splat instead
// of once per thread (exact).
template <class V>
struct Stage {
    V4<V> a[kStage], b[kStage];
    V blue[kStage];
    uint8_t pos[kStage];  // list position of each staged splat, from the first entry of the 32
};

struct SplatIn {  // what the rasteriser reads of a splat record
    float4 xa, co;
    float blue;
};

__device__ __forceinline__ SplatIn splat_in(const float *__restrict__ splats, uint32_t g) {
    const float4 *r = reinterpret_cast<const float4 *>(splats + (int64_t)g * kSplat);
    SplatIn s;
    s.xa = __ldg(r);
    s.co = __ldg(r + 1);
    s.blue = __ldg(reinterpret_cast<const float *>(r + 2));
    return s;
}

// Whether every value of the record is finite (0 x is NaN where x is not).
__device__ __forceinline__ bool all_finite(const SplatIn &s) {
    const float p = fmaf(0.f, s.xa.z, fmaf(0.f, s.xa.y, 0.f * s.xa.x));
    const float q = fmaf(0.f, s.co.y, fmaf(0.f, s.co.x, 0.f * s.xa.w));
    const float r = fmaf(0.f, s.blue, fmaf(0.f, s.co.w, 0.f * s.co.z));
    return p + q + r == 0.f;
}

template <class V>
__device__ __forceinline__ void stage_splat(Stage<V> &S, int q, const SplatIn &s) {
    S.a[q] = V4<V>{v_dup<V>(s.xa.x), v_dup<V>(s.xa.y), v_dup<V>(__fmul_rn(-0.5f, s.xa.z)), v_dup<V>(-s.xa.w)};
    S.b[q] = V4<V>{v_dup<V>(__fmul_rn(-0.5f, s.co.x)), v_dup<V>(s.co.y), v_dup<V>(s.co.z), v_dup<V>(s.co.w)};
    S.blue[q] = v_dup<V>(s.blue);
}

// Whether the splat may blend at a pixel of the block [x0, x1] x [y0, y1]
// (pixel centres). False only when alpha stays below 1/255 on the whole
// block: q = d^T Q d exceeds tau + 2e-3 (1 + |tau|), tau = 2 ln(255 o),
// everywhere on it. For a centre outside the block the least q lies on an
// edge that faces the centre, at the clamped minimiser of that edge; both
// facing edges are tried (any point of the block only lowers the least value
// found). Rounding: with kappa = (a + |b| + c)(a + c) / det, this evaluation
// and the compositing's own exponent are each off by at most 4 u kappa q
// (u = 2^-24); up to kappa = 1e3 that is 5e-4 q together, inside the margin,
// and conics beyond are never rejected. So the pixels' results do not depend
// on this test.
__device__ __forceinline__ bool block_hit(const SplatIn &s, float x0, float x1, float y0, float y1) {
    const float mx = s.xa.x, my = s.xa.y, a = s.xa.z, b = s.xa.w, c = s.co.x;
    const float det = a * c - b * b;
    if (!(det > 0.f) || !(a > 0.f) || !(c > 0.f)) return true;
    if (!((a + fabsf(b) + c) * (a + c) <= 1e3f * det)) return true;
    const float tau = 2.f * __logf(255.f * s.co.y);
    const float lim = tau + 2e-3f * (1.f + fabsf(tau));
    const float dx = fminf(fmaxf(mx, x0), x1) - mx, dy = fminf(fmaxf(my, y0), y1) - my;
    const float yy = fminf(fmaxf(my - __fdividef(b, c) * dx, y0), y1) - my;
    const float xx = fminf(fmaxf(mx - __fdividef(b, a) * dy, x0), x1) - mx;
    const float q1 = a * dx * dx + 2.f * b * dx * yy + c * yy * yy;
    const float q2 = a * xx * xx + 2.f * b * xx * dy + c * dy * dy;
    return !(fminf(q1, q2) > lim);
}

// Alpha of one splat at the L pixels of a value (0 where the splat is skipped:
// positive exponent or alpha < 1/255), with splat_power's rounded operations.
template <int L, class V>
__device__ __forceinline__ void alphas(V px, V py, const V4<V> &a, const V4<V> &b, float (&al)[L], bool (&use)[L],
                                       V &dy, float (&oG)[L]) {  // use: in, whether the pixel takes part
    const V dx = v_sub(a.x, px);
    const V c0 = v_mul(a.z, v_mul(dx, dx)), c1 = v_mul(a.w, dx);
    dy = v_sub(a.y, py);
    const V pw = v_fma(v_fma(b.x, dy, c1), dy, c0);
    float p[L], x[L], G[L];
    v_get(pw, p);
    v_get(v_mul(pw, v_dup<V>(kLog2e)), x);
#pragma unroll
    for (int l = 0; l < L; ++l) G[l] = ex2_ftz(x[l]);
    V g;
    v_set(g, G);
    v_get(v_mul(b.y, g), oG);
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const float m = fminf(kAlphaMax, oG[l]);
        use[l] = use[l] && p[l] <= 0.f && m >= kAlphaMin;
        al[l] = use[l] ? m : 0.f;
    }
}

// The compositing forward of one tile. It is bound by instruction issue and by
// the longest tile's chain of splats, not by memory.
//
// What a step does per pixel: two compares decide whether the splat blends,
// a select zeroes alpha if not, and from there on nothing is conditional (an
// alpha of 0 leaves T and, the splat's colour being finite, the colour as they
// are, bit for bit). A pixel that
// has stopped gets a NaN row coordinate, so that every later exponent is NaN
// and fails its compare: no done flag is tested. G splats are evaluated
// together -- their alphas do not depend on one another, only T runs through
// them -- and the stop T < 1e-4 is tested once per G, on the last T (T never
// grows): only a group that crosses it is gone through splat by splat.
//
// With RES, the walk also records where the backward may start: of every 32
// list entries that have an unfrozen one, the state after the last of them
// (resume_pos[tile] = 1 + its list position, 0 if the tile has none; per pixel
// resume = (T there, the colour blended behind it)), so that the backward
// skips the frozen splats behind it: they carry no gradient, and the state
// they would rebuild is this one. Rays that all stop in front of that entry,
// but among its 32, have their final state there: no unfrozen splat that was
// blended lies behind the recorded position, and at most 31 frozen ones in
// front of it are visited for nothing. The position depends on the list, the
// freeze map and the tile's deepest ray alone, not on how the tile is cut
// into warps: the groups of 32 are the list's, and the deepest warp's decides.
//
// Measured against the kernel before it (a barrier-separated batch per CTA,
// done flags and a stop test per splat, every warp through the whole tile's
// list), tiles ascending: 1M Gaussians, 1237x822, 8-pixel tiles, two pixels per
// thread with the record 199 -> 136 us; 3M at 1920x1080, 16-pixel tiles, one
// pixel per thread 671 -> 325 us; 400K at 800x800, 16-pixel tiles, one pixel, with
// the record 262 -> 98 us; 2K at 128x128 33 -> 12.5 us; the same bits in image, T
// and last contributor. (With a record kept per batch of the list 140, 103 and
// 14 us.)
template <int TS, int PPT, bool RES>
__device__ __forceinline__ void render_tile(const float *__restrict__ splats, const uint32_t *__restrict__ vals,
                                            const uint32_t *__restrict__ ranges, const DevCam &cam,
                                            float *__restrict__ image, float *__restrict__ t_final,
                                            int32_t *__restrict__ n_last, int tile,
                                            const uint8_t *__restrict__ frozen = nullptr,
                                            float4 *__restrict__ resume = nullptr,
                                            int32_t *__restrict__ resume_pos = nullptr,
                                            int32_t *__restrict__ depth = nullptr) {
    constexpr int L = Lanes<PPT>::L, NP = Lanes<PPT>::NP;
    typedef typename ValueOf<L>::T V;
    constexpr int kWarps = TS * TS / PPT / 32, kH = 4 * PPT;
    constexpr bool kWholeTile = TS == 8 && kH == 8;  // the warp's block is the tile
    constexpr int kG = 4;
    // RES: the snapshot (T, colour) of every pixel waits in shared memory (in
    // registers for 32-pixel tiles, whose staging takes most of it)
    constexpr bool kSnapShared = RES && TS <= 16;
    __shared__ Stage<V> s_stage[kWarps];
    __shared__ float4 s_snap[kSnapShared ? TS * TS : 1];
    __shared__ int s_upos;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Stage<V> &S = s_stage[warp];
    const int bx = (tile % cam.tiles_x) * TS + (warp % (TS / 8)) * 8;
    const int by = (tile / cam.tiles_x) * TS + (warp / (TS / 8)) * kH;
    const int px = bx + (lane & 7), py0 = by + (lane >> 3);
    const uint32_t start = ranges[2 * tile];
    const int n = (int)(ranges[2 * tile + 1] - start);
    const uint32_t *list = vals + start;
    const float nan = __int_as_float(0x7fffffff);

    const V fx = v_dup<V>((float)px), one = v_dup<V>(1.f);
    V T[NP], r[NP], g[NP], b[NP];
    float fy[PPT];  // row coordinate; NaN once the pixel is done (or outside the image)
    int last[PPT], hit_last[PPT];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        T[h] = one;
        r[h] = g[h] = b[h] = v_dup<V>(0.f);
    }
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int y = py0 + 4 * k;
        fy[k] = px < cam.W && y < cam.H ? (float)y : nan;
        last[k] = 0;
        hit_last[k] = -1;
    }
    float4 u[PPT];  // RES: T and colour after the last unfrozen splat passed
    int upos = 0, snap_at = -1;  // snap_at: the staged splat the snapshot is yet to be taken after
    auto state = [&](float4 (&o)[PPT]) {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            float t_[L], r_[L], g_[L], b_[L];
            v_get(T[h], t_); v_get(r[h], r_); v_get(g[h], g_); v_get(b[h], b_);
#pragma unroll
            for (int l = 0; l < L; ++l) o[L * h + l] = make_float4(t_[l], r_[l], g_[l], b_[l]);
        }
    };
    auto snapshot = [&]() {
        snap_at = -1;
        state(u);
        if (kSnapShared) {
#pragma unroll
            for (int k = 0; k < PPT; ++k) s_snap[k * (TS * TS / PPT) + threadIdx.x] = u[k];
        }
    };
    auto snapped = [&](int k) -> float4 { return kSnapShared ? s_snap[k * (TS * TS / PPT) + threadIdx.x] : u[k]; };
    if (RES) snapshot();
    auto all_done = [&]() {
        bool d = true;
#pragma unroll
        for (int k = 0; k < PPT; ++k) d = d && !(fy[k] == fy[k]);
        return __all_sync(kFull, d) != 0;
    };

    // Staged splats j .. j + G - 1 for this thread's pixels; true once all
    // pixels of the warp are done.
    auto blend = [&](auto Gc, int j) -> bool {
        constexpr int G = decltype(Gc)::value;
        float al[G][NP][L];
        int before[PPT];  // hit_last in front of this group
#pragma unroll
        for (int k = 0; k < PPT; ++k) before[k] = hit_last[k];
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const V4<V> sa = S.a[j + i], sb = S.b[j + i];
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                float y[L], oG[L];
                bool use[L];
                V py, dy;
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    y[l] = fy[L * h + l];
                    use[l] = true;
                }
                v_set(py, y);
                alphas<L, V>(fx, py, sa, sb, al[i][h], use, dy, oG);
#pragma unroll
                for (int l = 0; l < L; ++l) hit_last[L * h + l] = use[l] ? j + i : hit_last[L * h + l];
            }
        }
        V t[G + 1][NP];
        bool stop = false;
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            t[0][h] = T[h];
#pragma unroll
            for (int i = 0; i < G; ++i) {
                V a;
                v_set(a, al[i][h]);
                t[i + 1][h] = v_mul(t[i][h], v_sub(one, a));
            }
            float e[L];
            v_get(t[G][h], e);
#pragma unroll
            for (int l = 0; l < L; ++l) stop = stop || e[l] < kTMin;
        }
        const bool any_stop = __any_sync(kFull, stop);
        if (any_stop) {  // some ray ends in this group, before the splat that would take T below the floor
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                float e[L];
                v_get(t[G][h], e);
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    const int k = L * h + l;
                    fy[k] = e[l] < kTMin ? nan : fy[k];  // T never grows: the last one is below if any is
                    hit_last[k] = before[k];
                }
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    v_get(t[i + 1][h], e);
#pragma unroll
                    for (int l = 0; l < L; ++l) al[i][h][l] = e[l] < kTMin ? 0.f : al[i][h][l];
                }
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    V a;
                    v_set(a, al[i][h]);
                    t[i + 1][h] = v_mul(t[i][h], v_sub(one, a));
#pragma unroll
                    for (int l = 0; l < L; ++l)
                        hit_last[L * h + l] = al[i][h][l] > 0.f ? j + i : hit_last[L * h + l];
                }
            }
        }
        auto add = [&](int i) {
            const V4<V> sb = S.b[j + i];
            const V sblue = S.blue[j + i];
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                V a;
                v_set(a, al[i][h]);
                const V w = v_mul(a, t[i][h]);
                r[h] = v_fma(sb.z, w, r[h]);
                g[h] = v_fma(sb.w, w, g[h]);
                b[h] = v_fma(sblue, w, b[h]);
                T[h] = t[i + 1][h];
            }
        };
        if (RES && (unsigned)(snap_at - j) < (unsigned)G) {  // uniform
#pragma unroll
            for (int i = 0; i < G; ++i) {
                add(i);
                if (snap_at == j + i) snapshot();
            }
        } else {
#pragma unroll
            for (int i = 0; i < G; ++i) add(i);
        }
        return any_stop && all_done();
    };
    auto walk = [&](int &j, int to) -> bool {
        for (; j + kG <= to; j += kG)
            if (blend(IntC<kG>(), j)) return true;
        for (; j < to; ++j)
            if (blend(IntC<1>(), j)) return true;
        return false;
    };

    // The records (and freeze flags) of the next 32 entries are loaded while the
    // current ones are blended, their indices one round earlier.
    bool dead = all_done();
    uint32_t g1 = 0;
    SplatIn rec;
    rec.xa = rec.co = make_float4(0.f, 0.f, 0.f, 0.f);
    rec.blue = 0.f;
    unsigned asleep = 0;  // the entry's freeze flag, as loaded (compared only when it is staged)
    if (!dead) {
        if (lane < n) {
            const uint32_t g0 = list[lane];
            rec = splat_in(splats, g0);
            if (RES && frozen) asleep = frozen[g0];
        }
        if (lane + kStage < n) g1 = list[lane + kStage];
    }
    for (int base = 0; base < n && !dead; base += kStage) {
        const bool valid = base + lane < n;
        bool hit = valid;
        if (!kWholeTile && valid)
            hit = block_hit(rec, (float)bx, (float)(bx + 7), (float)by, (float)(by + kH - 1));
        const unsigned hits = __ballot_sync(kFull, hit);
        const unsigned wake = RES ? __ballot_sync(kFull, valid && asleep == 0) : 0u;
        const int cnt = __popc(hits);
        if (hit) {
            const int q = kWholeTile ? lane : __popc(hits & ((1u << lane) - 1u));
            stage_splat(S, q, rec);
            if (!kWholeTile) S.pos[q] = (uint8_t)lane;
        }
        if (base + kStage + lane < n) {
            rec = splat_in(splats, g1);
            if (RES && frozen) asleep = frozen[g1];
        }
        if (base + 2 * kStage + lane < n) g1 = list[base + 2 * kStage + lane];
        __syncwarp();
        const int lu = 31 - __clz(wake);  // the last unfrozen of the 32
        if (RES && wake) {
            snap_at = __popc(hits & (kFull >> (31 - lu))) - 1;
            if (snap_at < 0) snapshot();  // in front of the first staged splat
        }
        int j = 0;
        dead = walk(j, cnt);
        if (RES && wake) {
            if (snap_at >= 0) snapshot();  // every ray stopped in front of that entry: final
            upos = base + lu + 1;
        }
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
            if (hit_last[k] >= 0) last[k] = base + 1 + (kWholeTile ? hit_last[k] : (int)S.pos[hit_last[k]]);
            hit_last[k] = -1;
        }
        __syncwarp();  // the staged splats are no longer read
    }
    if (RES) {
        // A warp whose pixels were done before the splat the tile resumes behind
        // has its final state there.
        int umax = upos;
        if (kWarps > 1) {
            if (threadIdx.x == 0) s_upos = 0;
            __syncthreads();
            if (lane == 0 && upos > 0) atomicMax(&s_upos, upos);
            __syncthreads();
            umax = s_upos;
            if (upos < umax) snapshot();
        }
        if (threadIdx.x == 0) resume_pos[tile] = umax;
    }
    if (depth) {  // how far the tile's walk got: the backward takes the tiles by it
        int d = last[0];
#pragma unroll
        for (int k = 1; k < PPT; ++k) d = max(d, last[k]);
        d = __reduce_max_sync(kFull, d);
        if (lane == 0 && d > 0) atomicMax(depth + tile, d);
    }
    float4 f[PPT];
    state(f);
    const int64_t HW = (int64_t)cam.W * cam.H;
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int y = py0 + 4 * k;
        if (px < cam.W && y < cam.H) {
            const int64_t pix = (int64_t)y * cam.W + px;
            image[pix] = f[k].y + f[k].x * cam.bg[0];
            image[HW + pix] = f[k].z + f[k].x * cam.bg[1];
            image[2 * HW + pix] = f[k].w + f[k].x * cam.bg[2];
            t_final[pix] = f[k].x;
            n_last[pix] = last[k];
            if (RES) {
                const float4 v = snapped(k);
                resume[pix] = make_float4(v.x, __fsub_rn(f[k].y, v.y), __fsub_rn(f[k].z, v.z), __fsub_rn(f[k].w, v.w));
            }
        }
    }
}

// Blocks to keep resident per SM: with one pixel per thread 32 warps, which cost
// registers the step can spare (3M Gaussians at 1920x1080, 16-pixel tiles: 325 us
// against 358 without); 24 when the resume record is kept, whose state would
// spill (400K at 800x800: 97.5 us against 96.7 without, so it holds the kernel at
// what it takes anyway); with two or four the G splats in flight need them (136 us
// at 1M, 1237x822, at 103 registers).
template <int TS, int PPT, bool RES>
constexpr int fwd_blocks() {
    constexpr int warps = PPT == 1 ? (RES ? 24 : 32) : 1, per = TS * TS / PPT / 32;
    return warps / per > 1 ? warps / per : 1;
}

template <int TS, int PPT, bool RES>
__global__ void __launch_bounds__(TS * TS / PPT, fwd_blocks<TS, PPT, RES>())
    k_render_fwd(const float *__restrict__ splats, const uint32_t *__restrict__ vals, const uint32_t *__restrict__ ranges,
                 DevCam cam, float *__restrict__ image, float *__restrict__ t_final, int32_t *__restrict__ n_last,
                 const uint8_t *__restrict__ frozen, float4 *__restrict__ resume,
                 int32_t *__restrict__ resume_pos, TileOrder order, int32_t *__restrict__ depth) {
    wait_prior_grid();
    render_tile<TS, PPT, RES>(splats, vals, ranges, cam, image, t_final, n_last, ordered_tile(order), frozen, resume,
                              resume_pos, depth);
}

// Sums over a warp by recursive halving: at each xor level a lane keeps half
// of its remaining slots and adds the partner's copy of them.
__device__ __forceinline__ float keep_half(bool upper, float lo, float hi, int mask) {
    return (upper ? hi : lo) + __shfl_xor_sync(kFull, upper ? lo : hi, mask);
}

// Which of a splat's nine gradient values lane l holds after sum_columns (-1:
// none): lanes with bit 3 clear hold the six of mean, conic and opacity, split
// by bit 2 as {0-2 | 3-5} and by bits 1 and 0 as {0, 1 | 2}; lanes with bit 3
// set the colour's three.
__device__ __forceinline__ int slot_of(int lane) {
    const int q = lane & 3;
    if (q == 3 || (lane & 12) == 12) return -1;
    return (lane & 8 ? 6 : lane & 4 ? 3 : 0) + q;
}

// What the totals of slot are multiplied by: rows of grad2d hold dL/d(mean,
// conic, opacity, colour), and dpower/da = -dx^2 / 2 and so on.
__device__ __forceinline__ float grad_scale(int slot) {
    return slot == 2 || slot == 4 ? -0.5f : slot == 3 ? -1.f : 1.f;
}

// What a splat's gradient takes from its record, by the lanes that sum it.
struct SplatSum {
    float x, ha, nb, hc;  // mean's column, -a/2, -b, -c/2
};

// The sums of one splat over a block of 8 columns, from the six sums of each
// thread's own pixels: s0, s1, s2 (dL/dpower, times dy and dy^2) and the
// colour's three, held by the 16 lanes of half a warp, two rows of pixels. The
// four rows of a column share dx: the six are summed over the rows first, and
// only then turned into the moments of dx, half of the lanes with s0-s2 and half
// with the colour; the columns are summed last. Lane l gets the total of value
// slot_of(l).
__device__ __forceinline__ float sum_columns(const float (&r)[6], const SplatSum &sp, float fpx, int lane) {
    const bool h3 = lane & 8, h2 = lane & 4, h1 = lane & 2, h0 = lane & 1;
    float q[3], w[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) q[j] = keep_half(h3, r[j], r[3 + j], 8);
    // -(a mx + b s1), -(b mx + c s1), dx^2 s0 | dx s1, s2, s0
    const float dx = __fsub_rn(sp.x, fpx), mx = dx * q[0];
    const float v0 = h3 ? q[0] : fmaf(sp.ha, mx + mx, sp.nb * q[1]);
    const float v1 = h3 ? q[1] : fmaf(sp.hc, q[1] + q[1], sp.nb * mx);
    const float v2 = h3 ? q[2] : dx * mx;
    w[0] = keep_half(h2, v0, dx * q[1], 4);
    w[1] = keep_half(h2, v1, q[2], 4);
    w[2] = keep_half(h2, v2, q[0], 4);
    const float u0 = keep_half(h1, w[0], w[2], 2), u1 = w[1] + __shfl_xor_sync(kFull, w[1], 2);
    return keep_half(h0, u0, u1, 1);
}

// Two splats' sums at once: lanes 0-15 get the totals of a, lanes 16-31 those of
// b, sp being each lane's own.
__device__ __forceinline__ float sum_pair(const float (&a)[6], const float (&b)[6], const SplatSum &sp, float fpx,
                                          int lane) {
    float r[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) r[j] = keep_half(lane & 16, a[j], b[j], 16);
    return sum_columns(r, sp, fpx, lane);
}

// One splat's: both half-warps get its totals.
__device__ __forceinline__ float sum_one(const float (&a)[6], const SplatSum &sp, float fpx, int lane) {
    float r[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) r[j] = a[j] + __shfl_xor_sync(kFull, a[j], 16);
    return sum_columns(r, sp, fpx, lane);
}

// Backward state of one pixel: recovered transmittance T, dL/dC, and the
// colour blended behind the current splat with the background, kept only as
// G = dL/dC . (sum over the splats k behind it of c_k alpha_k T_k + T_final bg)
// (all dL/dalpha needs): a splat with alpha and T in front of it has dL/dalpha
// = T dL/dC . c - G / (1 - alpha), and adds dL/dC . c alpha T to G.
struct PixBwd {
    float T, dC0, dC1, dC2;
    float G;
    int nl;
};

// One (pixel, splat) step of the backward blend, skipped where the splat is not
// blended. The exponent's derivatives with respect to the 2-D mean and conic
// are dx/dy polynomials and the thread's pixels share dx, so the dy moments of
// dL/dpower are summed (g[0] += dpow, g[1] += dy dpow, g[2] += dy^2 dpow), the
// opacity's gradient in g[5], the colour's in g[6..8].
__device__ __forceinline__ bool pix_bwd(PixBwd &p, bool frz, const SplatRow &row, float dy, const float4 &co,
                                        float blue, float (&g)[9]) {
    const float power = splat_power(row, dy);
    const float G = splat_falloff(power);
    const float oG = __fmul_rn(co.y, G);
    const float alpha = fminf(kAlphaMax, oG);
    if (!(power <= 0.f && alpha >= kAlphaMin)) return false;
    const float r = rcp_ftz(1.f - alpha);
    p.T *= r;  // transmittance in front of this splat
    const float dcc = p.dC0 * co.z + p.dC1 * co.w + p.dC2 * blue;
    if (!frz) {
        const float dA = p.T * dcc - p.G * r;
        const float wT = alpha * p.T;
        g[6] += wT * p.dC0;
        g[7] += wT * p.dC1;
        g[8] += wT * p.dC2;
        if (!(oG > kAlphaMax)) {
            const float dpow = dA * oG;
            const float ydp = dy * dpow;
            g[5] += dA * G;
            g[0] += dpow;
            g[1] += ydp;
            g[2] += dy * ydp;
        }
    }
    p.G = fmaf(dcc * alpha, p.T, p.G);
    return true;
}

// The walk starts from the pixel's final state (T = T_final, nothing behind),
// or, with resume, from the state the forward recorded after the tile's last
// unfrozen splat (T there, and the colour blended behind it).
__device__ __forceinline__ void pix_load(PixBwd &p, bool inside, int64_t pix, int64_t HW, const float *t_final,
                                         const int32_t *n_last, const float *dl, const float4 *resume,
                                         const DevCam &cam) {
    p.T = 1.f; p.dC0 = p.dC1 = p.dC2 = 0.f; p.nl = 0;
    if (inside) {
        p.T = t_final[pix];
        p.nl = n_last[pix];
        p.dC0 = dl[pix];
        p.dC1 = dl[HW + pix];
        p.dC2 = dl[2 * HW + pix];
    }
    p.G = p.T * (cam.bg[0] * p.dC0 + cam.bg[1] * p.dC1 + cam.bg[2] * p.dC2);
    if (inside && resume) {
        const float4 r = resume[pix];
        p.T = r.x;
        p.G += p.dC0 * r.y + p.dC1 * r.z + p.dC2 * r.w;
    }
}

// The staged splats of a warp, one (pixel, splat) step at a time: see
// raster_bwd_tile. p[k].nl is the first staged splat of pixel k here. Not
// inlined: it is rare, and its registers would be the packed path's too.
template <int PPT, class V>
__device__ __noinline__ void scalar_steps(PixBwd *p, const Stage<V> &S, const uint32_t *gid, int cnt, unsigned fz,
                                          float fpx, float fpy0, float *grad2d) {
    const int lane = threadIdx.x & 31;
    for (int j = 0; j < cnt; ++j) {
        const float dx = __fsub_rn(v_lo(S.a[j].x), fpx), ha = v_lo(S.a[j].z), nb = v_lo(S.a[j].w), hc = v_lo(S.b[j].x);
        SplatRow row;
        row.c0 = __fmul_rn(ha, __fmul_rn(dx, dx));
        row.c1 = __fmul_rn(nb, dx);
        row.c2 = hc;
        const float4 co = make_float4(hc, v_lo(S.b[j].y), v_lo(S.b[j].z), v_lo(S.b[j].w));
        const bool frz = (fz >> j) & 1u;
        float g[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        bool c = false;
        for (int k = 0; k < PPT; ++k)
            if (j >= p[k].nl)
                c |= pix_bwd(p[k], frz, row, __fsub_rn(v_lo(S.a[j].y), fpy0 + (float)(4 * k)), co, v_lo(S.blue[j]), g);
        if (!frz && __any_sync(kFull, c)) {
            const float mx = dx * g[0];
            const float e[9] = {fmaf(ha, mx + mx, nb * g[1]), fmaf(hc, g[1] + g[1], nb * mx), dx * mx, dx * g[1], g[2],
                                g[5], g[6], g[7], g[8]};
            float tot = 0.f;  // lane l: the total of value l
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                float t = e[q];
#pragma unroll
                for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
                if (lane == q) tot = t * grad_scale(q);
            }
            if (lane < 9 && tot != 0.f) atomicAdd(grad2d + (int64_t)(gid[j] & 0x7fffffffu) * kG2d + lane, tot);
        }
    }
}

// The rasteriser backward of one tile: every warp walks its block's part of the
// list back to front (32 entries at a time, those that can reach the block, as
// in the forward), recovering T in front of each splat by a reciprocal of
// 1 - alpha. It is bound by instruction issue and, where one tile's list is
// much longer than the others', by that tile's chain of splats: two splats are
// gone through together so that their latencies overlap.
//
// An unfrozen splat needs nine sums over the block: mean's two and the conic's
// three from the moments of dL/dpower; the opacity's, which is the zeroth moment
// / opacity (dL/dpower = dL/dalpha alpha where alpha is not capped); the three of
// the colour. Two unfrozen splats are summed over the warp together, six sums of
// each over the rows first and nine over the columns (sum_columns: 15 shuffles
// for both, and the moments of dx are formed once per column; nine sums over
// all lanes took 20), and added to grad2d by the lanes that hold the totals, 18
// adds to two rows in one instruction: no shared accumulator, and per splat and
// block two sectors of atomics instead of nine scattered words.
//
// A frozen splat only moves T and G, a uniform branch.
//
// In the packed steps a pixel that does not use a splat contributes terms
// multiplied by alpha = 0, which is nothing only while they are finite, and a
// splat that no pixel uses is summed with one that is used: a block whose pixel
// state is not finite, or 32 splats with a record that is not, go through the
// scalar steps (pix_bwd), which skip.
//
// Measured against the kernel before it (a barrier-separated batch per CTA,
// scalar steps with divisions, one splat's sums at a time into a shared
// accumulator by atomics), the whole list walked and the tiles ascending: 1M
// Gaussians, 1237x822, 8-pixel tiles, two pixels per thread, nothing frozen 521 ->
// 350 us (7% more with nine sums over all lanes), 95% frozen 227 -> 168 us (one
// pixel per thread 220 -> 150 us); 400K at 800x800, 16-pixel tiles, half frozen
// 469 -> 174 us (one pixel 431 -> 176); 2K at 128x128, one pixel 77 -> 28 us.
template <int TS, int PPT>
__device__ __forceinline__ void raster_bwd_tile(const float *__restrict__ splats, const uint32_t *__restrict__ vals,
                                                const uint32_t *__restrict__ ranges, const DevCam &cam,
                                                const float *__restrict__ t_final, const int32_t *__restrict__ n_last,
                                                const float *__restrict__ dl_dimage, const uint8_t *__restrict__ frozen,
                                                float *__restrict__ grad2d, int tile,
                                                const float4 *__restrict__ resume = nullptr,
                                                const int32_t *__restrict__ resume_pos = nullptr) {
    constexpr int L = Lanes<PPT>::L, NP = Lanes<PPT>::NP;
    typedef typename ValueOf<L>::T V;
    constexpr int kWarps = TS * TS / PPT / 32, kH = 4 * PPT;
    constexpr bool kWholeTile = TS == 8 && kH == 8;
    __shared__ Stage<V> s_stage[kWarps];
    __shared__ uint32_t s_gid[kWarps][kStage];  // Gaussian index, bit 31: frozen
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Stage<V> &S = s_stage[warp];
    uint32_t *gid = s_gid[warp];
    const int bx = (tile % cam.tiles_x) * TS + (warp % (TS / 8)) * 8;
    const int by = (tile / cam.tiles_x) * TS + (warp / (TS / 8)) * kH;
    const int px = bx + (lane & 7), py0 = by + (lane >> 3);
    const uint32_t *list = vals + ranges[2 * tile];
    const int64_t HW = (int64_t)cam.W * cam.H;

    const float fpx = (float)px;
    const V fx = v_dup<V>(fpx), one = v_dup<V>(1.f);
    V T[NP], G[NP], d0[NP], d1[NP], d2[NP], fy[NP];  // G: dL/dC . (colour behind), background included
    int nl[PPT], nlmax = 0;
    bool finite = true;
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        float T_[L], G_[L], a_[L], b_[L], c_[L], y_[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const int k = L * h + l, y = py0 + 4 * k;
            PixBwd p;
            pix_load(p, px < cam.W && y < cam.H, (int64_t)y * cam.W + px, HW, t_final, n_last, dl_dimage, resume, cam);
            T_[l] = p.T; G_[l] = p.G; a_[l] = p.dC0; b_[l] = p.dC1; c_[l] = p.dC2;
            y_[l] = (float)y;
            nl[k] = p.nl;
            nlmax = max(nlmax, p.nl);
            finite = finite && isfinite(p.T) && isfinite(p.G) && isfinite(p.dC0) && isfinite(p.dC1) && isfinite(p.dC2);
        }
        v_set(T[h], T_); v_set(G[h], G_); v_set(d0[h], a_); v_set(d1[h], b_); v_set(d2[h], c_); v_set(fy[h], y_);
    }
    finite = __all_sync(kFull, finite);
    int end = __reduce_max_sync(kFull, nlmax);
    if (resume) end = min(end, resume_pos[tile]);  // the frozen splats behind the last unfrozen one are left out

    const int slot = slot_of(lane);
    const float scale = grad_scale(slot);
    float pend[6];  // the sums of an unfrozen splat that waits for a second one
    SplatSum pend_s = {};
    uint32_t pend_g = 0;
    float pend_o = 1.f;
    bool waiting = false;
    auto give = [&](float tot, uint32_t g, float o, bool holds) {
        const float v = slot == 5 ? __fdividef(tot, o) : tot * scale;
        if (holds && v != 0.f) atomicAdd(grad2d + (int64_t)g * kG2d + slot, v);
    };

    // entries in reverse: lane l takes entry bend - 1 - l, so that staged splats
    // 0, 1, ... go back to front
    uint32_t g0 = 0, g1 = 0;
    SplatIn rec;
    rec.xa = rec.co = make_float4(0.f, 0.f, 0.f, 0.f);
    rec.blue = 0.f;
    unsigned asleep = 0;
    if (lane < end) {
        g0 = list[end - 1 - lane];
        rec = splat_in(splats, g0);
        if (frozen) asleep = frozen[g0];
    }
    if (lane + kStage < end) g1 = list[end - kStage - 1 - lane];
    for (int bend = end; bend > 0; bend -= kStage) {
        const bool valid = lane < bend;
        bool hit = valid;
        if (!kWholeTile && valid)
            hit = block_hit(rec, (float)bx, (float)(bx + 7), (float)by, (float)(by + kH - 1));
        const unsigned hits = __ballot_sync(kFull, hit);
        const bool packed = finite && !__any_sync(kFull, hit && !all_finite(rec));
        const int cnt = __popc(hits);
        if (hit) {
            const int q = kWholeTile ? lane : __popc(hits & ((1u << lane) - 1u));
            // the opacity's gradient is a sum / opacity: for a splat too faint to be
            // blended anywhere the sum is 0, and so may its opacity be
            if (fabsf(rec.co.y) < 1e-3f) rec.co.y = 1e-3f;
            stage_splat(S, q, rec);
            gid[q] = g0 | (asleep ? 0x80000000u : 0u);
        }
        if (lane < bend - kStage) {
            g0 = g1;
            rec = splat_in(splats, g0);
            if (frozen) asleep = frozen[g0];
        }
        if (lane < bend - 2 * kStage) g1 = list[bend - 2 * kStage - 1 - lane];
        __syncwarp();
        // the first staged splat in front of each pixel's last contributor
        int from[PPT];
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
            const int l0 = bend - nl[k];  // entries of lanes below it lie behind
            from[k] = l0 <= 0 ? 0 : l0 >= 32 ? 32 : kWholeTile ? l0 : __popc(hits & ((1u << l0) - 1u));
        }
        const unsigned fz = __ballot_sync(kFull, lane < cnt && (gid[lane] >> 31));

        // K splats from staged j on, K = 2 where there are two: their alphas do not
        // depend on one another, T and G run through them; then the gradients of
        // the unfrozen ones, a uniform branch.
        auto steps = [&](auto Kc, int j) {
            constexpr int K = decltype(Kc)::value;
            float al[K][NP][L], oG[K][NP][L];
            V dy[K][NP], Tk[K][NP], Gk[K][NP], rk[K][NP], dk[K][NP];
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const V4<V> sa = S.a[j + i], sb = S.b[j + i];
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    bool use[L];
#pragma unroll
                    for (int l = 0; l < L; ++l) use[l] = j + i >= from[L * h + l];
                    alphas<L, V>(fx, fy[h], sa, sb, al[i][h], use, dy[i][h], oG[i][h]);
                }
            }
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const V4<V> sb = S.b[j + i];
                const V blue = S.blue[j + i];
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    V a;
                    v_set(a, al[i][h]);
                    float om[L];
                    v_get(v_sub(one, a), om);
#pragma unroll
                    for (int l = 0; l < L; ++l) om[l] = rcp_ftz(om[l]);
                    v_set(rk[i][h], om);
                    T[h] = v_mul(T[h], rk[i][h]);
                    dk[i][h] = v_fma(d2[h], blue, v_fma(d1[h], sb.w, v_mul(d0[h], sb.z)));
                    Tk[i][h] = T[h];
                    Gk[i][h] = G[h];
                    G[h] = v_fma(v_mul(dk[i][h], a), T[h], G[h]);
                }
            }
            // the six sums of splat i over this thread's pixels; false if none uses it
            auto sums = [&](int i, float (&g)[6]) -> bool {
                const V4<V> sb = S.b[j + i];
                auto total = [](V v) -> float {
                    float e[L];
                    v_get(v, e);
                    return L == 2 ? e[0] + e[L - 1] : e[0];
                };
                bool any = false;
                const bool capped = v_lo(sb.y) > kAlphaMax;  // uniform: only such a splat can be capped
                float s0 = 0.f, s1 = 0.f, s2 = 0.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    V w, ge;
                    v_set(w, al[i][h]);
                    w = v_mul(w, Tk[i][h]);
                    float e[L];
#pragma unroll
                    for (int l = 0; l < L; ++l) {
                        any = any || al[i][h][l] > 0.f;
                        e[l] = al[i][h][l];
                    }
                    if (capped) {  // no gradient through the cap
#pragma unroll
                        for (int l = 0; l < L; ++l) e[l] = oG[i][h][l] > kAlphaMax ? 0.f : e[l];
                    }
                    v_set(ge, e);
                    const V dA = v_sub(v_mul(Tk[i][h], dk[i][h]), v_mul(Gk[i][h], rk[i][h]));
                    const V dp = v_mul(dA, ge), ydp = v_mul(dy[i][h], dp);
                    s0 += total(dp);
                    s1 += total(ydp);
                    s2 += total(v_mul(dy[i][h], ydp));
                    c0 += total(v_mul(w, d0[h]));
                    c1 += total(v_mul(w, d1[h]));
                    c2 += total(v_mul(w, d2[h]));
                }
                g[0] = s0; g[1] = s1; g[2] = s2; g[3] = c0; g[4] = c1; g[5] = c2;
                return any;
            };
            auto part = [&](int i) {
                return SplatSum{v_lo(S.a[i].x), v_lo(S.a[i].z), v_lo(S.a[i].w), v_lo(S.b[i].x)};
            };
            const unsigned f = (fz >> j) & ((1u << K) - 1u);
            if (f == (1u << K) - 1u) return;  // frozen
            if (K == 2 && f == 0u) {
                float g[6], g2[6];
                bool any = sums(0, g);
                any = sums(K - 1, g2) || any;
                if (!__any_sync(kFull, any)) return;
                const int i = lane < 16 ? j : j + K - 1;
                give(sum_pair(g, g2, part(i), fpx, lane), gid[i], v_lo(S.b[i].y), slot >= 0);
                return;
            }
            float g[6];
            const int i = K == 2 && f == 1u ? K - 1 : 0;  // the unfrozen one
            const bool any = i ? sums(K - 1, g) : sums(0, g);
            if (!__any_sync(kFull, any)) return;
            const SplatSum own = part(j + i);
            const uint32_t own_g = gid[j + i];
            const float own_o = v_lo(S.b[j + i].y);
            if (waiting) {
                const bool first = lane < 16;
                const SplatSum sp{first ? pend_s.x : own.x, first ? pend_s.ha : own.ha, first ? pend_s.nb : own.nb,
                                  first ? pend_s.hc : own.hc};
                give(sum_pair(pend, g, sp, fpx, lane), first ? pend_g : own_g, first ? pend_o : own_o, slot >= 0);
            } else {
#pragma unroll
                for (int q = 0; q < 6; ++q) pend[q] = g[q];
                pend_s = own;
                pend_g = own_g;
                pend_o = own_o;
            }
            waiting = !waiting;
        };
        if (packed) {
            int j = 0;
            for (; j + 2 <= cnt; j += 2) steps(IntC<2>(), j);
            if (j < cnt) steps(IntC<1>(), j);
        } else {
            PixBwd p[PPT];
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                float e[5][L];
                v_get(T[h], e[0]); v_get(G[h], e[1]); v_get(d0[h], e[2]); v_get(d1[h], e[3]); v_get(d2[h], e[4]);
#pragma unroll
                for (int l = 0; l < L; ++l)
                    p[L * h + l] = PixBwd{e[0][l], e[2][l], e[3][l], e[4][l], e[1][l], from[L * h + l]};
            }
            scalar_steps<PPT, V>(p, S, gid, cnt, fz, fpx, (float)py0, grad2d);
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                float t_[L], g_[L];
#pragma unroll
                for (int l = 0; l < L; ++l) { t_[l] = p[L * h + l].T; g_[l] = p[L * h + l].G; }
                v_set(T[h], t_); v_set(G[h], g_);
            }
        }
        __syncwarp();  // the staged splats are no longer read
    }
    if (waiting) give(sum_one(pend, pend_s, fpx, lane), pend_g, pend_o, slot >= 0 && lane < 16);
}

// Warps to keep resident per SM: 24 with one pixel per thread (78 registers: 147
// us against 174 without the bound at 1M, 95% frozen, 177 against 199 at 400K, 79
// against 87 at 120K; few tiles would rather have the registers, 100K at 512x512 95
// against 89), 16 with two, which the kernel takes anyway (355 us against 353 at
// 1M, nothing frozen, at 111 registers and 18 warps).
template <int TS, int PPT>
constexpr int bwd_blocks() {
    constexpr int warps = PPT == 1 ? 24 : PPT == 2 ? 16 : 1, per = TS * TS / PPT / 32;
    return warps / per > 1 ? warps / per : 1;
}

template <int TS, int PPT>
__global__ void __launch_bounds__(TS * TS / PPT, bwd_blocks<TS, PPT>())
    k_raster_bwd(const float *__restrict__ splats, const uint32_t *__restrict__ vals, const uint32_t *__restrict__ ranges,
                 DevCam cam, const float *__restrict__ t_final, const int32_t *__restrict__ n_last,
                 const float *__restrict__ dl_dimage, const uint8_t *__restrict__ frozen, float *__restrict__ grad2d,
                 const float4 *__restrict__ resume, const int32_t *__restrict__ resume_pos, TileOrder order) {
    wait_prior_grid();
    raster_bwd_tile<TS, PPT>(splats, vals, ranges, cam, t_final, n_last, dl_dimage, frozen, grad2d, ordered_tile(order),
                             resume, resume_pos);
}

// ---- measurement support: the (pixel, splat) pairs the backward visits ----
// Whether splat g is blended at a pixel that is still alive: the rasteriser's decision.
__device__ __forceinline__ bool pair_blended(const float *__restrict__ splats, uint32_t g, float fpx, float fpy) {
    const float4 *r = reinterpret_cast<const float4 *>(splats + (int64_t)g * kSplat);
    const float4 xa = __ldg(r), co = __ldg(r + 1);
    const float power = splat_power(splat_row(__fsub_rn(xa.x, fpx), xa.z, xa.w, co.x), __fsub_rn(xa.y, fpy));
    const float alpha = fminf(kAlphaMax, __fmul_rn(co.y, splat_falloff(power)));
    return power <= 0.f && alpha >= kAlphaMin;
}

// Per Gaussian, the pixels of this view it is blended into (the "hits" of
// significance pruning, Sec. 3.3): one CTA per tile, one thread per pixel,
// all threads at the same list position at once, one atomic per warp and
// position with the number of its pixels that blend the splat there.
__global__ void k_hit_counts(const float *__restrict__ splats, const uint32_t *__restrict__ vals,
                             const uint32_t *__restrict__ ranges, DevCam cam, const int32_t *__restrict__ n_last,
                             uint32_t *__restrict__ hits) {
    __shared__ int s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    const int tile = blockIdx.x, TS = cam.tile;
    const int px = (tile % cam.tiles_x) * TS + (int)(threadIdx.x % TS);
    const int py = (tile / cam.tiles_x) * TS + (int)(threadIdx.x / TS);
    const bool inside = px < cam.W && py < cam.H;
    const int nl = inside ? n_last[(int64_t)py * cam.W + px] : 0;
    if (nl > 0) atomicMax(&s_max, nl);
    __syncthreads();
    const int jmax = s_max;
    const uint32_t start = ranges[2 * tile];
    const float fpx = (float)px, fpy = (float)py;
    const int lane = threadIdx.x & 31;
    for (int j = 0; j < jmax; ++j) {
        const uint32_t g = vals[start + j];
        const unsigned b = __ballot_sync(kFull, j < nl && pair_blended(splats, g, fpx, fpy));
        if (lane == 0 && b) atomicAdd(hits + g, (uint32_t)__popc(b));
    }
}

// One CTA per tile, one thread per pixel, walking the pixel's list with the
// forward's own decisions up to where the resuming backward walks it: the
// pixel's last contributor, or with a freeze map 1 + the tile's last unfrozen
// entry among those the tile's deepest contributor reaches, if that is less
// (a lower bound of the backward's walk, which goes on to the deepest
// contributor when an unfrozen entry lies behind it among the same 32 entries).
__global__ void k_pair_counts(const float *__restrict__ splats, const uint32_t *__restrict__ vals,
                              const uint32_t *__restrict__ ranges, DevCam cam, const int32_t *__restrict__ n_last,
                              const uint8_t *__restrict__ frozen, unsigned long long *__restrict__ counts) {
    __shared__ unsigned long long s_c[3];
    __shared__ int s_maxnl, s_lu;
    if (threadIdx.x < 3) s_c[threadIdx.x] = 0ull;
    if (threadIdx.x == 0) { s_maxnl = 0; s_lu = -1; }
    __syncthreads();
    const int tile = blockIdx.x, TS = cam.tile;
    const int px = (tile % cam.tiles_x) * TS + (int)(threadIdx.x % TS);
    const int py = (tile / cam.tiles_x) * TS + (int)(threadIdx.x / TS);
    const bool inside = px < cam.W && py < cam.H;
    const int nl = inside ? n_last[(int64_t)py * cam.W + px] : 0;
    const uint32_t start = ranges[2 * tile];
    if (nl > 0) atomicMax(&s_maxnl, nl);
    __syncthreads();
    if (frozen) {
        for (int j = (int)threadIdx.x; j < s_maxnl; j += (int)blockDim.x)
            if (!frozen[vals[start + j]]) atomicMax(&s_lu, j);
        __syncthreads();
    }
    const int upto = frozen ? min(nl, s_lu + 1) : nl;
    uint32_t c[3] = {0u, 0u, 0u};
    const float fpx = (float)px, fpy = (float)py;
    for (int j = 0; j < upto; ++j) {
        const uint32_t g = vals[start + j];
        if (pair_blended(splats, g, fpx, fpy))
            ++c[frozen && frozen[g] ? 1 : 0];
        else
            ++c[2];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        unsigned long long v = c[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_c[k], v);
    }
    __syncthreads();
    if (threadIdx.x < 3 && s_c[threadIdx.x]) atomicAdd(counts + threadIdx.x, s_c[threadIdx.x]);
}

// ---- many views of many scenes in one persistent launch ----
// CTAs pull (job, tile) items from a device counter until the batch is done,
// so jobs of uneven cost (scenes of different sizes) share the GPU without a
// per-job launch. Every job of a batch has the same image size and tile.
__device__ __forceinline__ int next_item(uint32_t *queue, int *s_item) {
    __syncthreads();  // every thread is done with the previous item's shared memory
    if (threadIdx.x == 0) *s_item = (int)atomicAdd(queue, 1u);
    __syncthreads();
    return *s_item;
}

__device__ uint32_t g_render_flags;

// A job whose camera does not have the batch's image size and tile would
// index its tile ranges and images with the wrong grid: it is skipped and
// GS_FLAG_BADJOB raised (uniform across the CTA: every thread reads the same job).
__device__ __forceinline__ bool job_ok(const DevCam &cam, int W, int H, int TS) {
    if (cam.W == W && cam.H == H && cam.tile == TS) return true;
    if (threadIdx.x == 0) atomicOr(&g_render_flags, GS_FLAG_BADJOB);
    return false;
}

template <int TS, int PPT>
__global__ void __launch_bounds__(TS * TS / PPT) k_render_fwd_batch(const gs_raster_job *__restrict__ jobs,
                                                                    int W, int H, int tiles_per_job, int total,
                                                                    uint32_t *__restrict__ queue) {
    __shared__ int s_item;
    for (int item = next_item(queue, &s_item); item < total; item = next_item(queue, &s_item)) {
        const gs_raster_job &j = jobs[item / tiles_per_job];
        const DevCam cam = make_cam(&j.cam);
        if (!job_ok(cam, W, H, TS)) continue;
        render_tile<TS, PPT, false>(j.splats, j.vals, j.ranges, cam, j.image, j.t_final, j.n_last,
                                    item % tiles_per_job);
    }
}

template <int TS, int PPT>
__global__ void __launch_bounds__(TS * TS / PPT) k_raster_bwd_batch(const gs_raster_job *__restrict__ jobs,
                                                                    int W, int H, int tiles_per_job, int total,
                                                                    uint32_t *__restrict__ queue) {
    __shared__ int s_item;
    for (int item = next_item(queue, &s_item); item < total; item = next_item(queue, &s_item)) {
        const gs_raster_job &j = jobs[item / tiles_per_job];
        const DevCam cam = make_cam(&j.cam);
        if (!job_ok(cam, W, H, TS)) continue;
        raster_bwd_tile<TS, PPT>(j.splats, j.vals, j.ranges, cam, j.t_final, j.n_last, j.dl_dimage, j.frozen,
                                    j.grad2d, item % tiles_per_job);
    }
}

// Launch shape used when the caller gives none: pixels per thread by tile size
// (timed on GB300; the autotuner may pick another per workload). The backward
// of 16-pixel tiles takes one pixel per thread while the tiles are few: below
// about 2048 the chip has fewer 8 x 8 blocks than warps it can hold, and halving
// the blocks shortens every chain (100K Gaussians at 512x512, 1024 tiles: 95 us
// against 112; 50K at 320x240 75 against 93); above, two per thread cost fewer
// instructions (tiles ascending, nothing frozen: 120K at 800x800, 2500 tiles 102 us
// against 104, 400K 223 against 236, 200K at 1237x822, 4056 tiles 167 against 200).
// Longest first, as a training step takes them, the line lies higher: one pixel
// is the better one at 2500 tiles (120K 85 against 97, 400K 205 against 211, half
// frozen 154 against 168), two at 4056 (155 against 189).
inline int default_ppt(int tile, int64_t tiles, bool bwd) {
    if (tile == 8) return 1;
    if (tile == 16) return bwd && tiles >= 2048 ? 2 : 1;
    return 2;
}

struct FwdArgs {
    const float *splats;
    const uint32_t *vals, *ranges;
    DevCam cam;
    float *image, *t_final;
    int32_t *n_last;
    const uint8_t *frozen;
    float4 *resume;
    int32_t *resume_pos;
    TileOrder order;
    int32_t *depth;
};

struct BwdArgs {
    const float *splats;
    const uint32_t *vals, *ranges;
    DevCam cam;
    const float *t_final;
    const int32_t *n_last;
    const float *dl;
    const uint8_t *frozen;
    float *grad2d;
    const float4 *resume;
    const int32_t *resume_pos;
    TileOrder order;
};

template <int TS, int PPT>
void launch(const FwdArgs &a, cudaStream_t s) {
    const int tiles = a.cam.tiles_x * a.cam.tiles_y;
    if (a.resume)
        launch_chained(k_render_fwd<TS, PPT, true>, tiles, TS * TS / PPT, s, a.splats, a.vals, a.ranges, a.cam, a.image,
                       a.t_final, a.n_last, a.frozen, a.resume, a.resume_pos, a.order, a.depth);
    else
        launch_chained(k_render_fwd<TS, PPT, false>, tiles, TS * TS / PPT, s, a.splats, a.vals, a.ranges, a.cam,
                       a.image, a.t_final, a.n_last, a.frozen, a.resume, a.resume_pos, a.order, a.depth);
}

template <int TS, int PPT>
void launch(const BwdArgs &a, cudaStream_t s) {
    launch_chained(k_raster_bwd<TS, PPT>, a.cam.tiles_x * a.cam.tiles_y, TS * TS / PPT, s, a.splats, a.vals, a.ranges,
                   a.cam, a.t_final, a.n_last, a.dl, a.frozen, a.grad2d, a.resume, a.resume_pos, a.order);
}

struct BatchArgs {
    const gs_raster_job *jobs;
    int W, H, tiles_per_job, total;
    uint32_t *queue;
    bool bwd;
};

template <class K>
int resident_ctas(K kernel, int threads) {
    int per_sm = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    return (sms > 0 ? sms : 152) * per_sm;
}

template <int TS, int PPT>
void launch(const BatchArgs &a, cudaStream_t s) {
    constexpr int NT = TS * TS / PPT;
    if (a.bwd) {
        const int grid = resident_ctas(k_raster_bwd_batch<TS, PPT>, NT);
        k_raster_bwd_batch<TS, PPT><<<grid, NT, 0, s>>>(a.jobs, a.W, a.H, a.tiles_per_job, a.total, a.queue);
    } else {
        const int grid = resident_ctas(k_render_fwd_batch<TS, PPT>, NT);
        k_render_fwd_batch<TS, PPT><<<grid, NT, 0, s>>>(a.jobs, a.W, a.H, a.tiles_per_job, a.total, a.queue);
    }
}

template <class A>
int dispatch(int tile, int ppt, const A &a, cudaStream_t s) {
    switch (tile * 10 + ppt) {
        case 81: launch<8, 1>(a, s); break;
        case 82: launch<8, 2>(a, s); break;
        case 161: launch<16, 1>(a, s); break;
        case 162: launch<16, 2>(a, s); break;
        case 164: launch<16, 4>(a, s); break;
        case 321: launch<32, 1>(a, s); break;
        case 324: launch<32, 4>(a, s); break;
        default: launch<32, 2>(a, s); break;
    }
    note_launches(1);
    return launch_status();
}

// Four pixels per thread only where a tile still fills whole warps (16, 32).
inline bool config_ok(const gs_raster_config *c, int tile) {
    return !c || ((c->pixels_per_thread == 1 || c->pixels_per_thread == 2 ||
                   (c->pixels_per_thread == 4 && tile >= 16)) &&
                  (c->batch == 32 || c->batch == 64 || c->batch == 128 || c->batch == 256));
}

}  // namespace
}  // namespace gs

using namespace gs;

namespace gs {
int render_fwd_ordered(const float *splats, const uint32_t *vals, const uint32_t *ranges, const gs_camera *cam,
                       const gs_raster_config *cfg, const uint8_t *frozen, float *image, float *t_final,
                       int32_t *n_last, float *resume, int32_t *resume_pos, const TileOrder &order, int32_t *depth,
                       gs_stream_t stream) {
    if (!camera_ok(cam) || !config_ok(cfg, cam->tile) || !ranges || !image || !t_final || !n_last)
        return GS_ERR_INVALID_ARG;
    if ((resume == nullptr) != (resume_pos == nullptr)) return GS_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(splats) | reinterpret_cast<uintptr_t>(resume)) & 15) return GS_ERR_INVALID_ARG;
    FwdArgs a{splats, vals, ranges, make_cam(cam), image, t_final, n_last, frozen, reinterpret_cast<float4 *>(resume),
              resume_pos, order, depth};
    const int ppt = cfg ? cfg->pixels_per_thread
                        : default_ppt(a.cam.tile, (int64_t)a.cam.tiles_x * a.cam.tiles_y, false);
    return dispatch(a.cam.tile, ppt, a, as_stream(stream));
}

int raster_bwd_ordered(const float *splats, const uint32_t *vals, const uint32_t *ranges, const gs_camera *cam,
                       const gs_raster_config *cfg, const float *t_final, const int32_t *n_last,
                       const float *dl_dimage, const uint8_t *frozen, const float *resume, const int32_t *resume_pos,
                       float *grad2d, const TileOrder &order, gs_stream_t stream) {
    if (!camera_ok(cam) || !config_ok(cfg, cam->tile) || !ranges || !t_final || !n_last || !dl_dimage || !grad2d)
        return GS_ERR_INVALID_ARG;
    if ((resume == nullptr) != (resume_pos == nullptr)) return GS_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(splats) | reinterpret_cast<uintptr_t>(resume)) & 15) return GS_ERR_INVALID_ARG;
    BwdArgs a{splats, vals, ranges, make_cam(cam), t_final, n_last, dl_dimage, frozen, grad2d,
              reinterpret_cast<const float4 *>(resume), resume_pos, order};
    const int ppt = cfg ? cfg->pixels_per_thread
                        : default_ppt(a.cam.tile, (int64_t)a.cam.tiles_x * a.cam.tiles_y, true);
    return dispatch(a.cam.tile, ppt, a, as_stream(stream));
}
}  // namespace gs

// The order in a sort's workspace, used if it is marked as this grid's.
static TileOrder order_in(const gs_camera *cam, const void *sort_ws, size_t sort_ws_bytes) {
    TileOrder o{};
    if (!sort_ws || !camera_ok(cam)) return o;
    const DevCam dc = make_cam(cam);
    const int64_t tiles = (int64_t)dc.tiles_x * dc.tiles_y;
    const SortFront f = sort_front(const_cast<void *>(sort_ws), tiles);
    if (tiles < kOrderMinTiles || sort_ws_bytes < f.bytes || (reinterpret_cast<uintptr_t>(sort_ws) & 255)) return o;
    return TileOrder{f.order, f.stamp, tile_order_key(dc.tiles_x, dc.tiles_y, dc.tile)};
}

extern "C" int gs_render_fwd_sorted(const float *splats, const uint32_t *vals, const uint32_t *ranges,
                                    const gs_camera *cam, const gs_raster_config *cfg, const uint8_t *frozen,
                                    float *image, float *t_final, int32_t *n_last, float *resume,
                                    int32_t *resume_pos, const void *sort_ws, size_t sort_ws_bytes,
                                    gs_stream_t stream) {
    return render_fwd_ordered(splats, vals, ranges, cam, cfg, frozen, image, t_final, n_last, resume, resume_pos,
                              order_in(cam, sort_ws, sort_ws_bytes), nullptr, stream);
}

extern "C" int gs_raster_bwd_sorted(const float *splats, const uint32_t *vals, const uint32_t *ranges,
                                    const gs_camera *cam, const gs_raster_config *cfg, const float *t_final,
                                    const int32_t *n_last, const float *dl_dimage, const uint8_t *frozen,
                                    const float *resume, const int32_t *resume_pos, float *grad2d,
                                    const void *sort_ws, size_t sort_ws_bytes, gs_stream_t stream) {
    return raster_bwd_ordered(splats, vals, ranges, cam, cfg, t_final, n_last, dl_dimage, frozen, resume, resume_pos,
                              grad2d, order_in(cam, sort_ws, sort_ws_bytes), stream);
}

extern "C" int gs_render_fwd_resume(const float *splats, const uint32_t *vals, const uint32_t *ranges,
                                    const gs_camera *cam, const gs_raster_config *cfg, const uint8_t *frozen,
                                    float *image, float *t_final, int32_t *n_last, float *resume,
                                    int32_t *resume_pos, gs_stream_t stream) {
    return render_fwd_ordered(splats, vals, ranges, cam, cfg, frozen, image, t_final, n_last, resume, resume_pos,
                              TileOrder{}, nullptr, stream);
}

extern "C" int gs_render_fwd_cfg(const float *splats, const uint32_t *vals, const uint32_t *ranges,
                                 const gs_camera *cam, const gs_raster_config *cfg, float *image, float *t_final,
                                 int32_t *n_last, gs_stream_t stream) {
    return gs_render_fwd_resume(splats, vals, ranges, cam, cfg, nullptr, image, t_final, n_last, nullptr, nullptr,
                                stream);
}

extern "C" int gs_render_fwd(const float *splats, const uint32_t *vals, const uint32_t *ranges, const gs_camera *cam,
                             float *image, float *t_final, int32_t *n_last, gs_stream_t stream) {
    return gs_render_fwd_cfg(splats, vals, ranges, cam, nullptr, image, t_final, n_last, stream);
}

extern "C" int gs_raster_bwd_resume(const float *splats, const uint32_t *vals, const uint32_t *ranges,
                                    const gs_camera *cam, const gs_raster_config *cfg, const float *t_final,
                                    const int32_t *n_last, const float *dl_dimage, const uint8_t *frozen,
                                    const float *resume, const int32_t *resume_pos, float *grad2d,
                                    gs_stream_t stream) {
    return raster_bwd_ordered(splats, vals, ranges, cam, cfg, t_final, n_last, dl_dimage, frozen, resume, resume_pos,
                              grad2d, TileOrder{}, stream);
}

extern "C" int gs_raster_bwd_cfg(const float *splats, const uint32_t *vals, const uint32_t *ranges,
                                 const gs_camera *cam, const gs_raster_config *cfg, const float *t_final,
                                 const int32_t *n_last, const float *dl_dimage, const uint8_t *frozen, float *grad2d,
                                 gs_stream_t stream) {
    return gs_raster_bwd_resume(splats, vals, ranges, cam, cfg, t_final, n_last, dl_dimage, frozen, nullptr, nullptr,
                                grad2d, stream);
}

extern "C" int gs_raster_bwd(const float *splats, const uint32_t *vals, const uint32_t *ranges, const gs_camera *cam,
                             const float *t_final, const int32_t *n_last, const float *dl_dimage,
                             const uint8_t *frozen, float *grad2d, gs_stream_t stream) {
    return gs_raster_bwd_cfg(splats, vals, ranges, cam, nullptr, t_final, n_last, dl_dimage, frozen, grad2d, stream);
}

static int batch_common(const gs_raster_job *jobs_dev, int32_t n_jobs, int32_t width, int32_t height, int32_t tile,
                        const gs_raster_config *cfg, uint32_t *queue_dev, gs_stream_t stream, bool bwd) {
    if (!jobs_dev || !queue_dev || n_jobs < 0 || width <= 0 || height <= 0 || !tile_ok(tile) ||
        !config_ok(cfg, tile))
        return GS_ERR_INVALID_ARG;
    if (n_jobs == 0) return GS_OK;
    const int64_t tiles = (int64_t)((width + tile - 1) / tile) * ((height + tile - 1) / tile);
    if (tiles * n_jobs > INT32_MAX) return GS_ERR_INVALID_ARG;
    cudaStream_t s = as_stream(stream);
    if (cudaMemsetAsync(queue_dev, 0, sizeof(uint32_t), s) != cudaSuccess) return GS_ERR_CUDA;
    BatchArgs a{jobs_dev, width, height, (int)tiles, (int)(tiles * n_jobs), queue_dev, bwd};
    return dispatch(tile, cfg ? cfg->pixels_per_thread : default_ppt(tile, tiles * n_jobs, bwd), a, s);
}

extern "C" int gs_render_fwd_batch(const gs_raster_job *jobs_dev, int32_t n_jobs, int32_t width, int32_t height,
                                   int32_t tile, const gs_raster_config *cfg, uint32_t *queue_dev, gs_stream_t stream) {
    return batch_common(jobs_dev, n_jobs, width, height, tile, cfg, queue_dev, stream, false);
}

extern "C" int gs_raster_bwd_batch(const gs_raster_job *jobs_dev, int32_t n_jobs, int32_t width, int32_t height,
                                   int32_t tile, const gs_raster_config *cfg, uint32_t *queue_dev, gs_stream_t stream) {
    return batch_common(jobs_dev, n_jobs, width, height, tile, cfg, queue_dev, stream, true);
}

namespace gs {
uint32_t take_render_flags() {
    uint32_t f = 0, z = 0;
    cudaMemcpyFromSymbol(&f, g_render_flags, sizeof(f));
    cudaMemcpyToSymbol(g_render_flags, &z, sizeof(z));
    return f;
}
}  // namespace gs

extern "C" int gs_raster_pair_counts(const float *splats, const uint32_t *vals, const uint32_t *ranges,
                                     const gs_camera *cam, const int32_t *n_last, const uint8_t *frozen,
                                     uint64_t *counts_dev, gs_stream_t stream) {
    if (!camera_ok(cam) || !splats || !vals || !ranges || !n_last || !counts_dev) return GS_ERR_INVALID_ARG;
    const DevCam dc = make_cam(cam);
    k_pair_counts<<<dc.tiles_x * dc.tiles_y, dc.tile * dc.tile, 0, as_stream(stream)>>>(
        splats, vals, ranges, dc, n_last, frozen, reinterpret_cast<unsigned long long *>(counts_dev));
    note_launches(1);
    return launch_status();
}

extern "C" int gs_hit_counts(const float *splats, const uint32_t *vals, const uint32_t *ranges, const gs_camera *cam,
                             const int32_t *n_last, uint32_t *hits_dev, gs_stream_t stream) {
    if (!camera_ok(cam) || !splats || !vals || !ranges || !n_last || !hits_dev) return GS_ERR_INVALID_ARG;
    const DevCam dc = make_cam(cam);
    k_hit_counts<<<dc.tiles_x * dc.tiles_y, dc.tile * dc.tile, 0, as_stream(stream)>>>(splats, vals, ranges, dc,
                                                                                      n_last, hits_dev);
    note_launches(1);
    return launch_status();
}
