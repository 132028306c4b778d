// Multi-attribute compute rasterizer (Sec. 3.2): clear, render (visibility) and
// resolve passes, plus packing of the G-buffer into the network input.
//
// Render pass: every point is read once for all views of the batch and
// projected with a fixed FP32 operation sequence written with explicit
// round-to-nearest intrinsics, so no compiler contraction can change a bit:
//   c_r = ((m_r0*x + m_r1*y) + m_r2*z) + m_r3   for rows r = 0, 1, 3
//   keep if znear <= w <= zfar;  ndc = c.xy / w  (IEEE division)
//   sx = (ndc.x + 1) * W/2,  sy = (1 - ndc.y) * H/2,  keep if on screen.
// The per-pixel winner is the minimum of the 64-bit key (bits(w) << 32 | i):
// w > 0 so its bits order like its value, and equal depths go to the lowest
// index.  An early depth test (Sec. 3.2, "early z-buffer testing") reads the
// current key from L2 first and issues the atomic only when the point is in
// front of it; keys only ever decrease, so a stale read only costs an atomic.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <utility>

#include "internal.h"
#include "project.cuh"

namespace nrv {

// Programmatic dependent launch inside the render and resolve passes (unless NRV_PDL=0): each
// of their kernels is launched while the previous one drains and waits (griddepcontrol.wait)
// for it to complete before reading anything it wrote.  The clear before them is a plain launch
// that lets the next one start at once, so what a kernel reads ahead of its wait (positions, the
// table of views) was complete before the clear began.  Both instructions do nothing for a plain
// launch.
__device__ __forceinline__ void pdl_wait_and_release() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
static bool render_pdl() {
    static int on = -1;
    if (on < 0) {
        const char* e = getenv("NRV_PDL");
        on = (e && e[0] == '0') ? 0 : 1;
    }
    return on == 1;
}
template <typename... KArgs, typename... Args>
static nrv_status launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, cudaStream_t s,
                             Args&&... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = render_pdl() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    NRV_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

__global__ void clear_keys_kernel(RViews vs) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int v = blockIdx.y;
    if (v >= vs.n) return;
    const uint64_t npx = (uint64_t)vs.v[v].width * vs.v[v].height;
    ulonglong2* k2 = reinterpret_cast<ulonglong2*>(vs.v[v].key);
    const ulonglong2 e = make_ulonglong2(~0ull, ~0ull);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < npx / 2;
         i += (uint64_t)gridDim.x * blockDim.x)
        k2[i] = e;
    if ((npx & 1) && blockIdx.x == 0 && threadIdx.x == 0) vs.v[v].key[npx - 1] = ~0ull;
}

nrv_status launch_clear_keys(const RViews& views, cudaStream_t s) {
    dim3 grid(4 * 152, views.n);
    clear_keys_kernel<<<grid, 256, 0, s>>>(views);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

// Tiles of the chunk-culling variants: TILE x TILE pixels; bound[t] holds the largest
// depth word (key >> 32) over the tile's pixels after a first pass over a
// subset of the points.  Keys only decrease afterwards, so a point whose depth
// word exceeds its tile's bound can never win there.
constexpr int TILE = 16;

// The bounds of one view form a pyramid: level 0 one word per tile, level l (up to
// HIZ_LEVELS - 1) one word per 2^l x 2^l level-0 tiles (the maximum over those that exist),
// level after level; the views' pyramids lie back to back.  A box test reads the level at
// which the box's tile range spans at most 2 x 2 words.
constexpr int HIZ_LEVELS = 4;
struct TileDims {
    int off[HIZ_LEVELS];   // word offset of each level in the view's pyramid (off[0] = 0)
    int w0, h0;            // level-0 tiles per row and rows
    int words;             // words of the pyramid
};
__host__ __device__ inline TileDims tile_dims(int width, int height) {
    TileDims d;
    d.w0 = (width + TILE - 1) / TILE;
    d.h0 = (height + TILE - 1) / TILE;
    int off = 0;
    for (int l = 0; l < HIZ_LEVELS; ++l) {
        d.off[l] = off;
        off += (((d.w0 - 1) >> l) + 1) * (((d.h0 - 1) >> l) + 1);
    }
    d.words = off;
    return d;
}

// Projection, clipping, early depth test and atomic of one point for one view, by the scalar
// sequence.
__device__ __forceinline__ void render_point(const RView& v, float x, float y, float z,
                                             uint32_t idx) {
    const float cw = __fadd_rn(
        __fadd_rn(__fadd_rn(__fmul_rn(v.m[8], x), __fmul_rn(v.m[9], y)), __fmul_rn(v.m[10], z)),
        v.m[11]);
    if (!(cw >= v.znear && cw <= v.zfar)) return;
    const float cx = __fadd_rn(
        __fadd_rn(__fadd_rn(__fmul_rn(v.m[0], x), __fmul_rn(v.m[1], y)), __fmul_rn(v.m[2], z)),
        v.m[3]);
    const float cy = __fadd_rn(
        __fadd_rn(__fadd_rn(__fmul_rn(v.m[4], x), __fmul_rn(v.m[5], y)), __fmul_rn(v.m[6], z)),
        v.m[7]);
    const float sx = __fmul_rn(__fadd_rn(__fdiv_rn(cx, cw), 1.0f), v.hw);
    const float sy = __fmul_rn(__fsub_rn(1.0f, __fdiv_rn(cy, cw)), v.hh);
    if (!(sx >= 0.0f && sx < v.fw && sy >= 0.0f && sy < v.fh)) return;
    const int px = __float2int_rz(sx), py = __float2int_rz(sy);
    const unsigned long long key = ((unsigned long long)__float_as_uint(cw) << 32) | idx;
    unsigned long long* p = v.key + (size_t)py * v.width + px;
    if (key < __ldcg(p)) atomicMin(p, key);
}

// A point whose depth lies inside the view's range but outside project4's (depths below
// 2^-60 or above 2^125; views with such ranges only).
__device__ __noinline__ void render_point_wide(const RView& v, float x, float y, float z,
                                               uint32_t idx) {
    const float cw = __fadd_rn(
        __fadd_rn(__fadd_rn(__fmul_rn(v.m[8], x), __fmul_rn(v.m[9], y)), __fmul_rn(v.m[10], z)),
        v.m[11]);
    const uint32_t b = __float_as_uint(cw);
    if (b >= FAST_W_LO && b <= FAST_W_HI) return;
    render_point(v, x, y, z, idx);
}

// The points of a group that project4 leaves to the wide path.  Few scenes have one, however wide
// the view's range (an unbounded far plane is common), so the four depths come first, two by two
// and by project4's sequence; f: the same view in shared memory.  Kept out of render_view: a mask
// returned from there cost the bounded views 1 to 4%.  Terrain, 9M points, eight views of 960 x
// 540: 291 us with the plain division of every point, 233 here, 221 with a bounded range.
__device__ __forceinline__ void render_wide4(const FView& f, const RView& v, const f2* X, const f2* Y,
                                             const f2* Z, const uint32_t* idx, uint32_t in) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const f2 xy = f2_fma(f2_mul(f.m[9], Y[h]), f.one, f2_mul(f.m[8], X[h]));
        float w[2];
        f2_unpack(f2_add(f2_fma(f2_mul(f.m[10], Z[h]), f.one, xy), f.m[11]), w[0], w[1]);
        // bits order like the values of non-negative floats; negative ones and NaN are above infinity
        auto fast = [](float d) {
            const uint32_t b = __float_as_uint(d);
            return b - FAST_W_LO <= FAST_W_HI - FAST_W_LO || b > 0x7F800000u;
        };
        if (fast(w[0]) && fast(w[1])) continue;
        float x[2], y[2], z[2];
        f2_unpack(X[h], x[0], x[1]);
        f2_unpack(Y[h], y[0], y[1]);
        f2_unpack(Z[h], z[0], z[1]);
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if ((in >> (2 * h + e)) & 1u) render_point_wide(v, x[e], y[e], z[e], idx[2 * h + e]);
    }
}

// Four points of one view: project, read the depth words of their pixels together (keys only
// decrease: a point strictly behind that word cannot win), then the atomics still needed.
// in: bit j set where point j is present; idx: its key's low word.  MERGE (ascending idx, points
// next to one another in the scene): a run of points in one pixel leaves only its nearest, the
// lowest index among equals -- about a third of the points of a dense scan are left to read
// the key image and fewer still to write it.
template <bool MERGE>
__device__ __forceinline__ void render_view(const FView& v, const f2* X, const f2* Y, const f2* Z,
                                            const uint32_t* idx_in, uint32_t in) {
    uint32_t pix[4], db[4], cur[4], idx[4];
    bool ok[4];
    project4(v, X, Y, Z, pix, db, ok);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        idx[j] = idx_in[j];
        ok[j] = ok[j] & ((in >> j) & 1u);
    }
    if (MERGE) {
#pragma unroll
        for (int j = 1; j < 4; ++j) {
            const bool same = ok[j] & ok[j - 1] & (pix[j] == pix[j - 1]);
            const bool prev = same & (db[j - 1] <= db[j]);
            ok[j - 1] = ok[j - 1] & !same;
            db[j] = prev ? db[j - 1] : db[j];
            idx[j] = prev ? idx[j - 1] : idx[j];
        }
    }
    // predicated, not branched around: a branch per point and its reconvergence cost a tenth of
    // the pass's instructions
#pragma unroll
    for (int j = 0; j < 4; ++j)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %2, 0;\n\t"
            "mov.u32 %0, 0;\n\t"
            "@p ld.global.cg.u32 %0, [%1+4];\n\t}"
            : "=r"(cur[j])
            : "l"(v.key + pix[j]), "r"((uint32_t)ok[j])
            : "memory");
#pragma unroll
    for (int j = 0; j < 4; ++j)
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.ne.u32 q, %4, 0;\n\t"
            "setp.le.and.u32 p, %1, %3, q;\n\t"
            "@p red.relaxed.gpu.global.min.u64 [%0], %2;\n\t}" ::"l"(v.key + pix[j]),
            "r"(db[j]), "l"(((unsigned long long)db[j] << 32) | idx[j]), "r"(cur[j]), "r"((uint32_t)ok[j])
            : "memory");
}

// One thread handles 4 consecutive points (48 bytes, three 16-byte loads).  Per view they are
// projected first and their early-depth reads issued together.
// The views come by value, or -- when a captured frame is replayed with new cameras -- from
// device memory (views_dev); each block keeps them in shared memory, and a thread copies one
// view at a time into registers (read per use, the views made 40% of the pass's shared/L1
// wavefronts).
// Variants (picked per scene by the launcher's timing, see below):
//   SINGLE   one view, kept in registers for the whole pass;
//   PREFETCH the next group's coordinates are loaded before this group is done;
//   MINB     register budget: at least MINB blocks of 256 threads per SM.
// A block works through `span` consecutive groups: scenes are stored along scan lines, particle
// paths or cells, so neighbours in the array share pixels.  Strided over the whole grid, the
// 0.5M points in flight were neighbours and most saw their pixel still empty, every one an
// atomic; in one block the next 1024 points see what the last ones wrote.
// Eight-view terrain of 200M points: 4.39 ms with project4 alone (4.85 with the scalar
// sequence), 3.68 with runs of points in a pixel merged, 3.53 with the views' register copies,
// 3.27 with contiguous spans, 2.93 with the predicated reads and atomics and a reciprocal without
// subnormal handling.  It is then bound by issue and by the sectors of its
// key reads and atomics (0.36 per point and view) about equally; eight points per thread
// measured slower (3.43 at three blocks per SM with spills, 3.87 at two).
// Indices are 32-bit: N < 2^32, so there are fewer than 2^30 groups.
template <bool SINGLE, bool PREFETCH, int MINB>
__global__ void __launch_bounds__(256, MINB) visibility_kernel(const float4* __restrict__ xyz4,
                                                               uint32_t ngroups,
                                                               const float* __restrict__ xyz,
                                                               uint64_t n,
                                                               const __grid_constant__ RViews vs_arg,
                                                               const RViews* __restrict__ views_dev,
                                                               uint32_t span) {
    __shared__ RViews vs;
    __shared__ FView fs[SINGLE ? 1 : 8];
    {
        // the views: a word-wise copy into shared memory (no local copy of the parameter)
        const uint32_t* src = reinterpret_cast<const uint32_t*>(views_dev ? views_dev : &vs_arg);
        for (int i = threadIdx.x; i < (int)(sizeof(RViews) / 4); i += blockDim.x)
            reinterpret_cast<uint32_t*>(&vs)[i] = src[i];
    }
    __syncthreads();
    const int nv = SINGLE ? 1 : vs.n;
    if (threadIdx.x < nv) fview_init(fs[threadIdx.x], vs.v[threadIdx.x]);
    __syncthreads();
    FView f0;
    if (SINGLE) f0 = fs[0];
    // this block's contiguous run of groups
    const uint32_t g0 = blockIdx.x * span, g1 = g0 + span < ngroups ? g0 + span : ngroups;
    uint32_t g = g0 + threadIdx.x;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a, c = a;
    auto load = [&](uint32_t gq, float4& p, float4& r, float4& t) {
        if (gq < g1) {
            p = __ldcs(xyz4 + 3 * gq);
            r = __ldcs(xyz4 + 3 * gq + 1);
            t = __ldcs(xyz4 + 3 * gq + 2);
        }
    };
    if (PREFETCH) load(g, a, b, c);
    pdl_wait_and_release();   // the cleared key images
    for (; g < g1; g += blockDim.x) {
        float4 na = a, nb = b, nc = c;
        if (PREFETCH) load(g + blockDim.x, na, nb, nc);
        else load(g, a, b, c);
        const f2 X[2] = {f2_pack(a.x, a.w), f2_pack(b.z, c.y)};
        const f2 Y[2] = {f2_pack(a.y, b.x), f2_pack(b.w, c.z)};
        const f2 Z[2] = {f2_pack(a.z, b.y), f2_pack(c.x, c.w)};
        const uint32_t i0 = 4 * g + vs.base;
        const uint32_t idx[4] = {i0, i0 + 1, i0 + 2, i0 + 3};
#pragma unroll 1
        for (int v = 0; v < nv; ++v) {
            FView fv;
            if (!SINGLE) fv = fs[v];
            render_view<true>(SINGLE ? f0 : fv, X, Y, Z, idx, 15u);
            if (fs[v].wide) render_wide4(fs[v], vs.v[v], X, Y, Z, idx, 15u);
        }
        if (PREFETCH) {
            a = na;
            b = nb;
            c = nc;
        }
    }
    // the last n mod 4 points
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) {
        const uint64_t i = 4 * (uint64_t)ngroups + threadIdx.x;
        for (int v = 0; v < nv; ++v)
            render_point(vs.v[v], xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], (uint32_t)i + vs.base);
    }
}

// Render pass over a strided subset (a masked pass, e.g. over glyph points): scene point j is
// array point j * S, its key carries j * S + base.  One point per thread, the exact projection
// and the early depth test of the full pass, no culling (the subset is sparse).
__global__ void __launch_bounds__(256) visibility_strided_kernel(const float* __restrict__ xyz,
                                                                 uint64_t n, uint32_t S,
                                                                 const __grid_constant__ RViews vs_arg,
                                                                 const RViews* __restrict__ views_dev) {
    __shared__ RViews vs;
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(views_dev ? views_dev : &vs_arg);
        for (int i = threadIdx.x; i < (int)(sizeof(RViews) / 4); i += blockDim.x)
            reinterpret_cast<uint32_t*>(&vs)[i] = src[i];
    }
    __syncthreads();
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n;
         j += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t i = j * S;
        const float x = __ldg(xyz + 3 * i), y = __ldg(xyz + 3 * i + 1), z = __ldg(xyz + 3 * i + 2);
        for (int v = 0; v < vs.n; ++v) render_point(vs.v[v], x, y, z, (uint32_t)i + vs.base);
    }
}

nrv_status launch_visibility_strided(const float* xyz, uint64_t n, int stride, const RViews& views,
                                     cudaStream_t s, const RViews* views_dev) {
    if (n == 0) return NRV_OK;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    visibility_strided_kernel<<<(unsigned)blocks, 256, 0, s>>>(xyz, n, (uint32_t)stride, views,
                                                               views_dev);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

// Tile bounds: one warp per tile takes the maximum depth word over its pixels
// (empty pixels hold ~0, so a tile with an empty pixel never culls).
__global__ void tile_bound_kernel(RViews vs_arg, const RViews* __restrict__ views_dev,
                                  uint32_t* __restrict__ bound) {
    pdl_wait_and_release();
    const RViews& vs = views_dev ? *views_dev : vs_arg;
    int t = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) / 32);
    const int lane = threadIdx.x & 31;
    int v = 0;
    uint32_t* out = bound;
    for (; v < vs.n; ++v) {
        const TileDims d = tile_dims(vs.v[v].width, vs.v[v].height);
        if (t < d.w0 * d.h0) break;
        t -= d.w0 * d.h0;
        out += d.words;
    }
    if (v >= vs.n) return;    // whole warps leave together
    const RView& vw = vs.v[v];
    const int tx = (vw.width + TILE - 1) / TILE;
    // a load of the warp covers 32 / TILE whole rows of the tile: each 32-byte sector once (0.8M
    // sectors for a 1080p image against 2.1M with two lanes to a row)
    constexpr int RPL = 32 / TILE;
    const int x = (t % tx) * TILE + lane % TILE, y0 = (t / tx) * TILE + lane / TILE;
    const uint32_t* depth = reinterpret_cast<const uint32_t*>(vw.key) + 1;
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < TILE; k += RPL)
        if (x < vw.width && y0 + k < vw.height)
            m = max(m, __ldcg(depth + 2 * ((size_t)(y0 + k) * vw.width + x)));
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) out[t] = m;
}

// Levels 1.. of the bound pyramids: one warp per word, its lanes taking the maximum over the
// word's level-0 tiles.
__global__ void tile_pyramid_kernel(RViews vs_arg, const RViews* __restrict__ views_dev,
                                    uint32_t* __restrict__ bound) {
    pdl_wait_and_release();
    const RViews& vs = views_dev ? *views_dev : vs_arg;
    int t = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) / 32);
    const int lane = threadIdx.x & 31;
    uint32_t* pyr = bound;
    for (int v = 0; v < vs.n; ++v) {
        const TileDims d = tile_dims(vs.v[v].width, vs.v[v].height);
        const int coarse = d.words - d.off[1];
        if (t < coarse) {
            int l = 1, lo = 0;
            for (int k = 2; k < HIZ_LEVELS; ++k)
                if (t >= d.off[k] - d.off[1]) {
                    l = k;
                    lo = d.off[k] - d.off[1];
                }
            const int i = t - lo;
            const int wl = ((d.w0 - 1) >> l) + 1;
            const int x0 = (i % wl) << l, y0 = (i / wl) << l;
            const int nx = min(x0 + (1 << l), d.w0) - x0, ny = min(y0 + (1 << l), d.h0) - y0;
            uint32_t m = 0;
            for (int q = lane; q < nx * ny; q += 32) m = max(m, pyr[(y0 + q / nx) * d.w0 + x0 + q % nx]);
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) pyr[d.off[1] + t] = m;
            return;      // whole warps leave together
        }
        t -= coarse;
        pyr += d.words;
    }
}

static void tile_counts(const RViews& views, size_t& level0, size_t& coarse) {
    level0 = coarse = 0;
    for (int v = 0; v < views.n; ++v) {
        const TileDims d = tile_dims(views.v[v].width, views.v[v].height);
        level0 += (size_t)d.w0 * d.h0;
        coarse += (size_t)(d.words - d.off[1]);
    }
}

// Tile bounds of every view (level 0), and with hiz the levels above it.
static nrv_status launch_tile_bounds(const RViews& views, const RViews* views_dev, uint32_t* tiles,
                                     bool hiz, cudaStream_t s) {
    size_t level0, coarse;
    tile_counts(views, level0, coarse);
    NRV_TRY(launch_pdl(tile_bound_kernel, dim3((unsigned)((level0 * 32 + 255) / 256)), dim3(256), s,
                       views, views_dev, tiles));
    if (hiz)
        NRV_TRY(launch_pdl(tile_pyramid_kernel, dim3((unsigned)((coarse * 32 + 255) / 256)), dim3(256),
                           s, views, views_dev, tiles));
    return NRV_OK;
}

// ------------------------------------------------------------------ chunk culling
// The points are taken in chunks of 32 consecutive points, each with a bounding
// box (centre and half extents) computed from the positions once per scene.  A
// chunk-culling render pass renders every S-th chunk in full, turns the keys
// into tile depth bounds, then tests every other chunk's box against them, view
// by view (in one or two parts, the bounds rebuilt before the second): a chunk wholly outside the depth range or the screen, or whose
// nearest possible depth lies behind every pixel of the tiles it can touch, is
// skipped; the others render point by point.  Keys do not change: a skipped
// point could not have set one (keys only decrease, so a bound read earlier
// stays a valid bound).

// Box of a chunk or sub-chunk: centre c = (lo + hi) / 2 and half extents
// e >= max(hi - c, c - lo), the differences rounded up, so |p - c| <= e holds
// exactly for every point p.  Stored as 6 floats: cx cy cz ex ey ez; the chunk
// boxes first, then the sub-chunk boxes (sub-chunk s of chunk c at 4c + s).
// One warp per chunk: the minimum and maximum over each group of 8 lanes give
// the sub-chunk boxes, over all 32 lanes the chunk box.
__global__ void chunk_bounds_kernel(const float* __restrict__ xyz, uint64_t n,
                                    float* __restrict__ out) {
    const int lane = threadIdx.x & 31, sub = lane / RENDER_SUB, sl = lane % RENDER_SUB;
    const uint64_t nch = chunk_count(n);
    float* const out_sub = out + 6 * nch;
    const uint64_t warps = (gridDim.x * (uint64_t)blockDim.x) / 32;
    for (uint64_t c = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) / 32; c < nch; c += warps) {
        const uint64_t i0 = c * RENDER_CHUNK;
        const uint64_t i = i0 + lane < n ? i0 + lane : i0;   // lanes past the end repeat the first point
        float v[3] = {xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2]};
        float* const sb = out_sub + 6 * (RENDER_SUBS * c + sub);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            float lo = v[d], hi = v[d];
            for (int o = 1; o < 32; o <<= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                if (o == RENDER_SUB / 2) {
                    // lo, hi: this lane's sub-chunk
                    const float ctr = 0.5f * lo + 0.5f * hi;
                    const float e = fmaxf(__fsub_ru(hi, ctr), __fsub_ru(ctr, lo));
                    if (sl == d) sb[d] = ctr;
                    if (sl == 3 + d) sb[3 + d] = e;
                }
            }
            const float ctr = 0.5f * lo + 0.5f * hi;
            const float e = fmaxf(__fsub_ru(hi, ctr), __fsub_ru(ctr, lo));
            if (lane == d) out[6 * c + d] = ctr;
            if (lane == 3 + d) out[6 * c + 3 + d] = e;
        }
    }
}

nrv_status launch_chunk_bounds(const float* xyz, uint64_t n, void* chunks, cudaStream_t s) {
    if (n == 0) return NRV_OK;
    uint64_t blocks = (chunk_count(n) * 32 + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    chunk_bounds_kernel<<<(unsigned)blocks, 256, 0, s>>>(xyz, n, (float*)chunks);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

constexpr uint32_t RENDER_RUN = 8;   // chunk groups (1024 points each) per run of the culled pass: one per warp

// True when no point in the box (c, e) can set a key of view v, given the tile
// depth bounds (null: depth range and screen only; HIZ: the view's bound pyramid,
// read at one level, else its level-0 tiles).  Allowances: 1e-5 of the
// magnitudes summed in each clip coordinate covers the rounding of the points'
// own FP32 sequences and of this arithmetic (both below 1e-6 of that sum); the
// screen rectangle is widened by half a pixel plus 1e-5 of its extent.
template <bool HIZ>
__device__ __forceinline__ bool chunk_hidden(const RView& v, const float* c, const float* e,
                                             const uint32_t* __restrict__ bound, const TileDims& td) {
    const int tiles_x = td.w0, tiles_y = td.h0;
    const float ax = fabsf(c[0]) + e[0], ay = fabsf(c[1]) + e[1], az = fabsf(c[2]) + e[2];
    const float w = fmaf(v.m[8], c[0], fmaf(v.m[9], c[1], fmaf(v.m[10], c[2], v.m[11])));
    const float X = fmaf(v.m[0], c[0], fmaf(v.m[1], c[1], fmaf(v.m[2], c[2], v.m[3])));
    const float Y = fmaf(v.m[4], c[0], fmaf(v.m[5], c[1], fmaf(v.m[6], c[2], v.m[7])));
    // |row . (p - c)| <= |row| . e over the box, plus the allowance
    auto spread = [&](int r, float& allow) {
        const float* m = v.m + 4 * r;
        allow = 1e-5f * (fabsf(m[0]) * ax + fabsf(m[1]) * ay + fabsf(m[2]) * az + fabsf(m[3]));
        return fabsf(m[0]) * e[0] + fabsf(m[1]) * e[1] + fabsf(m[2]) * e[2];
    };
    float ew, ex, ey;
    const float dw = spread(2, ew) + ew;
    const float wlo = w - dw, whi = w + dw;
    if (whi < v.znear || wlo > v.zfar) return true;           // wholly outside the depth range
    if (!(wlo > 0.5f * v.znear)) return false;                // w may come near 0: no screen bound
    const float dx = spread(0, ex) + ex, dy = spread(1, ey) + ey;
    const float xl = X - dx, xh = X + dx, yl = Y - dy, yh = Y + dy;
    // 0 < wlo <= w <= whi over the box: the smallest quotient x / w is x / whi for x >= 0 and
    // x / wlo otherwise (the largest the other way round); fast reciprocals, whose error the
    // margins below cover
    const float rlo = __fdividef(1.0f, wlo), rhi = __fdividef(1.0f, whi);
    const float nxl = xl * (xl >= 0.0f ? rhi : rlo), nxh = xh * (xh >= 0.0f ? rlo : rhi);
    const float nyl = yl * (yl >= 0.0f ? rhi : rlo), nyh = yh * (yh >= 0.0f ? rlo : rhi);
    const float mx = 0.5f + 1e-5f * v.hw * (fabsf(nxl) + fabsf(nxh) + 2.0f);
    const float my = 0.5f + 1e-5f * v.hh * (fabsf(nyl) + fabsf(nyh) + 2.0f);
    const float sx0 = (nxl + 1.0f) * v.hw - mx, sx1 = (nxh + 1.0f) * v.hw + mx;
    const float sy0 = (1.0f - nyh) * v.hh - my, sy1 = (1.0f - nyl) * v.hh + my;
    if (!(sx1 >= 0.0f && sy1 >= 0.0f && sx0 < v.fw && sy0 < v.fh)) {
        // wholly off screen -- unless a NaN made every comparison fail
        return sx1 < 0.0f || sy1 < 0.0f || sx0 >= v.fw || sy0 >= v.fh;
    }
    if (!bound) return false;
    const int tx0 = sx0 > 0.0f ? (int)(sx0 * (1.0f / TILE)) : 0;
    const int ty0 = sy0 > 0.0f ? (int)(sy0 * (1.0f / TILE)) : 0;
    const int tx1 = sx1 < v.fw ? (int)(sx1 * (1.0f / TILE)) : tiles_x - 1;
    const int ty1 = sy1 < v.fh ? (int)(sy1 * (1.0f / TILE)) : tiles_y - 1;
    uint32_t m = 0;
    if (HIZ) {
        // the lowest pyramid level at which the tile range spans at most 2 x 2 words
        int l = 0;
        while ((tx1 >> l) - (tx0 >> l) > 1 || (ty1 >> l) - (ty0 >> l) > 1)
            if (++l == HIZ_LEVELS) return false;                  // wider still: not tested
        const int off = l == 0 ? 0 : l == 1 ? td.off[1] : l == 2 ? td.off[2] : td.off[3];
        const int wl = ((tiles_x - 1) >> l) + 1;
        const uint32_t* b = bound + off;
        const int x0 = tx0 >> l, x1 = tx1 >> l, r0 = (ty0 >> l) * wl, r1 = (ty1 >> l) * wl;
        m = max(max(__ldg(b + r0 + x0), __ldg(b + r0 + x1)), max(__ldg(b + r1 + x0), __ldg(b + r1 + x1)));
    } else {
        if (tx1 - tx0 >= 8 || ty1 - ty0 >= 8) return false;    // larger than 8 x 8 tiles: not tested
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx) m = max(m, __ldg(bound + ty * tiles_x + tx));
    }
    // an empty pixel leaves the bound at 0xFFFFFFFF (a NaN): never hidden
    return wlo > __uint_as_float(m);
}

// Chunk-culling render pass (SINGLE: one view, its parameters held in registers rather than
// read from shared memory for every point).  S is a power of two.  prepass != 0: chunks 0, S,
// 2S, ... in full, four per warp step, one point of each per lane.  prepass == 0: every other
// chunk of the groups [g_begin, g_end), 32 chunks per warp step -- each lane tests one chunk
// against every view and the survivors join the warp's queue in shared memory; whenever four
// are queued the
// warp renders them (each lane takes one point of each, so four early depth
// reads are in flight per lane).  Rendering only full groups of four keeps the
// lanes busy: a group costs the same instructions however many chunks it holds.
// SUB: the surviving chunks are tested again, eight at a time, by their 8-point
// sub-chunk boxes (one per lane); the surviving sub-chunks join a second queue
// and render sixteen at a time (each lane takes one point of four of them).
// HIZ: box tests read the bound pyramid (at most four words) instead of every
// level-0 tile the box reaches.
template <bool SINGLE, bool SUB, bool HIZ>
__global__ void __launch_bounds__(256, 4) chunk_render_kernel(const float* __restrict__ xyz, uint64_t n,
                                                           const float* __restrict__ chunks,
                                                           const __grid_constant__ RViews vs_arg,
                                                           const RViews* __restrict__ views_dev,
                                                           const uint32_t* __restrict__ bound,
                                                           int prepass, uint32_t S, uint32_t r_begin,
                                                           uint32_t r_end, uint32_t run_step,
                                                           uint32_t nruns) {
    pdl_wait_and_release();
    __shared__ RViews vs;
    __shared__ FView fs[SINGLE ? 1 : 8];
    __shared__ int tile_off[8];
    __shared__ TileDims tdim[8];
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(views_dev ? views_dev : &vs_arg);
        for (int i = threadIdx.x; i < (int)(sizeof(RViews) / 4); i += blockDim.x)
            reinterpret_cast<uint32_t*>(&vs)[i] = src[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int off = 0;
        for (int v = 0; v < vs.n; ++v) {
            tdim[v] = tile_dims(vs.v[v].width, vs.v[v].height);
            tile_off[v] = off;
            off += tdim[v].words;
        }
    }
    if (threadIdx.x < vs.n) fview_init(fs[threadIdx.x], vs.v[threadIdx.x]);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t nch = (uint32_t)chunk_count(n);
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) / 32;
    const uint32_t nwarps = (gridDim.x * blockDim.x) / 32;
    const uint32_t all = (1u << vs.n) - 1u;
    // one view: its parameters live in registers for the whole pass
    RView vreg;
    FView freg;
    TileDims treg;
    if (SINGLE) {
        freg = fs[0];
        vreg = vs.v[0];
        treg = tdim[0];
    }
    // the views of mask vm in which the box (c, e) may set a key
    auto box_visible = [&](const float* c, const float* e, uint32_t vm) -> uint32_t {
        if (SINGLE) {
            // the matrix: the low halves of the paired registers
            float dup;
#pragma unroll
            for (int i = 0; i < 12; ++i) f2_unpack(freg.m[i], vreg.m[i], dup);
        }
        if (SINGLE) return chunk_hidden<HIZ>(vreg, c, e, bound, treg) ? 0u : 1u;
        uint32_t vis = 0;
        for (int v = 0; v < vs.n; ++v)
            if (((vm >> v) & 1u) &&
                !chunk_hidden<HIZ>(vs.v[v], c, e, bound ? bound + tile_off[v] : nullptr, tdim[v]))
                vis |= 1u << v;
        return vis;
    };
    // points ip[j] of this lane (those with in[j]), each in the views of its mask vm[j]:
    // per view four projections, four early depth reads, then the atomics
    auto render_pts = [&](const uint64_t* ip, const bool* in, const uint32_t* vm) {
        float x[4], y[4], z[4];
        uint32_t idx[4];
        uint32_t vall = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint64_t i = ip[j];
            idx[j] = (uint32_t)i + vs.base;
            x[j] = y[j] = z[j] = 0.0f;
            if (in[j]) {
                x[j] = xyz[3 * i];
                y[j] = xyz[3 * i + 1];
                z[j] = xyz[3 * i + 2];
                vall |= vm[j];
            }
        }
        const f2 X[2] = {f2_pack(x[0], x[1]), f2_pack(x[2], x[3])};
        const f2 Y[2] = {f2_pack(y[0], y[1]), f2_pack(y[2], y[3])};
        const f2 Z[2] = {f2_pack(z[0], z[1]), f2_pack(z[2], z[3])};
        while (vall) {
            const int v = SINGLE ? 0 : __ffs(vall) - 1;
            vall &= vall - 1;
            uint32_t inv = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) inv |= (in[j] && ((vm[j] >> v) & 1u)) ? 1u << j : 0u;
            FView fv;
            if (!SINGLE) fv = fs[v];
            render_view<false>(SINGLE ? freg : fv, X, Y, Z, idx, inv);
            if (fs[v].wide) render_wide4(fs[v], vs.v[v], X, Y, Z, idx, inv);
        }
    };
    // up to four chunks: one point of each per lane
    auto render4 = [&](const uint32_t* k, const uint32_t* vm, int cnt) {
        uint64_t ip[4];
        bool in[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            ip[j] = (uint64_t)k[j] * RENDER_CHUNK + lane;
            in[j] = j < cnt && ip[j] < n;
        }
        render_pts(ip, in, vm);
    };
    if (prepass) {
        // four prepass chunks per warp step
        for (uint32_t k0 = warp * 4 * S; k0 < nch; k0 += nwarps * 4 * S) {
            uint32_t k[4], vm[4];
            int cnt = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                k[j] = k0 + j * S;
                vm[j] = all;
                if (k[j] < nch) cnt = j + 1;
            }
            render4(k, vm, cnt);
        }
        return;
    }
    // this warp's queue of surviving chunks (at most 7 left over + 32 new) and, SUB, of
    // surviving sub-chunks (at most 15 left over + 32 new)
    __shared__ uint32_t q_k[8][40];
    __shared__ uint8_t q_m[8][40];
    __shared__ uint32_t s_k[SUB ? 8 : 1][48];
    __shared__ uint8_t s_m[SUB ? 8 : 1][48];
    uint32_t* qk = q_k[threadIdx.x / 32];
    uint8_t* qm = q_m[threadIdx.x / 32];
    uint32_t* sk = s_k[SUB ? threadIdx.x / 32 : 0];
    uint8_t* sm = s_m[SUB ? threadIdx.x / 32 : 0];
    int qn = 0, sn = 0;   // queued, the same in every lane
    auto render_queued = [&](int from, int cnt) {
        uint32_t k[4] = {0u, 0u, 0u, 0u}, vm[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < cnt) {
                k[j] = qk[from + j];
                vm[j] = qm[from + j];
            }
        render4(k, vm, cnt);
    };
    // sub-chunks sk[from .. from + cnt), cnt <= 16: lane takes point lane % 8 of
    // sub-chunks 4j + lane / 8, j = 0..3
    auto render_subs = [&](int from, int cnt) {
        uint64_t ip[4];
        bool in[4];
        uint32_t vm[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = 4 * j + lane / RENDER_SUB;
            const bool have = q < cnt;
            const uint32_t ks = have ? sk[from + q] : 0u;
            vm[j] = have ? sm[from + q] : 0u;
            ip[j] = (uint64_t)ks * RENDER_SUB + lane % RENDER_SUB;
            in[j] = have && ip[j] < n;
        }
        render_pts(ip, in, vm);
    };
    // sub-chunk tests of the queued chunks qk[from .. from + cnt), cnt <= 8: lane tests
    // sub-chunk lane % 4 of chunk lane / 4 in the views its chunk survived; the visible
    // ones join the sub-chunk queue, which renders whenever sixteen are queued
    auto test_subs = [&](int from, int cnt) {
        const int c = lane / RENDER_SUBS;
        uint32_t vis = 0, ks = 0;
        if (c < cnt) {
            ks = qk[from + c] * RENDER_SUBS + lane % RENDER_SUBS;
            if ((uint64_t)ks * RENDER_SUB < n) {   // a sub-chunk past the last point holds none
                const float2* cp = reinterpret_cast<const float2*>(chunks + 6 * ((size_t)nch + ks));
                const float2 a = __ldg(cp), b = __ldg(cp + 1), d = __ldg(cp + 2);
                const float cc[3] = {a.x, a.y, b.x}, ee[3] = {b.y, d.x, d.y};
                vis = box_visible(cc, ee, qm[from + c]);
            }
        }
        const uint32_t ball = __ballot_sync(0xffffffffu, vis != 0);
        if (vis) {
            const int at = sn + __popc(ball & ((1u << lane) - 1u));
            sk[at] = ks;
            sm[at] = (uint8_t)vis;
        }
        sn += __popc(ball);
        __syncwarp();
        while (sn >= 16) {
            sn -= 16;
            render_subs(sn, 16);
        }
        __syncwarp();
    };
    // culled pass over the runs at places [r_begin, r_end) of the run order, one group of 32
    // chunks per warp and run
    const uint32_t ngroups = (nch + 31) / 32;
    uint32_t run = (uint32_t)((uint64_t)(r_begin + blockIdx.x) * run_step % nruns);
    const uint32_t run_inc = (uint32_t)((uint64_t)gridDim.x * run_step % nruns);
    for (uint32_t t = r_begin + blockIdx.x; t < r_end; t += gridDim.x) {
        const uint32_t g = run * RENDER_RUN + threadIdx.x / 32;
        run += run_inc;
        if (run >= nruns) run -= nruns;
        if (g >= ngroups) continue;
        const uint32_t kk = g * 32 + lane;
        uint32_t vis = 0;
        if (kk < nch && (kk & (S - 1)) != 0) {
            const float2* cp = reinterpret_cast<const float2*>(chunks + 6 * (size_t)kk);
            const float2 a = __ldg(cp), b = __ldg(cp + 1), d = __ldg(cp + 2);
            const float c[3] = {a.x, a.y, b.x}, e[3] = {b.y, d.x, d.y};
            vis = box_visible(c, e, all);
        }
        const uint32_t ball = __ballot_sync(0xffffffffu, vis != 0);
        if (vis) {
            const int at = qn + __popc(ball & ((1u << lane) - 1u));
            qk[at] = kk;
            qm[at] = (uint8_t)vis;
        }
        qn += __popc(ball);
        __syncwarp();
        if (SUB) {
            while (qn >= 8) {
                qn -= 8;
                test_subs(qn, 8);
            }
        } else {
            while (qn >= 4) {
                qn -= 4;
                render_queued(qn, 4);
            }
        }
        __syncwarp();
    }
    if (SUB) {
        if (qn > 0) test_subs(0, qn);
        if (sn > 0) render_subs(0, sn);
    } else if (qn > 0) {
        render_queued(0, qn);
    }
}

size_t visibility_scratch_bytes(const RViews& views) {
    size_t words = 0;
    for (int v = 0; v < views.n; ++v) words += (size_t)tile_dims(views.v[v].width, views.v[v].height).words;
    return words * sizeof(uint32_t);
}

// ------------------------------------------------------------------ variant choice
// The best variant depends on the point order and the views (how many early
// depth reads hit, how many atomics are left).  The first launch for a
// (single/multi view, size class) tries every variant on the real data -- each
// run computes the same keys -- and keeps the fastest for later launches.  No
// choice is made during a stream capture: the default variant is used until an
// uncaptured launch has tuned.
//
typedef void (*VisFn)(const float4*, uint32_t, const float*, uint64_t, RViews, const RViews*,
                      uint32_t);

constexpr uint64_t SPAN_MAX = 4096;   // groups of 4 points (16K points)

struct VisVariant {
    VisFn fn;            // null for a chunk-culling variant
    const char* name;
    int blocks_per_sm;   // resident blocks, from the compiled register count
    uint32_t chunk_S;    // chunk culling: every S-th chunk renders in the prepass (0: not chunked;
                         // otherwise a power of two)
    int phases;          // chunk culling: culled passes, tile bounds rebuilt before each
    int single;          // chunk culling, one view: the view's parameters held in registers
    int sub;             // chunk culling: surviving chunks tested again by their 8-point sub-chunks
    int hiz;             // chunk culling: box tests read the bound pyramid (at most 4 words)
    int first_part;      // chunk culling, two parts: the first part's share in percent (0: equal)
};

static VisVariant kSingle[] = {
    {visibility_kernel<true, false, 3>, "single/plain/3", 0},
    {visibility_kernel<true, true, 3>, "single/prefetch/3", 0},
    {visibility_kernel<true, true, 2>, "single/prefetch/2", 0},
    {visibility_kernel<true, false, 2>, "single/plain/2", 0},
    {nullptr, "single/chunks/16x2/r/33", 0, 16, 2, 1, 0, 0, 33},
    {nullptr, "single/chunks/16x2/r/25", 0, 16, 2, 1, 0, 0, 25},
    {nullptr, "single/chunks/32x2/r", 0, 32, 2, 1},
    {nullptr, "single/chunks/16x2/r/hiz/33", 0, 16, 2, 1, 0, 1, 33},
    {nullptr, "single/chunks/16", 0, 16, 1},
    {nullptr, "single/chunks/16x2", 0, 16, 2},
    {nullptr, "single/chunks/16x4", 0, 16, 4},
    {nullptr, "single/chunks/16/r", 0, 16, 1, 1},
    {nullptr, "single/chunks/16x2/r", 0, 16, 2, 1},
    {nullptr, "single/chunks/16x4/r", 0, 16, 4, 1},
    {nullptr, "single/chunks/16/r/sub", 0, 16, 1, 1, 1},
    {nullptr, "single/chunks/16x2/r/sub", 0, 16, 2, 1, 1},
    {nullptr, "single/chunks/16x4/r/sub", 0, 16, 4, 1, 1},
    {nullptr, "single/chunks/16x2/r/hiz", 0, 16, 2, 1, 0, 1},
    {nullptr, "single/chunks/16/r/sub/hiz", 0, 16, 1, 1, 1, 1},
    {nullptr, "single/chunks/16x2/r/sub/hiz", 0, 16, 2, 1, 1, 1},
    {nullptr, "single/chunks/16x4/r/sub/hiz", 0, 16, 4, 1, 1, 1},
    {nullptr, "single/chunks/32x2/r/sub/hiz", 0, 32, 2, 1, 1, 1},
    {nullptr, "single/chunks/8x2/r/sub/hiz", 0, 8, 2, 1, 1, 1},
    {nullptr, "single/chunks/16x2/r/sub/hiz/33", 0, 16, 2, 1, 1, 1, 33},
    {nullptr, "single/chunks/16x2/r/sub/hiz/25", 0, 16, 2, 1, 1, 1, 25},
};
static VisVariant kMulti[] = {
    {visibility_kernel<false, true, 3>, "multi/prefetch/3", 0},
    {visibility_kernel<false, false, 3>, "multi/plain/3", 0},
    {visibility_kernel<false, true, 2>, "multi/prefetch/2", 0},
    {nullptr, "multi/chunks/16x2/33", 0, 16, 2, 0, 0, 0, 33},
    {nullptr, "multi/chunks/16", 0, 16, 1},
    {nullptr, "multi/chunks/16x2", 0, 16, 2},
    {nullptr, "multi/chunks/16x4", 0, 16, 4},
    {nullptr, "multi/chunks/16x2/sub", 0, 16, 2, 0, 1},
    {nullptr, "multi/chunks/16x2/sub/hiz", 0, 16, 2, 0, 1, 1},
    {visibility_kernel<false, false, 4>, "multi/plain/4", 0},
};

typedef void (*ChunkFn)(const float*, uint64_t, const float*, RViews, const RViews*,
                        const uint32_t*, int, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t);
template <bool SINGLE>
static ChunkFn chunk_kernel_of(const VisVariant& v) {
    if (v.hiz) return v.sub ? chunk_render_kernel<SINGLE, true, true> : chunk_render_kernel<SINGLE, false, true>;
    return v.sub ? chunk_render_kernel<SINGLE, true, false> : chunk_render_kernel<SINGLE, false, false>;
}
static ChunkFn chunk_kernel(const VisVariant& v) {
    return v.single ? chunk_kernel_of<true>(v) : chunk_kernel_of<false>(v);
}

// The culled pass takes the scene in runs of RENDER_RUN groups (8K points), run i of the pass
// being run (i * step) mod nruns of the scene: with a step near the golden section of nruns and
// coprime to it, every prefix of the pass is spread over the whole scene.  A scene stored far
// to near along the view axis (a grid, layer by layer) would otherwise have every layer pass
// the tests and overwrite the last one, and a first part of the pass that occludes nothing.
static uint32_t run_order_step(uint32_t nruns) {
    uint32_t step = (uint32_t)(0.6180339887 * nruns);
    if (step < 1) step = 1;
    auto gcd = [](uint32_t a, uint32_t b) {
        while (b) {
            const uint32_t t = a % b;
            a = b;
            b = t;
        }
        return a;
    };
    while (gcd(step, nruns) != 1) ++step;
    return step;
}

static nrv_status resident_blocks(VisVariant& v) {
    if (v.blocks_per_sm) return NRV_OK;
    cudaFuncAttributes fa;
    if (v.fn) NRV_CHECK_CUDA(cudaFuncGetAttributes(&fa, v.fn));
    else NRV_CHECK_CUDA(cudaFuncGetAttributes(&fa, chunk_kernel(v)));
    const int regs_per_warp = (fa.numRegs * 32 + 255) / 256 * 256;
    int b = 65536 / (regs_per_warp * 8);
    if (b > 8) b = 8;
    v.blocks_per_sm = b > 0 ? b : 1;
    return NRV_OK;
}

static int g_vis_choice[2][48];   // [multi][log2 of the point count]; 0 = untuned
static int g_vis_sms = 0;

static nrv_status run_variant(VisVariant& v, const float* xyz, uint64_t n,
                              const RViews& views, cudaStream_t s, const RViews* views_dev,
                              uint32_t* tiles, const void* chunks) {
    NRV_TRY(resident_blocks(v));
    if (v.chunk_S) {
        if (!tiles || !chunks) return fail(NRV_ERR_ARG, "chunk culling needs tiles and chunk bounds");
        const int blocks = g_vis_sms * v.blocks_per_sm;
        const float* ch = reinterpret_cast<const float*>(chunks);
        const uint32_t ngroups = (uint32_t)((chunk_count(n) + 31) / 32);
        const ChunkFn kern = chunk_kernel(v);
        const uint32_t nruns = (ngroups + RENDER_RUN - 1) / RENDER_RUN;
        const uint32_t step = run_order_step(nruns);
        NRV_TRY(launch_pdl(kern, dim3(blocks), dim3(256), s, xyz, n, ch, views, views_dev,
                           (const uint32_t*)nullptr, 1, v.chunk_S, 0u, 0u, step, nruns));
        // the chunk groups in `phases` consecutive parts, the tile bounds rebuilt from the
        // keys so far before each part (later parts meet tighter bounds)
        for (int ph = 0; ph < v.phases; ++ph) {
            uint32_t g0 = (uint32_t)((uint64_t)nruns * ph / v.phases);
            uint32_t g1 = (uint32_t)((uint64_t)nruns * (ph + 1) / v.phases);
            if (v.phases == 2 && v.first_part) {
                const uint32_t cut = (uint32_t)((uint64_t)nruns * v.first_part / 100);
                g0 = ph ? cut : 0u;
                g1 = ph ? nruns : cut;
            }
            NRV_TRY(launch_tile_bounds(views, views_dev, tiles, v.hiz != 0, s));
            NRV_TRY(launch_pdl(kern, dim3(blocks), dim3(256), s, xyz, n, ch, views, views_dev,
                               (const uint32_t*)tiles, 0, v.chunk_S, g0, g1, step, nruns));
        }
        return NRV_OK;
    }
    const uint64_t ngroups = n / 4;
    // spans of at most 16K points, at least eight per resident block where there are that many;
    // a smaller scene in one wave (1M points, 512 x 512: 25.3 us against 26.6 for 1024-point
    // spans in 2.1 waves)
    const uint64_t step = 256, resident = (uint64_t)g_vis_sms * v.blocks_per_sm;
    uint64_t span = ngroups / (resident * 8) / step * step;
    if (span < step) span = ((ngroups + resident - 1) / resident + step - 1) / step * step;
    if (span > SPAN_MAX) span = SPAN_MAX;
    if (span < step) span = step;
    const uint64_t blocks = (ngroups + span - 1) / span;
    return launch_pdl(v.fn, dim3((unsigned)(blocks > 0 ? blocks : 1)), dim3(256), s,
                      reinterpret_cast<const float4*>(xyz), (uint32_t)ngroups, xyz, n, views, views_dev,
                      (uint32_t)span);
}

int visibility_variant_count(int multi) {
    return multi ? (int)(sizeof(kMulti) / sizeof(kMulti[0])) : (int)(sizeof(kSingle) / sizeof(kSingle[0]));
}
const char* visibility_variant_name(int multi, int i) { return (multi ? kMulti : kSingle)[i].name; }

// FNV-1a over the names of a variant table, in order.  A stored choice is an index into the table:
// with the table's hash in its key, a file saved with other variants selects none of these.
static uint32_t variant_table_hash(int multi) {
    uint32_t h = 2166136261u;
    for (int i = 0; i < visibility_variant_count(multi); ++i)
        for (const char* c = visibility_variant_name(multi, i);; ++c) {
            h = (h ^ (uint8_t)*c) * 16777619u;
            if (!*c) break;
        }
    return h;
}

static bool verbose() {
    static int v = -1;
    if (v < 0) {
        const char* e = getenv("NRV_VERBOSE");
        v = e && *e && *e != '0';
    }
    return v == 1;
}

nrv_status launch_visibility(const float* xyz, uint64_t n, const RViews& views, cudaStream_t s,
                             const RViews* views_dev, uint32_t* tiles, const void* chunks) {
    if (n == 0) return NRV_OK;
    if (!g_vis_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_vis_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_vis_sms <= 0) g_vis_sms = 148;
    }
    const int multi = views.n > 1;
    VisVariant* tab = multi ? kMulti : kSingle;
    const int count = visibility_variant_count(multi);
    int cls = 0;
    while (cls < 47 && (1ull << (cls + 1)) <= n) ++cls;
    int& choice = g_vis_choice[multi][cls];
    static const uint32_t table[2] = {variant_table_hash(0), variant_table_hash(1)};
    char tkey[64];
    snprintf(tkey, sizeof(tkey), "render multi=%d log2n=%d table=%08x", multi, cls, table[multi]);
    if (choice == 0) {
        int v = 0;
        if (tune_get(tkey, &v) && v >= 0 && v < count) choice = v + 1;
    }
    // NRV_VIS_VARIANT=<i> pins variant i (used to check every variant)
    if (const char* e = getenv("NRV_VIS_VARIANT")) {
        const int i = atoi(e);
        if (i >= 0 && i < count) {
            if (tab[i].chunk_S && (!tiles || !chunks))
                return fail(NRV_ERR_ARG, "variant %d needs tile scratch and chunk bounds", i);
            return run_variant(tab[i], xyz, n, views, s, views_dev, tiles, chunks);
        }
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    NRV_CHECK_CUDA(cudaStreamIsCapturing(s, &cap));
    if (choice == 0 && cap == cudaStreamCaptureStatusNone && n >= (1u << 20)) {
        // time each variant twice on the real data; keep the faster second run
        cudaEvent_t e0, e1;
        NRV_CHECK_CUDA(cudaEventCreate(&e0));
        NRV_CHECK_CUDA(cudaEventCreate(&e1));
        float best = 1e30f;
        int arg = 0;
        for (int i = 0; i < count; ++i) {
            if (tab[i].chunk_S && (!tiles || !chunks)) continue;
            float ms = 0.0f;
            for (int rep = 0; rep < 2; ++rep) {
                NRV_TRY(launch_clear_keys(views, s));
                NRV_CHECK_CUDA(cudaEventRecord(e0, s));
                NRV_TRY(run_variant(tab[i], xyz, n, views, s, views_dev, tiles, chunks));
                NRV_CHECK_CUDA(cudaEventRecord(e1, s));
                NRV_CHECK_CUDA(cudaEventSynchronize(e1));
                NRV_CHECK_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            }
            if (verbose()) fprintf(stderr, "nrv: render pass %d %-26s %.3f ms\n", i, tab[i].name, ms);
            if (ms < best) {
                best = ms;
                arg = i;
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        choice = arg + 1;
        tune_put(tkey, arg);
        tune_count_timing();
        NRV_TRY(launch_clear_keys(views, s));
    }
    int pick = choice > 0 ? choice - 1 : 0;
    if (tab[pick].chunk_S && (!tiles || !chunks)) pick = 0;
    return run_variant(tab[pick], xyz, n, views, s, views_dev, tiles, chunks);
}

// ------------------------------------------------------------------ pack helpers

// Word k of a record held in registers (an indexed array would live in local memory).
template <int SW>
__device__ __forceinline__ uint32_t pick(const uint32_t* w, int k) {
    uint32_t r = w[0];
#pragma unroll
    for (int j = 1; j < SW; ++j) r = k == j ? w[j] : r;
    return r;
}

// Derived channels (Sec. 4.5 "Vel2D", Sec. 3.2 splat radius) of the point at p, in FP32.
// v' = (ds/dp) v with s the screen map: for c = M (p, 1),
// ds_x/dp = (W/2) (M_0 - (c.x/c.w) M_3) / c.w and ds_y/dp = -(H/2) (M_1 - (c.y/c.w) M_3) / c.w
// (M_r the first three entries of row r).  The reciprocal depth is shared by every channel of
// the pixel, the projected velocity by the channels of one velocity.
struct Camera {
    float m[12];   // rows 0, 1 and 3 of the view-projection
    float hw, hh;
};
struct Derived {
    const Camera* k;
    const float* p;
    float iw, px, py;
    int wd;        // the velocity's first word px, py belong to (-1: none yet)
    __device__ __forceinline__ void init(const Camera* cam, const float* pt) {
        k = cam;
        p = pt;
        const float* m = cam->m;
        iw = 1.0f / fmaf(m[8], p[0], fmaf(m[9], p[1], fmaf(m[10], p[2], m[11])));
        wd = -1;
    }
    template <int SW>
    __device__ __forceinline__ float channel(int fmt, const uint32_t* words, int w) {
        const float* m = k->m;
        if (fmt == NRV_SPLAT_RADIUS) {
            const float r1 = sqrtf(fmaf(m[4], m[4], fmaf(m[5], m[5], m[6] * m[6])));
            return __uint_as_float(pick<SW>(words, w)) * k->hh * r1 * iw;
        }
        if (w != wd) {
            wd = w;
            const float vx = __uint_as_float(pick<SW>(words, w)), vy = __uint_as_float(pick<SW>(words, w + 1)),
                        vz = __uint_as_float(pick<SW>(words, w + 2));
            const float cx = fmaf(m[0], p[0], fmaf(m[1], p[1], fmaf(m[2], p[2], m[3])));
            const float cy = fmaf(m[4], p[0], fmaf(m[5], p[1], fmaf(m[6], p[2], m[7])));
            const float mv0 = fmaf(m[0], vx, fmaf(m[1], vy, m[2] * vz));
            const float mv1 = fmaf(m[4], vx, fmaf(m[5], vy, m[6] * vz));
            const float mv3 = fmaf(m[8], vx, fmaf(m[9], vy, m[10] * vz));
            px = k->hw * iw * fmaf(-cx * iw, mv3, mv0);
            py = -k->hh * iw * fmaf(-cy * iw, mv3, mv1);
        }
        if (fmt == NRV_VEL2D_X) return px;
        if (fmt == NRV_VEL2D_Y) return py;
        if (fmt == NRV_VEL2D_ANGLE) return atan2f(py, px);
        return sqrtf(fmaf(px, px, py * py));
    }
};

// The up to 8 channels f of one covered pixel; dv null without derived channels.
template <int SW>
__device__ __forceinline__ void pack_channels(const ResolveArgs& a, uint32_t depth_bits,
                                              const uint32_t* words, float* f, Derived* dv) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        f[j] = 0.0f;
        if (j < 6 && j < a.n_ch) {
            float v;
            if (dv && a.ch_fmt[j] >= NRV_VEL2D_X) {
                v = dv->channel<SW>(a.ch_fmt[j], words, a.ch_word[j]);
            } else {
                const uint32_t w = pick<SW>(words, a.ch_word[j]);
                if (a.ch_fmt[j] == NRV_F32) v = __uint_as_float(w);
                else if (a.ch_fmt[j] == NRV_U32) v = __uint2float_rn(w);
                else v = (float)((w >> (8 * a.ch_comp[j])) & 255u);
            }
            f[j] = __fadd_rn(__fmul_rn(v, a.ch_scale[j]), a.ch_offset[j]);
        }
        if (j == a.n_ch) f[j] = __fadd_rn(__fmul_rn(__uint_as_float(depth_bits), a.d_scale), a.d_offset);
        if (j == a.n_ch + 1) f[j] = 1.0f;
    }
}

// Write one canvas pixel of the network input (all channels, zero padded).
__device__ __forceinline__ void store_netin(const ResolveArgs& a, size_t q, const float* f) {
    if (a.out_fmt == 0) {
        float4* o = reinterpret_cast<float4*>(a.netin) + 2 * q;
        o[0] = make_float4(f[0], f[1], f[2], f[3]);
        o[1] = make_float4(f[4], f[5], f[6], f[7]);
    } else if (a.out_fmt == 1) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
            w[j] = *reinterpret_cast<uint32_t*>(&h);
        }
        reinterpret_cast<uint4*>(a.netin)[q] = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const __nv_fp8_storage_t b = __nv_cvt_float_to_fp8(__fmul_rn(f[j], a.in_scale_inv),
                                                               __NV_SATFINITE, __NV_E4M3);
            w[j >> 2] |= (uint32_t)b << (8 * (j & 3));
        }
        reinterpret_cast<uint4*>(a.netin)[q] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Resolve pass (Sec. 3.2) of the views of one call (blockIdx.y): reads the key of each canvas
// pixel, gathers the winner's record and writes the raw planes and/or the packed network input.
// Bound by the latency of key -> record -> store, so a thread takes four pixels, 256 apart, and
// has their keys and then their records in flight together; records stay in registers and
// indices in 32 bits (a canvas has at most 2^28 pixels).  SW: words per record; PACK: 0 planes
// only, 1 packed input, 2 packed input with derived channels.
// 1080p: planes of five words 24.9 -> 14.1 us, packing with four Vel2D channels 42.6 -> 28.1 us.
// (With derived channels a thread takes one pixel: four copies of that arithmetic are bound by
// instruction fetch, 59.4 us.)
struct ResolveBatch {
    ResolveArgs a[8];
};
constexpr int res_px(int pack) { return pack == 2 ? 1 : 4; }
template <int SW, int PACK>
__global__ void __launch_bounds__(256) resolve_kernel(const __grid_constant__ ResolveBatch batch) {
    constexpr int RES_PX = res_px(PACK);
    pdl_wait_and_release();
    const ResolveArgs& a = batch.a[blockIdx.y];
    const uint32_t wc = PACK ? a.wn : a.width, hc = PACK ? a.hn : a.height, total = wc * hc;
    const uint32_t npx = (uint32_t)a.width * a.height;
    const uint32_t q0 = blockIdx.x * (256 * RES_PX) + threadIdx.x;
    unsigned long long key[RES_PX];
    uint32_t p[RES_PX], words[RES_PX][SW];
    bool inside[RES_PX], hit[RES_PX];
    float pt[RES_PX][3];
#pragma unroll
    for (int j = 0; j < RES_PX; ++j) {
        const uint32_t q = q0 + 256 * j;
        p[j] = q;
        inside[j] = q < total;
        if (PACK) {
            const uint32_t y = q / wc, x = q - y * wc;
            inside[j] = inside[j] && x < (uint32_t)a.width && y < (uint32_t)a.height;
            p[j] = y * (uint32_t)a.width + x;
        }
        key[j] = inside[j] ? __ldcs(a.key + p[j]) : ~0ull;
    }
#pragma unroll
    for (int j = 0; j < RES_PX; ++j) {
        // the winner's index relative to this scene (a winner from another shard: empty here)
        const uint32_t idx = (uint32_t)key[j] - a.base;
        hit[j] = key[j] != ~0ull && idx < a.n_local;
#pragma unroll
        for (int k = 0; k < SW; ++k) words[j][k] = 0u;
        pt[j][0] = pt[j][1] = pt[j][2] = 0.0f;
        if (hit[j]) {
            const uint32_t* rec = a.attr + (size_t)idx * SW;
            if constexpr (SW >= 4) {
#pragma unroll
                for (int k = 0; k < SW / 4; ++k) {
                    const uint4 r = __ldg(reinterpret_cast<const uint4*>(rec) + k);
                    words[j][4 * k] = r.x;
                    words[j][4 * k + 1] = r.y;
                    words[j][4 * k + 2] = r.z;
                    words[j][4 * k + 3] = r.w;
                }
            } else if constexpr (SW == 2) {
                const uint2 r = __ldg(reinterpret_cast<const uint2*>(rec));
                words[j][0] = r.x;
                words[j][1] = r.y;
            } else {
                words[j][0] = __ldg(rec);
            }
            if (PACK == 2) {
                const float* xp = a.xyz + 3 * (size_t)idx;
                pt[j][0] = __ldg(xp);
                pt[j][1] = __ldg(xp + 1);
                pt[j][2] = __ldg(xp + 2);
            }
        }
    }
    Camera cam;
    if (PACK == 2) {
        const float* src = a.view_dev ? a.view_dev->m : a.vm;
#pragma unroll
        for (int j = 0; j < 12; ++j) cam.m[j] = src[j];
        cam.hw = a.view_dev ? a.view_dev->hw : a.vhw;
        cam.hh = a.view_dev ? a.view_dev->hh : a.vhh;
    }
#pragma unroll
    for (int j = 0; j < RES_PX; ++j) {
        const uint32_t depth_bits = hit[j] ? (uint32_t)(key[j] >> 32) : 0u;
        if (inside[j]) {
            if (a.depth) a.depth[p[j]] = depth_bits;
            if (a.mask) a.mask[p[j]] = hit[j] ? 1 : 0;
            if (a.gattr) {
#pragma unroll
                for (int c = 0; c < SW; ++c)
                    if (c < a.n_words) a.gattr[(size_t)c * npx + p[j]] = words[j][c];
            }
        }
        if (PACK && q0 + 256 * j < total) {
            float f[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) f[k] = 0.0f;
            if (hit[j]) {
                Derived dv;
                if (PACK == 2) dv.init(&cam, pt[j]);
                pack_channels<SW>(a, depth_bits, words[j], f, PACK == 2 ? &dv : nullptr);
            }
            store_netin(a, q0 + 256 * j, f);
        }
    }
}

__global__ void flip_sign_kernel(unsigned long long* k, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        k[i] ^= 0x8000000000000000ull;
}

static int grid_for(size_t work, int per_block = 256) {
    size_t b = (work + per_block - 1) / per_block;
    const size_t cap = 152 * 16;
    if (b > cap) b = cap;
    return (int)(b > 0 ? b : 1);
}

nrv_status launch_flip_sign(uint64_t* keys, int64_t n, cudaStream_t s) {
    flip_sign_kernel<<<grid_for((size_t)n), 256, 0, s>>>(reinterpret_cast<unsigned long long*>(keys), n);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

template <int SW>
static nrv_status resolve_words(const ResolveBatch& b, dim3 grid, int pack, cudaStream_t s) {
    auto kern = pack == 0 ? resolve_kernel<SW, 0> : pack == 1 ? resolve_kernel<SW, 1> : resolve_kernel<SW, 2>;
    return launch_pdl(kern, grid, dim3(256), s, b);
}

// n views of one call: one scene, one kind of output.
nrv_status launch_resolve(const ResolveArgs* a, int n, cudaStream_t s) {
    ResolveBatch b;
    memset(&b, 0, sizeof(b));
    size_t most = 1;
    for (int i = 0; i < n; ++i) {
        b.a[i] = a[i];
        const size_t total = a[i].netin ? (size_t)a[i].wn * a[i].hn : (size_t)a[i].width * a[i].height;
        if (total > most) most = total;
    }
    const int pack = !a[0].netin ? 0 : a[0].derived ? 2 : 1, per = 256 * res_px(pack);
    const dim3 grid((unsigned)((most + per - 1) / per), (unsigned)n);
    switch (a[0].stride_words) {
        case 8: return resolve_words<8>(b, grid, pack, s);
        case 4: return resolve_words<4>(b, grid, pack, s);
        case 2: return resolve_words<2>(b, grid, pack, s);
        default: return resolve_words<1>(b, grid, pack, s);
    }
}

// Pack from already-resolved planes (nrv_pack).
__global__ void __launch_bounds__(256) pack_planes_kernel(const uint32_t* __restrict__ depth,
                                                          const uint8_t* __restrict__ mask,
                                                          const uint32_t* __restrict__ gattr,
                                                          const __grid_constant__ ResolveArgs a) {
    const uint32_t total = (uint32_t)a.wn * a.hn;
    const size_t npx = (size_t)a.width * a.height;
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < total; q += gridDim.x * blockDim.x) {
        const uint32_t y = q / (uint32_t)a.wn, x = q - y * (uint32_t)a.wn;
        float f[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = 0.0f;
        if (x < (uint32_t)a.width && y < (uint32_t)a.height) {
            const size_t p = (size_t)y * a.width + x;
            if (mask[p]) {
                // channel j's word in place j
                uint32_t words[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
                for (int j = 0; j < 6; ++j)
                    if (j < a.n_ch) words[j] = gattr[(size_t)a.ch_word[j] * npx + p];
                ResolveArgs b = a;
#pragma unroll
                for (int j = 0; j < 6; ++j) b.ch_word[j] = j;
                pack_channels<8>(b, depth[p], words, f, nullptr);
            }
        }
        store_netin(a, q, f);
    }
}

nrv_status launch_pack_planes(const uint32_t* depth, const uint8_t* mask, const uint32_t* gattr,
                              const ResolveArgs& a, cudaStream_t s) {
    pack_planes_kernel<<<grid_for((size_t)a.wn * a.hn), 256, 0, s>>>(depth, mask, gattr, a);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

}  // namespace nrv
