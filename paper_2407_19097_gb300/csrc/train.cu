// Training of the post-processing network (Sec. 3.3, training details): the
// backward pass of every layer, the L1 reconstruction loss and Adam.
//
// Gradients of the weights are reductions over all pixels.  They are computed
// in fixed pixel chunks whose partial sums are added in a fixed order by a
// second kernel, so a step is bit-for-bit reproducible.
#include <mutex>

#include "f32.h"
#include "net.h"
#include "net_simt.cuh"
#include "project.cuh"

namespace nrv {

// ------------------------------------------------------------------ weight gradients, 3x3 conv
// part[blk][o][tap*cin + c] = sum over the pixels of block blk's tiles of g[q][o] * x[q + tap][c];
// partb[blk][o] = sum of g.  A tile is 256 pixels: R rows x TW pixels, TW = 128, 64 or 32
// (the widest that the image width fills), R = 256 / TW.  The block stages the tile's
// gradients (16 output channels) and its input rows with a one-pixel halo (CG input
// channels) in shared memory as FP32, then each thread accumulates a 4 (output) x 4 (input)
// block of one tap -- 16 FMAs per pair of 16-byte shared loads.  Grid: (blocks over tiles,
// output groups of 16, input groups of CG); 144 threads = 9 taps x 4 x 4 blocks (CG = 16) or
// 72 (CG = 8).  Each block takes a contiguous run of tiles, so partials are summed in a
// fixed order: the result is deterministic.
constexpr int WG_TILE = 256;          // pixels per tile
constexpr int WG_THREADS = 144;
constexpr int WG_XS = 520;            // staged input pixels: max over TW of (R + 2) x (TW + 2)

inline int wgrad_tile_width(int w) { return w >= 128 ? 128 : (w >= 64 ? 64 : 32); }

template <typename T>
__global__ void __launch_bounds__(WG_THREADS) wgrad3_kernel(TView<const T> g, int cout,
                                                            TView<const T> x1, int c1,
                                                            TView<const T> x2, int c2, int n,
                                                            int h, int w, int TW,
                                                            int tiles_per_block, float* part,
                                                            float* partb) {
    constexpr int CGMAX = 16;
    __shared__ __align__(16) float gs[WG_TILE][16];
    __shared__ __align__(16) float xs[WG_XS][CGMAX];
    const int R = WG_TILE / TW;
    const int cin = c1 + c2;
    const int CG = cin < 16 ? cin : 16;   // 8 (the packed first-layer input) or 16
    const int og = blockIdx.y * 16, cg = blockIdx.z * CG;
    const int t = threadIdx.x;
    const int ncb = CG / 4;               // 4-channel blocks of the input group
    const bool active = t < 9 * 4 * ncb;
    const int tap = t / (4 * ncb), ob = (t / ncb) % 4, cb = t % ncb;
    const int dy = tap / 3, dx = tap % 3;
    // which source holds this input group
    const TView<const T> xv = cg < c1 ? x1 : x2;
    const int cx = cg < c1 ? cg : cg - c1;
    const int tiles_x = (w + TW - 1) / TW, pairs = (h + R - 1) / R;
    const long long ntiles = (long long)n * pairs * tiles_x;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    float bsum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    const long long t0 = (long long)blockIdx.x * tiles_per_block;
    const long long t1 = t0 + tiles_per_block < ntiles ? t0 + tiles_per_block : ntiles;
    for (long long tile = t0; tile < t1; ++tile) {
        const int xt = (int)(tile % tiles_x);
        const long long rest = tile / tiles_x;
        const int pr = (int)(rest % pairs);
        const int img = (int)(rest / pairs);
        const int x0 = xt * TW, y0 = R * pr;
        __syncthreads();
        // gradients of the tile's R x TW pixels, 16 output channels (zero outside the image)
        for (int i = t; i < WG_TILE * 2; i += WG_THREADS) {
            const int half = i & 1, px = (i >> 1) % TW, py = (i >> 1) / TW;
            const int y = y0 + py, x = x0 + px;
            float v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            if (y < h && x < w) ld8<T>(g.at((size_t)img * h + y, x, og + 8 * half, w), v);
#pragma unroll
            for (int k = 0; k < 8; ++k) gs[py * TW + px][8 * half + k] = v[k];
        }
        // input rows y0-1 .. y0+R, pixels x0-1 .. x0+TW, CG channels (zero padding)
        const int nxh = CG / 8;
        for (int i = t; i < (R + 2) * (TW + 2) * nxh; i += WG_THREADS) {
            const int part8 = i % nxh, px = (i / nxh) % (TW + 2), ry = (i / nxh) / (TW + 2);
            const int y = y0 - 1 + ry, x = x0 - 1 + px;
            float v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            if (y >= 0 && y < h && x >= 0 && x < w)
                ld8<T>(xv.at((size_t)img * h + y, x, cx + 8 * part8, w), v);
#pragma unroll
            for (int k = 0; k < 8; ++k) xs[ry * (TW + 2) + px][8 * part8 + k] = v[k];
        }
        __syncthreads();
        if (active) {
            for (int py = 0; py < R; ++py) {
                const float* grow = &gs[py * TW][4 * ob];
                const float* xrow = &xs[(py + dy) * (TW + 2) + dx][4 * cb];
#pragma unroll 4
                for (int px = 0; px < TW; ++px) {
                    const float4 gv = *reinterpret_cast<const float4*>(grow + px * 16);
                    const float4 xv4 = *reinterpret_cast<const float4*>(xrow + px * CGMAX);
                    const float ga[4] = {gv.x, gv.y, gv.z, gv.w};
                    const float xa[4] = {xv4.x, xv4.y, xv4.z, xv4.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ga[i], xa[j], acc[i][j]);
                    if (tap == 0 && cb == 0) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) bsum[i] += ga[i];
                    }
                }
            }
        }
    }
    if (!active) return;
    const int K = 9 * cin;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            part[((size_t)blockIdx.x * cout + og + 4 * ob + i) * K + tap * cin + cg + 4 * cb + j] =
                acc[i][j];
    if (blockIdx.z == 0 && tap == 0 && cb == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) partb[(size_t)blockIdx.x * cout + og + 4 * ob + i] = bsum[i];
}

// Sums of per-chunk partials: sum i = part[0*stride + i] + part[1*stride + i] + ..., eight
// threads per sum each taking every eighth chunk, their results added in a fixed order (the
// result does not depend on timing).  `mode` says where sum i goes (PyTorch layouts):
//  0  3x3 conv weight: i = o*9*cin + tap*cin + c -> dw[(o*cin_real + c)*9 + tap] (c < cin_real)
//  1  transposed conv weight: i = c*4*cout + ab*cout + o -> dw[(c*cout + o)*4 + ab]
//  2  copy: dw[i]
//  3  transposed conv bias: i = o, each chunk contributing part[ab*cout + o] for ab = 0..3
struct ReduceSeg {
    const float* part;
    int nchunks;
    size_t stride;
    int count, mode, cout, cin, cin_real;
    float* dw;
};

// Every segment in one launch: block b belongs to the segment whose range of blocks holds it.
// Each thread reads eight chunks of four sums before it adds them, so the pass is bound by the
// partials' bytes (123 MB in the 16 x 256^2 training step) and not by a chain of dependent loads.
// Before the search by halves and the batched loads of the odd segments, single blocks with
// chains of dependent loads ran 78k cycles against a mean of 27k (45 us; now 27).
constexpr int MAX_SEGS = 2 * NUM_LAYERS;
struct ReduceTable {
    int n;
    int first[MAX_SEGS + 1];   // first block of each segment
    ReduceSeg seg[MAX_SEGS];
};
// four consecutive sums per thread?
__host__ __device__ inline bool reduce_vec(const ReduceSeg& R) {
    return R.mode != 3 && R.count % 4 == 0 && R.stride % 4 == 0;
}
__host__ __device__ inline int reduce_blocks(const ReduceSeg& R) {
    const int per = reduce_vec(R) ? 128 : 32;
    return (R.count + per - 1) / per;
}

__device__ __forceinline__ void reduce_put(const ReduceSeg& R, int i, float t) {
    if (R.mode == 0) {
        const int K = 9 * R.cin, o = i / K, q = i % K, tap = q / R.cin, c = q % R.cin;
        if (c < R.cin_real) R.dw[((size_t)o * R.cin_real + c) * 9 + tap] = t;
    } else if (R.mode == 1) {
        const int K = 4 * R.cout, c = i / K, q = i % K, ab = q / R.cout, o = q % R.cout;
        R.dw[((size_t)c * R.cout + o) * 4 + ab] = t;
    } else {
        R.dw[i] = t;
    }
}

__global__ void __launch_bounds__(256) reduce_partials_kernel(const __grid_constant__ ReduceTable T) {
    __shared__ float red[8][132];
    int k = 0, end = T.n;      // first[k] <= block < first[end]
    while (end - k > 1) {
        const int mid = (k + end) >> 1;
        if ((int)blockIdx.x >= T.first[mid]) k = mid;
        else end = mid;
    }
    const ReduceSeg& R = T.seg[k];
    const int tx = threadIdx.x, ty = threadIdx.y, blk = (int)blockIdx.x - T.first[k];
    if (reduce_vec(R)) {
        const int i = blk * 128 + 4 * tx;
        float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (i < R.count)
            for (int c0 = ty; c0 < R.nchunks; c0 += 64) {
                float4 v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int ch = c0 + 8 * j;
                    v[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (ch < R.nchunks) v[j] = __ldcs(reinterpret_cast<const float4*>(R.part + (size_t)ch * R.stride + i));
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    s[0] += v[j].x;
                    s[1] += v[j].y;
                    s[2] += v[j].z;
                    s[3] += v[j].w;
                }
            }
#pragma unroll
        for (int e = 0; e < 4; ++e) red[ty][4 * tx + e] = s[e];
        __syncthreads();
        // 128 sums, the first 128 threads one each
        const int t = ty * 32 + tx;
        if (t >= 128 || blk * 128 + t >= R.count) return;
        float a = red[0][t];
        for (int j = 1; j < 8; ++j) a += red[j][t];
        reduce_put(R, blk * 128 + t, a);
        return;
    }
    // The few odd segments (the head's 51 sums, biases of transposed convs) have the longest
    // chains of chunks, and their blocks end last.
    const int i = blk * 32 + tx;
    float s = 0.0f;
    auto eight = [&](int c0, int off, float (&v)[8]) {
        const float* pc = R.part + (size_t)c0 * R.stride + off + i;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            v[j] = 0.0f;
            if (c0 + 8 * j < R.nchunks) v[j] = __ldcs(pc + (size_t)(8 * j) * R.stride);
        }
    };
    if (i < R.count) {
        if (R.mode == 3) {
            for (int c0 = ty; c0 < R.nchunks; c0 += 64) {
                float v[4][8];
#pragma unroll
                for (int ab = 0; ab < 4; ++ab) eight(c0, ab * R.cout, v[ab]);
#pragma unroll
                for (int j = 0; j < 8; ++j) s += ((v[0][j] + v[1][j]) + v[2][j]) + v[3][j];
            }
        } else {
            for (int c0 = ty; c0 < R.nchunks; c0 += 64) {
                float v[8];
                eight(c0, 0, v);
#pragma unroll
                for (int j = 0; j < 8; ++j) s += v[j];
            }
        }
    }
    red[ty][tx] = s;
    __syncthreads();
    if (ty != 0 || i >= R.count) return;
    float a = red[0][tx];
    for (int j = 1; j < 8; ++j) a += red[j][tx];
    reduce_put(R, i, a);
}

// The partial sums of a backward pass: one region per layer of the net's buffer, and the table
// of the segments to reduce once every partial is written.
struct Partials {
    DevBuf* buf;
    size_t used = 0;           // floats
    ReduceTable T;
    explicit Partials(DevBuf* b) : buf(b) { T.n = 0; T.first[0] = 0; }
    // `floats` floats; the buffer was sized for the whole pass (reserve), so nothing moves
    float* take(size_t floats) {
        float* p = (float*)buf->p + used;
        used += (floats + 31) / 32 * 32;
        return used * sizeof(float) <= buf->bytes ? p : nullptr;
    }
    void add(const ReduceSeg& R) {
        T.seg[T.n] = R;
        T.first[T.n + 1] = T.first[T.n] + reduce_blocks(R);
        ++T.n;
    }
    nrv_status flush(cudaStream_t s) {
        if (T.n == 0) return NRV_OK;
        reduce_partials_kernel<<<T.first[T.n], dim3(32, 8), 0, s>>>(T);
        NRV_CHECK_LAUNCH();
        T.n = 0;
        used = 0;
        return NRV_OK;
    }
};

// ------------------------------------------------------------------ weight gradients, 2x2 transposed conv
// part[chunk][c][ab*cout + o] = sum_{input px in chunk} x[q][c] * g[out(q, ab)][o]
// partb[chunk][ab*cout + o]   = sum g   (only written by the c-group 0 blocks)
template <typename T>
__global__ void __launch_bounds__(256) wgrad_up_kernel(TView<const T> x, int cin, TView<const T> g,
                                                       int cout, int n, int hi, int wi,
                                                       size_t chunk_px, float* part, float* partb) {
    __shared__ float xs[32][16];
    const int cg = blockIdx.y * 16;
    const int K = 4 * cout;
    const size_t npx = (size_t)n * hi * wi;
    const size_t q0 = blockIdx.x * chunk_px;
    const size_t q1 = q0 + chunk_px < npx ? q0 + chunk_px : npx;
    float acc[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j] = 0.0f;
    float bsum = 0.0f;
    const int k = threadIdx.x;
    const int ab = k / cout, o = k % cout;
    for (size_t qb = q0; qb < q1; qb += 32) {
        __syncthreads();
        for (int i = threadIdx.x; i < 512; i += 256) {
            const size_t q = qb + (i >> 4);
            xs[i >> 4][i & 15] =
                q < q1 ? ld1<T>(x.at(q / wi, (int)(q % wi), cg + (i & 15), wi)) : 0.0f;
        }
        __syncthreads();
        const int nb = (int)(q1 - qb < 32 ? q1 - qb : 32);
        if (k < K)
            for (int r = 0; r < nb; ++r) {
                const size_t q = qb + r;
                const int X = (int)(q % wi), Y = (int)((q / wi) % hi);
                const size_t img = q / ((size_t)wi * hi);
                const float gv = ld1<T>(
                    g.at(img * 2 * hi + 2 * Y + (ab >> 1), 2 * X + (ab & 1), o, 2 * wi));
                bsum += gv;
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[j] = fmaf(xs[r][j], gv, acc[j]);
            }
    }
    if (k < K) {
#pragma unroll
        for (int j = 0; j < 16; ++j) part[((size_t)blockIdx.x * cin + cg + j) * K + k] = acc[j];
        if (blockIdx.y == 0) partb[(size_t)blockIdx.x * K + k] = bsum;
    }
}

// ------------------------------------------------------------------ head
// One pass over the last conv's output x and the image gradient makes both head gradients (two
// passes read them twice, 42 us in the 16 x 256^2 step):
//   gd[q][c] = (sum_o drgb[o] W[o][c]) * (x[q][c] > 0) over the canvas (zero outside the view);
//   part[blk][o*16 + c] = sum drgb[o] * x[c], part[blk][48 + o] = sum drgb[o] over the block's chunk
// of cropped pixels: every thread keeps all 51 sums, then the block adds them (warp shuffles,
// then the 8 warps in order).
// Latency- and issue-bound (78 MB would take 12 us there): channels in pairs, and the position
// advanced by the block's width instead of divided out per pixel, 38 -> 26 us; two threads per
// pixel at twice the warps measured 48.
template <typename T>
__global__ void __launch_bounds__(256, 2) head_bwd_kernel(const float* drgb, const float* __restrict__ w,
                                                       TView<const T> x, TView<T> gd, int n, int hn, int wn,
                                                       int h, int wd, size_t chunk, float* part) {
    __shared__ float red[8][51];
    __shared__ __align__(16) float ws[48];
    if (threadIdx.x < 48) ws[threadIdx.x] = w[threadIdx.x];
    __syncthreads();
    f2 acc[3][8];        // channel pairs
    float accb[3];
#pragma unroll
    for (int o = 0; o < 3; ++o) {
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[o][j] = 0ull;
        accb[o] = 0.0f;
    }
    const size_t total = (size_t)n * h * wd;
    const size_t i0 = blockIdx.x * chunk, i1 = i0 + chunk < total ? i0 + chunk : total;
    // row and column from the block's first pixel on, in 32 bits
    const uint64_t row0 = i0 / (uint32_t)wd;
    const uint32_t X0 = (uint32_t)(i0 - row0 * (uint32_t)wd), cnt = i1 > i0 ? (uint32_t)(i1 - i0) : 0;
    const uint32_t img0 = (uint32_t)(row0 / (uint32_t)h), Y0 = (uint32_t)(row0 - (uint64_t)img0 * (uint32_t)h);
    const uint32_t q0 = X0 + threadIdx.x, r0 = Y0 + q0 / (uint32_t)wd;
    uint32_t X = q0 % (uint32_t)wd, Y = r0 % (uint32_t)h, img = img0 + r0 / (uint32_t)h;
    const uint32_t stepY = 256u / (uint32_t)wd, stepX = 256u - stepY * (uint32_t)wd;
    // both tensors hold 16 channels: the elements of a row, and from one half of a pixel to the other
    const T* const xb = x.at(0, 0, 0, wn);
    T* const gb = gd.at(0, 0, 0, wn);
    const bool planar = gd.planar;
    const uint32_t row_e = 16u * (uint32_t)wn, half = planar ? 8u * (uint32_t)wn : 8u;
    const float* dp = drgb + 3 * (i0 + threadIdx.x);
    for (uint32_t p = threadIdx.x; p < cnt; p += 256, dp += 768) {
        const size_t at = ((size_t)img * (uint32_t)hn + Y) * row_e + X * (planar ? 8u : 16u);
        X += stepX;
        Y += stepY;
        if (X >= (uint32_t)wd) {
            X -= (uint32_t)wd;
            ++Y;
        }
        while (Y >= (uint32_t)h) {
            Y -= (uint32_t)h;
            ++img;
        }
        float v[16];
        ld8<T>(xb + at, v);
        ld8<T>(xb + at + half, v + 8);
        const float d[3] = {dp[0], dp[1], dp[2]};
        const f2 dd[3] = {f2_pack(d[0], d[0]), f2_pack(d[1], d[1]), f2_pack(d[2], d[2])};
        const f2* w2 = reinterpret_cast<const f2*>(ws);
        float out[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const f2 s = f2_fma(dd[2], w2[16 + j], f2_fma(dd[1], w2[8 + j], f2_mul(dd[0], w2[j])));
            float s0, s1;
            f2_unpack(s, s0, s1);
            out[2 * j] = v[2 * j] > 0.0f ? s0 : 0.0f;
            out[2 * j + 1] = v[2 * j + 1] > 0.0f ? s1 : 0.0f;
        }
        st8<T>(gb + at, out);
        st8<T>(gb + at + half, out + 8);
#pragma unroll
        for (int o = 0; o < 3; ++o) {
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[o][j] = f2_fma(dd[o], f2_pack(v[2 * j], v[2 * j + 1]), acc[o][j]);
            accb[o] += d[o];
        }
    }
    // the canvas margin
    if (hn != h || wn != wd) {
        float zero[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) zero[c] = 0.0f;
        const uint32_t rows = (uint32_t)n * hn;
        for (uint32_t r = blockIdx.x; r < rows; r += gridDim.x) {
            const int x0 = (int)(r % (uint32_t)hn) < h ? wd : 0;
            for (int X = x0 + (int)threadIdx.x; X < wn; X += blockDim.x) {
                st8<T>(gd.at(r, X, 0, wn), zero);
                st8<T>(gd.at(r, X, 8, wn), zero);
            }
        }
    }
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    auto put = [&](float a, int k) {
        for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if (lane == 0) red[wp][k] = a;
    };
#pragma unroll
    for (int o = 0; o < 3; ++o) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float a0, a1;
            f2_unpack(acc[o][j], a0, a1);
            put(a0, o * 16 + 2 * j);
            put(a1, o * 16 + 2 * j + 1);
        }
        put(accb[o], 48 + o);
    }
    __syncthreads();
    if (threadIdx.x < 51) {
        float a = red[0][threadIdx.x];
        for (int k = 1; k < (int)(blockDim.x / 32); ++k) a += red[k][threadIdx.x];
        part[blockIdx.x * 51 + threadIdx.x] = a;
    }
}

// ------------------------------------------------------------------ pooling backward
// ge[q][c] = (0.25 * gp[q/2][c] + gs[q][c]) * (e[q][c] > 0): a thread makes 8 channels of 2 x 2
// pixels, so each pooled gradient is read once and nine loads are in flight.  Bound by memory
// (16 channels of 16 x 256^2 pixels: 107 MB in 22 us; one pixel per thread 26; 32 and 64
// channels at levels 1 and 2: 16 -> 13.6 and 12 -> 8).
template <typename T>
__global__ void __launch_bounds__(256) pool_bwd_kernel(TView<const T> gp, TView<const T> gs, TView<const T> e,
                                                       TView<T> ge, int c, int rows2, int w) {
    const uint32_t w2 = w / 2, ng = c / 8, u = blockIdx.x * 256u + threadIdx.x;
    if (u >= w2 * ng) return;
    // neighbouring threads take neighbouring memory: pixels of a plane, or channels of a pixel
    const uint32_t grp = ge.planar ? u / w2 : u % ng, X = ge.planar ? u - grp * w2 : u / ng;
    const int cg = 8 * (int)grp;
    for (int r2 = blockIdx.y; r2 < rows2; r2 += gridDim.y) {
        float a[8], b[4][8], m[4][8];
        ld8<T>(gp.at(r2, X, cg, w2), a);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            ld8<T>(gs.at(2 * (size_t)r2 + (k >> 1), 2 * X + (k & 1), cg, w), b[k]);
            ld8<T>(e.at(2 * (size_t)r2 + (k >> 1), 2 * X + (k & 1), cg, w), m[k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int j = 0; j < 8; ++j) b[k][j] = m[k][j] > 0.0f ? fmaf(0.25f, a[j], b[k][j]) : 0.0f;
            st8<T>(ge.at(2 * (size_t)r2 + (k >> 1), 2 * X + (k & 1), cg, w), b[k]);
        }
    }
}

// ------------------------------------------------------------------ loss and optimizer
// Four values per thread and step where the pointers allow (vec), else one.
__global__ void __launch_bounds__(256) l1_partial_kernel(const float* y, const float* t, int64_t n, float* dy,
                                                         float inv_n, float* part, int vec) {
    __shared__ float red[256];
    float s = 0.0f;
    auto one = [&](float a, float b, float& g) {
        const float d = a - b;
        s += fabsf(d);
        g = d > 0.0f ? inv_n : (d < 0.0f ? -inv_n : 0.0f);
    };
    const int64_t n4 = vec ? n / 4 : 0, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
#pragma unroll 2
    for (int64_t i = i0; i < n4; i += stride) {
        const float4 a = reinterpret_cast<const float4*>(y)[i], b = reinterpret_cast<const float4*>(t)[i];
        float4 g;
        one(a.x, b.x, g.x);
        one(a.y, b.y, g.y);
        one(a.z, b.z, g.z);
        one(a.w, b.w, g.w);
        if (dy) reinterpret_cast<float4*>(dy)[i] = g;
    }
    for (int64_t i = 4 * n4 + i0; i < n; i += stride) {
        float g;
        one(y[i], t[i], g);
        if (dy) dy[i] = g;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void l1_final_kernel(const float* part, int nb, double inv_n, float* loss) {
    __shared__ double red[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < nb; i += 256) s += part[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) loss[0] = (float)(red[0] * inv_n);
}

// Where a loss puts its LOSS_PARTS partial sums: the caller's memory (a net's, one call at a time
// anyway) or, for the free-standing losses, 2 KB of its own that the stream's order gives and
// takes back -- calls on other streams, threads and devices have theirs, and a captured call's
// belong to its graph.  They come from a pool per device that keeps its memory between calls (one
// reservation of the driver's, 32 MB, holds those of 16K calls in flight); emptied at every
// synchronisation it cost 170 us a call, kept 3 us over one buffer shared by all calls (a small
// loss waited for: 23 -> 26 us), which raced.
struct LossParts {
    static constexpr size_t BYTES = LOSS_PARTS * sizeof(float);
    float* p;
    cudaStream_t s;
    bool own = false;
    LossParts(float* given, cudaStream_t stream) : p(given), s(stream) {}
    LossParts(const LossParts&) = delete;
    LossParts& operator=(const LossParts&) = delete;
    ~LossParts() {
        if (own) cudaFreeAsync(p, s);
    }
    nrv_status take() {
        if (p) return NRV_OK;
        const cudaMemPool_t pool = device_pool();
        if (!pool || cudaMallocFromPoolAsync((void**)&p, BYTES, pool, s) != cudaSuccess) {
            cudaGetLastError();
            if (cudaMallocAsync((void**)&p, BYTES, s) != cudaSuccess) {
                p = nullptr;
                cudaGetLastError();
                return fail(NRV_ERR_OOM, "no device memory for a loss's partial sums");
            }
        }
        own = true;
        return NRV_OK;
    }
    // the current device's pool, made on first use; null where there is none
    static cudaMemPool_t device_pool() {
        static std::mutex mu;
        static cudaMemPool_t pools[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
        std::lock_guard<std::mutex> lock(mu);
        if (!pools[dev]) {
            cudaMemPoolProps props;
            memset(&props, 0, sizeof(props));
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t pool = nullptr;
            if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) return nullptr;
            uint64_t keep = ~0ull;
            int no = 0;   // one stream's call never waits for another's memory
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
            cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &no);
            pools[dev] = pool;
        }
        return pools[dev];
    }
};

nrv_status launch_l1(const float* y, const float* t, int64_t n, float* loss, float* dy,
                     cudaStream_t s, float* part) {
    LossParts parts(part, s);
    NRV_TRY(parts.take());
    const int vec = (((uintptr_t)y | (uintptr_t)t | (uintptr_t)dy) & 15) == 0;
    l1_partial_kernel<<<LOSS_PARTS, 256, 0, s>>>(y, t, n, dy, (float)(1.0 / (double)n), parts.p, vec);
    NRV_CHECK_LAUNCH();
    l1_final_kernel<<<1, 256, 0, s>>>(parts.p, LOSS_PARTS, 1.0 / (double)n, loss);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

// Reconstruction + total-variation loss (Eq. 1 without its perceptual term) on RGB images
// y, t [n][h][w][3]: l1 mean|y - t| + l2 mean (y - t)^2 + tv (mean over horizontal neighbour
// pairs of |y_right - y| + mean over vertical pairs of |y_below - y|), each mean over its
// own count.  dy (if not null) is the gradient, sign(0) = 0.  Partial sums per block, summed
// in a fixed order (deterministic).
__global__ void recon_partial_kernel(const float* __restrict__ y, const float* __restrict__ t,
                                     int64_t n, int h, int w, float* dy, float l1, float l2,
                                     float tv, float inv_n, float inv_nh, float inv_nv,
                                     float* part) {
    __shared__ float red[256];
    auto sgn = [](float d) { return d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f); };
    const int64_t row = 3 * (int64_t)w;
    float s = 0.0f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float yi = y[i], d = yi - t[i];
        const int x = (int)((i / 3) % w), yy = (int)((i / row) % h);
        float l = l1 * fabsf(d) * inv_n + l2 * d * d * inv_n;
        float g = l1 * sgn(d) * inv_n + 2.0f * l2 * d * inv_n;
        if (tv != 0.0f) {
            if (x + 1 < w) {
                const float e = y[i + 3] - yi;
                l += tv * fabsf(e) * inv_nh;
                g -= tv * sgn(e) * inv_nh;
            }
            if (x > 0) g += tv * sgn(yi - y[i - 3]) * inv_nh;
            if (yy + 1 < h) {
                const float e = y[i + row] - yi;
                l += tv * fabsf(e) * inv_nv;
                g -= tv * sgn(e) * inv_nv;
            }
            if (yy > 0) g += tv * sgn(yi - y[i - row]) * inv_nv;
        }
        s += l;
        if (dy) dy[i] = g;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

nrv_status launch_recon(const float* y, const float* t, int n_img, int h, int w,
                        const nrv_loss_weights& wt, float* loss, float* dy, cudaStream_t s, float* part) {
    LossParts parts(part, s);
    NRV_TRY(parts.take());
    const int64_t n = (int64_t)n_img * h * w * 3;
    const double nh = (double)n_img * h * (w - 1) * 3, nv = (double)n_img * (h - 1) * w * 3;
    recon_partial_kernel<<<LOSS_PARTS, 256, 0, s>>>(y, t, n, h, w, dy, wt.l1, wt.l2, wt.tv,
                                            (float)(1.0 / (double)n), nh > 0 ? (float)(1.0 / nh) : 0.0f,
                                            nv > 0 ? (float)(1.0 / nv) : 0.0f, parts.p);
    NRV_CHECK_LAUNCH();
    l1_final_kernel<<<1, 256, 0, s>>>(parts.p, LOSS_PARTS, 1.0, loss);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int64_t n, float lr,
                            float b1, float b2, float eps, float bc1, float bc2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    }
}

nrv_status launch_adam(float* p, const float* g, float* m, float* v, int64_t n, int step, float lr,
                       float b1, float b2, float eps, cudaStream_t s) {
    const float bc1 = (float)(1.0 - pow((double)b1, step));
    const float bc2 = (float)(1.0 - pow((double)b2, step));
    int blocks = (int)((n + 255) / 256);
    if (blocks > 152 * 8) blocks = 152 * 8;
    adam_kernel<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, bc1, bc2);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

// ------------------------------------------------------------------ backward orchestration
static int blocks_for(size_t work, int per = 256) {
    size_t b = (work + per - 1) / per;
    if (b > 152 * 32) b = 152 * 32;
    return (int)(b > 0 ? b : 1);
}

// Gradient tensors of a backward pass, each with a buffer of its own: the weight gradients on
// the side stream may read one long after the chain has gone on.
enum Grad {
    G_D0B, G_D0A, G_CAT0, G_E0B, G_E0A, G_D1B, G_D1A, G_CAT1, G_E1B, G_E1A, G_P0, G_D2B, G_D2A, G_CAT2,
    G_E2B, G_E2A, G_P1, G_E3B, G_E3A, G_P2, NUM_GRADS
};
static const int kGradLevel[NUM_GRADS] = {0, 0, 0, 0, 0, 1, 1, 1, 1, 1, 1, 2, 2, 2, 2, 2, 2, 3, 3, 3};
static const int kGradC[NUM_GRADS] = {16, 16, 32, 16, 16, 32, 32, 64, 32, 32, 16, 64, 64, 128, 64, 64, 32,
                                      128, 128, 64};

// The stream and events that the weight gradients run on, created on first use.
static nrv_status net_side_stream(Net* net) {
    if (net->side) return NRV_OK;
    for (cudaEvent_t& e : net->side_ev)
        if (!e) NRV_CHECK_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    NRV_CHECK_CUDA(cudaStreamCreateWithFlags(&net->side, cudaStreamNonBlocking));
    return NRV_OK;
}

template <typename T>
struct Bwd {
    Net* net;
    cudaStream_t s;
    const Geo& g;
    float* dparams;
    Partials parts;
    cudaStream_t sw;         // weight gradients (the side stream, or s itself)
    T* G[NUM_GRADS];         // gradient tensors

    Bwd(Net* net_, cudaStream_t s_, const Geo& g_, float* dp)
        : net(net_), s(s_), g(g_), dparams(dp), parts(&net_->partial), sw(s_) {}

    T* A(int a) const { return reinterpret_cast<T*>((char*)net->acts.p + net->act_off[a]); }
    // saved activations: row-planar in BF16 (the tensor-core layout), NHWC in FP32
    TView<const T> CA(int a) const {
        return TView<const T>{A(a), net->act_c[a], sizeof(T) == 2 ? 1 : 0};
    }

    nrv_status wgrad_conv(int l, TView<const T> gpre, TView<const T> x1, int c1, TView<const T> x2,
                          int c2, int level) {
        const Layer& L = net->layers[l];
        const int cin = c1 + c2;
        if (sizeof(T) == 2) {
            // BF16: the weight gradient on the tensor cores, the bias gradient beside it
            const bool fits = gpre.planar && !gpre.coff && gpre.ld == L.cout && x1.planar &&
                              !x1.coff && x1.ld == c1 &&
                              (!c2 || (x2.planar && !x2.coff && x2.ld == c2));
            if (fits) {
                int max_split = 0, nsplit = 0;
                NRV_TRY(tc_wgrad_splits(net, l, g.n, g.h[level], g.w[level], &max_split));
                const size_t per_split = (size_t)L.cout * 9 * cin, mark = parts.used;
                float* part = parts.take(max_split * per_split);
                float* partb = parts.take((size_t)max_split * L.cout);
                if (!part || !partb) return fail(NRV_ERR_STATE, "partial sums");
                const nrv_status st = tc_wgrad(net, l, gpre.p, x1.p, c1, c2 ? x2.p : nullptr, c2, g.n,
                                               g.h[level], g.w[level], part, max_split * per_split,
                                               partb, &nsplit, sw);
                if (st == NRV_OK) {
                    parts.add(ReduceSeg{part, nsplit, per_split, (int)per_split, 0, L.cout, cin, L.cin,
                                        dparams + L.woff});
                    parts.add(ReduceSeg{partb, nsplit, (size_t)L.cout, L.cout, 2, L.cout, cin, L.cin,
                                        dparams + L.boff});
                    return NRV_OK;
                }
                if (st != NRV_ERR_UNSUPPORTED) return st;
                clear_error();
                parts.used = mark;
            }
        }
        const int h = g.h[level], w = g.w[level];
        const size_t per_split = (size_t)L.cout * 9 * cin;
        int nblk, tpb = 0;
        if (sizeof(T) == 4) nblk = f32_wgrad_splits(cin, L.cout, g.n, h, w);
        else nblk = simt_splits(L.cout, cin, h, w, &tpb);
        float* part = parts.take(nblk * per_split);
        float* partb = parts.take((size_t)nblk * L.cout);
        if (!part || !partb) return fail(NRV_ERR_STATE, "partial sums");
        if constexpr (sizeof(T) == 4) {
            NRV_TRY(f32_wgrad(gpre.p, L.cout, x1.p, c1, x2.p, c2, g.n, h, w, part, partb, sw));
        } else {
            const int CG = cin < 16 ? cin : 16;
            if (cin % CG || (c2 && c1 % CG) || L.cout % 16)
                return fail(NRV_ERR_UNSUPPORTED, "weight gradient: channel groups");
            wgrad3_kernel<T><<<dim3((unsigned)nblk, L.cout / 16, cin / CG), WG_THREADS, 0, sw>>>(
                gpre, L.cout, x1, c1, x2, c2, g.n, h, w, wgrad_tile_width(w), tpb, part, partb);
            NRV_CHECK_LAUNCH();
        }
        parts.add(ReduceSeg{part, nblk, per_split, (int)per_split, 0, L.cout, cin, L.cin, dparams + L.woff});
        parts.add(ReduceSeg{partb, nblk, (size_t)L.cout, L.cout, 2, L.cout, cin, L.cin, dparams + L.boff});
        return NRV_OK;
    }

    // Splits of a layer's weight gradient on the CUDA cores in BF16: about four blocks per SM in
    // all, each a contiguous run of tpb tiles.
    int simt_splits(int cout, int cin, int h, int w, int* tpb) const {
        const int CG = cin < 16 ? cin : 16, TW = wgrad_tile_width(w), R = WG_TILE / TW;
        const long long ntiles = (long long)g.n * ((h + R - 1) / R) * ((w + TW - 1) / TW);
        const int groups = (cout / 16) * (cin / CG) > 0 ? (cout / 16) * (cin / CG) : 1;
        long long nblk = (152LL * 4 + groups - 1) / groups;
        if (nblk > ntiles) nblk = ntiles;
        if (nblk < 1) nblk = 1;
        *tpb = (int)((ntiles + nblk - 1) / nblk);
        return (int)((ntiles + *tpb - 1) / *tpb);
    }
    int simt_up_splits(int cin, size_t npx, size_t* chunk) const {
        const int groups = cin / 16;
        size_t nch = (608 + groups - 1) / groups;
        const size_t maxch = (npx + 127) / 128;
        if (nch > maxch) nch = maxch;
        if (nch < 1) nch = 1;
        *chunk = (npx + nch - 1) / nch;
        return (int)((npx + *chunk - 1) / *chunk);
    }
    // Floats of partial sums that layer l takes, its pixels at `level` of g: one path's, the larger
    // of the two in BF16 (the CUDA cores are for layers that the tensor cores refuse).
    nrv_status need(int l, int level, size_t* floats) const {
        const Layer& L = net->layers[l];
        const int h = g.h[level], w = g.w[level];
        const bool conv = L.kind == CONV3;
        const int cin = l == L_E0A ? net->c0p : L.cin;
        const size_t per = (conv ? 9 : 4) * (size_t)L.cout * cin, bias = conv ? L.cout : 4 * L.cout;
        auto room = [&](size_t ns) { return (ns * per + 31) / 32 * 32 + (ns * bias + 31) / 32 * 32; };
        if (sizeof(T) == 4) {
            *floats = room(conv ? f32_wgrad_splits(cin, L.cout, g.n, h, w)
                                : f32_wgrad_up_splits(cin, L.cout, g.n, h, w));
            return NRV_OK;
        }
        int tpb, tc = 0;
        size_t chunk;
        NRV_TRY(tc_wgrad_splits(net, l, g.n, h, w, &tc));
        const size_t simt = conv ? simt_splits(L.cout, cin, h, w, &tpb) : simt_up_splits(cin, g.px(level), &chunk);
        *floats = room(simt > (size_t)tc ? simt : (size_t)tc);
        return NRV_OK;
    }

    nrv_status dgrad_conv(int l, TView<const T> gpre, TView<T> out, TView<const T> mask,
                          int level) {
        // BF16: on the tensor cores (a 3x3 conv with the flipped, transposed kernel)
        if (sizeof(T) == 2) {
            const Layer& L = net->layers[l];
            const bool fits = gpre.planar && out.planar && !gpre.coff && !out.coff &&
                              gpre.ld == L.cout && out.ld == L.cin &&
                              (!mask.p || (mask.planar && !mask.coff && mask.ld == L.cin));
            if (fits) {
                const nrv_status st = tc_dgrad(net, l, gpre.p, out.p, mask.p, g.n, g.h[level],
                                               g.w[level], s);
                if (st != NRV_ERR_UNSUPPORTED) return st;
                clear_error();
            }
        }
        if constexpr (sizeof(T) == 4) {
            return f32_conv3(gpre.p, net->layers[l].cout, nullptr, 0,
                             (const float*)net->wtf32.p + net->wf_off[l], nullptr, 0, mask.p, out.p,
                             net->layers[l].cin, g.n, g.h[level], g.w[level], s);
        } else {
            // this translation unit has its own instance of the kernel template
            static bool attr = false;
            if (!attr) {
                NRV_CHECK_CUDA(cudaFuncSetAttribute(conv3_simt_kernel<T>,
                                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    9 * 128 * 16 * 4));
                attr = true;
            }
            const Layer& L = net->layers[l];
            Conv3Args<T> a;
            a.x1 = gpre;
            a.c1 = L.cout;
            a.x2 = TView<const T>{nullptr, 0};
            a.c2 = 0;
            a.w = (const float*)net->wtf32.p + net->wf_off[l];
            a.bias = nullptr;
            a.y = out;
            a.cout = L.cin;
            a.n = g.n; a.h = g.h[level]; a.w_ = g.w[level];
            a.relu = 0;
            a.mask = mask;
            const size_t npx = g.px(level);
            dim3 grid((unsigned)((npx + 127) / 128), L.cin / 16);
            conv3_simt_kernel<T><<<grid, 128, (size_t)9 * L.cout * 16 * 4, s>>>(a);
            NRV_CHECK_LAUNCH();
            return NRV_OK;
        }
    }

    // weight and bias gradient of transposed conv l: x at level_in, gout one level up
    nrv_status wgrad_up(int l, TView<const T> x, TView<const T> gout, int level_in) {
        const Layer& L = net->layers[l];
        if (sizeof(T) == 2 && x.planar && !x.coff && x.ld == L.cin && gout.planar &&
            gout.ld % 8 == 0 && gout.coff % 8 == 0 && gout.coff + L.cout <= gout.ld) {
            // BF16: on the tensor cores, the bias gradient beside it
            int max_split = 0, nsplit = 0;
            NRV_TRY(tc_wgrad_splits(net, l, g.n, g.h[level_in], g.w[level_in], &max_split));
            const size_t per_split = (size_t)L.cin * 4 * L.cout, mark = parts.used;
            float* part = parts.take(max_split * per_split);
            float* partb = parts.take((size_t)max_split * 4 * L.cout);
            if (!part || !partb) return fail(NRV_ERR_STATE, "partial sums");
            const nrv_status st = tc_wgrad_up(net, l, gout.p, gout.ld, gout.coff, x.p, g.n,
                                              g.h[level_in], g.w[level_in], part,
                                              max_split * per_split, partb, &nsplit, sw);
            if (st == NRV_OK) {
                // bias, per split: the four kernel positions' sums of each channel
                parts.add(ReduceSeg{part, nsplit, per_split, (int)per_split, 1, L.cout, L.cin, L.cin,
                                    dparams + L.woff});
                parts.add(ReduceSeg{partb, nsplit, (size_t)4 * L.cout, L.cout, 3, L.cout, L.cin, L.cin,
                                    dparams + L.boff});
                return NRV_OK;
            }
            if (st != NRV_ERR_UNSUPPORTED) return st;
            clear_error();
            parts.used = mark;
        }
        const size_t npx = g.px(level_in);
        const int K = 4 * L.cout;
        int nch;
        size_t chunk = 0;
        if (sizeof(T) == 4) nch = f32_wgrad_up_splits(L.cin, L.cout, g.n, g.h[level_in], g.w[level_in]);
        else nch = simt_up_splits(L.cin, npx, &chunk);
        float* part = parts.take((size_t)nch * L.cin * K);
        float* partb = parts.take((size_t)nch * K);
        if (!part || !partb) return fail(NRV_ERR_STATE, "partial sums");
        if constexpr (sizeof(T) == 4) {
            NRV_TRY(f32_wgrad_up(x.p, L.cin, gout.p + gout.coff, gout.ld, L.cout, g.n, g.h[level_in],
                                 g.w[level_in], part, partb, sw));
        } else {
            wgrad_up_kernel<T><<<dim3((unsigned)nch, L.cin / 16), 256, 0, sw>>>(
                x, L.cin, gout, L.cout, g.n, g.h[level_in], g.w[level_in], chunk, part, partb);
            NRV_CHECK_LAUNCH();
        }
        parts.add(ReduceSeg{part, nch, (size_t)L.cin * K, L.cin * K, 1, L.cout, L.cin, L.cin,
                            dparams + L.woff});
        parts.add(ReduceSeg{partb, nch, (size_t)K, L.cout, 3, L.cout, L.cin, L.cin, dparams + L.boff});
        return NRV_OK;
    }

    // data gradient of transposed conv l at level_in, zeroed where the layer's input xm (a
    // ReLU output) is not positive
    nrv_status dgrad_up(int l, TView<const T> gout, TView<const T> xm, TView<T> gx, int level_in) {
        const Layer& L = net->layers[l];
        if (sizeof(T) == 2 && gout.planar && gx.planar && !gx.coff && gx.ld == L.cin && xm.planar &&
            !xm.coff && xm.ld == L.cin) {
            // BF16: on the tensor cores
            const nrv_status st = tc_updgrad(net, l, gout.p, gout.ld, gout.coff, xm.p, gx.p, g.n,
                                             g.h[level_in], g.w[level_in], s);
            if (st != NRV_ERR_UNSUPPORTED) return st;
            clear_error();
        }
        if constexpr (sizeof(T) == 4) {
            return f32_upconv_dgrad(gout.p + gout.coff, gout.ld, L.cout,
                                    (const float*)net->wtf32.p + net->wf_off[l], xm.p, gx.p, L.cin, g.n,
                                    g.h[level_in], g.w[level_in], s);
        } else {
            dim3 grid((unsigned)((g.px(level_in) + 127) / 128), L.cin / 16);
            upconv2_dgrad_kernel<T><<<grid, 128, (size_t)4 * 16 * L.cout * 4, s>>>(
                gout, L.cout, (const float*)net->wf32.p + net->wf_off[l], L.cin, xm, gx, g.n,
                g.h[level_in], g.w[level_in]);
            NRV_CHECK_LAUNCH();
            return NRV_OK;
        }
    }

    nrv_status pool_bwd(TView<const T> gp, TView<const T> gs, int e, TView<T> ge, int level) {
        const int c = net->act_c[e];
        // the levels a pool reads are of even size: the canvas is a multiple of 8
        const long long rows2 = (long long)g.n * (g.h[level] / 2);
        const unsigned bx = (unsigned)((g.w[level] / 2 * (c / 8) + 255) / 256);
        pool_bwd_kernel<T><<<dim3(bx, (unsigned)(rows2 < 65535 ? rows2 : 65535)), 256, 0, s>>>(
            gp, gs, CA(e), ge, c, (int)rows2, g.w[level]);
        NRV_CHECK_LAUNCH();
        return NRV_OK;
    }

    // gradients: row-planar in BF16 (the tensor-core layout), NHWC in FP32; coff selects a
    // channel range (the skip half of a concatenation's gradient)
    static constexpr int kPlanar = sizeof(T) == 2 ? 1 : 0;
    static TView<T> V(T* p, int ld) { return TView<T>{p, ld, kPlanar}; }
    static TView<const T> C(T* p, int ld, int coff = 0) {
        return TView<const T>{p, ld, kPlanar, coff};
    }

    // The data gradients form a chain on s; each weight gradient needs one link of it and
    // nothing needs the weight gradients until the end, so they run beside it on sw: point()
    // lets sw go on once what s holds so far is done.
    int npoint = 0;
    nrv_status point() {
        if (sw == s) return NRV_OK;
        if (npoint >= Net::SIDE_EVENTS) return fail(NRV_ERR_STATE, "backward events");
        NRV_CHECK_CUDA(cudaEventRecord(net->side_ev[npoint], s));
        NRV_CHECK_CUDA(cudaStreamWaitEvent(sw, net->side_ev[npoint], 0));
        ++npoint;
        return NRV_OK;
    }
    // s continues after everything on sw
    nrv_status join() {
        if (sw == s) return NRV_OK;
        NRV_CHECK_CUDA(cudaEventRecord(net->side_ev[Net::SIDE_EVENTS], sw));
        NRV_CHECK_CUDA(cudaStreamWaitEvent(s, net->side_ev[Net::SIDE_EVENTS], 0));
        return NRV_OK;
    }

    nrv_status run(const float* drgb, const T* netin) {
        // every layer's partial sums side by side, reduced by one launch at the end
        static const int lvl[NUM_LAYERS] = {0, 0, 1, 1, 2, 2, 3, 3, 3, 2, 2, 2, 1, 1, 1, 0, 0, 0};
        const size_t tot = (size_t)g.n * net->geo_H * net->geo_W;
        size_t hch = 608, hchunk = (tot + hch - 1) / hch;
        if (hchunk < 64) hchunk = 64;
        hch = (tot + hchunk - 1) / hchunk;
        size_t floats = (hch * 51 + 31) / 32 * 32;
        for (int l = 0; l < L_HEAD; ++l) {
            size_t f = 0;
            NRV_TRY(need(l, lvl[l], &f));
            floats += f;
        }
        NRV_TRY(net->partial.ensure(floats * sizeof(float)));
        NRV_TRY(net_side_stream(net));
        sw = net->side;
        const nrv_status st = layers_bwd(drgb, netin, hch, hchunk);
        const nrv_status fs = st == NRV_OK ? parts.flush(sw) : st;
        const nrv_status js = join();   // also after a failure: nothing runs on past this call
        return fs != NRV_OK ? fs : js;
    }

    nrv_status layers_bwd(const float* drgb, const T* netin, size_t hch, size_t hchunk) {
        const TView<const T> none{nullptr, 0};
        const int H = net->geo_H, Wd = net->geo_W;
        // head
        const Layer& Lh = net->layers[L_HEAD];
        {
            float* part = parts.take(hch * 51);
            if (!part) return fail(NRV_ERR_STATE, "partial sums");
            head_bwd_kernel<T><<<(unsigned)hch, 256, 0, s>>>(
                drgb, (const float*)net->params.p + Lh.woff, CA(A_D0B), V(G[G_D0B], 16), g.n, g.h[0], g.w[0],
                H, Wd, hchunk, part);
            NRV_CHECK_LAUNCH();
            // weight (48) and bias (3) are consecutive in the parameter vector
            if (Lh.boff != Lh.woff + 48) return fail(NRV_ERR_STATE, "head parameter layout");
            parts.add(ReduceSeg{part, (int)hch, 51, 51, 2, 3, 16, 16, dparams + Lh.woff});
        }
        NRV_TRY(point());
        // level 0 decoder
        NRV_TRY(wgrad_conv(L_D0B, C(G[G_D0B], 16), CA(A_D0A), 16, none, 0, 0));
        NRV_TRY(dgrad_conv(L_D0B, C(G[G_D0B], 16), V(G[G_D0A], 16), CA(A_D0A), 0));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_D0A, C(G[G_D0A], 16), CA(A_UP1), 16, CA(A_E0B), 16, 0));
        NRV_TRY(dgrad_conv(L_D0A, C(G[G_D0A], 16), V(G[G_CAT0], 32), none, 0));
        NRV_TRY(point());
        NRV_TRY(wgrad_up(L_UP1, CA(A_D1B), C(G[G_CAT0], 32), 1));
        NRV_TRY(dgrad_up(L_UP1, C(G[G_CAT0], 32), CA(A_D1B), V(G[G_D1B], 32), 1));
        NRV_TRY(point());
        // level 1 decoder
        NRV_TRY(wgrad_conv(L_D1B, C(G[G_D1B], 32), CA(A_D1A), 32, none, 0, 1));
        NRV_TRY(dgrad_conv(L_D1B, C(G[G_D1B], 32), V(G[G_D1A], 32), CA(A_D1A), 1));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_D1A, C(G[G_D1A], 32), CA(A_UP2), 32, CA(A_E1B), 32, 1));
        NRV_TRY(dgrad_conv(L_D1A, C(G[G_D1A], 32), V(G[G_CAT1], 64), none, 1));
        NRV_TRY(point());
        NRV_TRY(wgrad_up(L_UP2, CA(A_D2B), C(G[G_CAT1], 64), 2));
        NRV_TRY(dgrad_up(L_UP2, C(G[G_CAT1], 64), CA(A_D2B), V(G[G_D2B], 64), 2));
        NRV_TRY(point());
        // level 2 decoder
        NRV_TRY(wgrad_conv(L_D2B, C(G[G_D2B], 64), CA(A_D2A), 64, none, 0, 2));
        NRV_TRY(dgrad_conv(L_D2B, C(G[G_D2B], 64), V(G[G_D2A], 64), CA(A_D2A), 2));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_D2A, C(G[G_D2A], 64), CA(A_UP3), 64, CA(A_E2B), 64, 2));
        NRV_TRY(dgrad_conv(L_D2A, C(G[G_D2A], 64), V(G[G_CAT2], 128), none, 2));
        NRV_TRY(point());
        NRV_TRY(wgrad_up(L_UP3, CA(A_E3B), C(G[G_CAT2], 128), 3));
        NRV_TRY(dgrad_up(L_UP3, C(G[G_CAT2], 128), CA(A_E3B), V(G[G_E3B], 128), 3));
        NRV_TRY(point());
        // bottom level
        NRV_TRY(wgrad_conv(L_E3B, C(G[G_E3B], 128), CA(A_E3A), 128, none, 0, 3));
        NRV_TRY(dgrad_conv(L_E3B, C(G[G_E3B], 128), V(G[G_E3A], 128), CA(A_E3A), 3));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_E3A, C(G[G_E3A], 128), CA(A_P2), 64, none, 0, 3));
        NRV_TRY(dgrad_conv(L_E3A, C(G[G_E3A], 128), V(G[G_P2], 64), none, 3));
        // level 2 encoder: the skip gradient is channels 64..127 of the concatenation's
        NRV_TRY(pool_bwd(C(G[G_P2], 64), C(G[G_CAT2], 128, 64), A_E2B, V(G[G_E2B], 64), 2));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_E2B, C(G[G_E2B], 64), CA(A_E2A), 64, none, 0, 2));
        NRV_TRY(dgrad_conv(L_E2B, C(G[G_E2B], 64), V(G[G_E2A], 64), CA(A_E2A), 2));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_E2A, C(G[G_E2A], 64), CA(A_P1), 32, none, 0, 2));
        NRV_TRY(dgrad_conv(L_E2A, C(G[G_E2A], 64), V(G[G_P1], 32), none, 2));
        // level 1 encoder: channels 32..63
        NRV_TRY(pool_bwd(C(G[G_P1], 32), C(G[G_CAT1], 64, 32), A_E1B, V(G[G_E1B], 32), 1));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_E1B, C(G[G_E1B], 32), CA(A_E1A), 32, none, 0, 1));
        NRV_TRY(dgrad_conv(L_E1B, C(G[G_E1B], 32), V(G[G_E1A], 32), CA(A_E1A), 1));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_E1A, C(G[G_E1A], 32), CA(A_P0), 16, none, 0, 1));
        NRV_TRY(dgrad_conv(L_E1A, C(G[G_E1A], 32), V(G[G_P0], 16), none, 1));
        // level 0 encoder: channels 16..31
        NRV_TRY(pool_bwd(C(G[G_P0], 16), C(G[G_CAT0], 32, 16), A_E0B, V(G[G_E0B], 16), 0));
        NRV_TRY(point());
        NRV_TRY(wgrad_conv(L_E0B, C(G[G_E0B], 16), CA(A_E0A), 16, none, 0, 0));
        NRV_TRY(dgrad_conv(L_E0B, C(G[G_E0B], 16), V(G[G_E0A], 16), CA(A_E0A), 0));
        NRV_TRY(point());
        return wgrad_conv(L_E0A, C(G[G_E0A], 16), C(const_cast<T*>(netin), net->c0p), net->c0p, none, 0, 0);
    }

    // one layer's weight gradient alone, on s
    template <typename Fn>
    nrv_status alone(int l, Fn fn) {
        size_t floats = 0;
        NRV_TRY(need(l, 0, &floats));
        NRV_TRY(net->partial.ensure(floats * sizeof(float)));
        NRV_TRY(fn());
        return parts.flush(s);
    }
};

// The training forward keeps its input pointer for the first layer's weight gradient.

nrv_status net_layer_wgrad(Net* net, int l, const void* dy, const void* x1, const void* x2, int n,
                           int h, int w, nrv_prec prec, float* dgrad, cudaStream_t s) {
    const Layer& L = net->layers[l];
    if (L.kind == UPCONV2) {
        // transposed conv: x1 at (n, h, w), dy at (n, 2h, 2w)
        if (x2) return fail(NRV_ERR_ARG, "layer %s: x2 must be NULL", L.name);
        Geo g;
        memset(&g, 0, sizeof(g));
        g.n = n;
        g.h[0] = h;
        g.w[0] = w;
        if (prec == NRV_PREC_F32) {
            using T = float;
            Bwd<T> b(net, s, g, dgrad);
            return b.alone(l, [&] {
                return b.wgrad_up(l, TView<const T>{(const T*)x1, L.cin},
                                  TView<const T>{(const T*)dy, L.cout}, 0);
            });
        }
        if (prec != NRV_PREC_BF16) return fail(NRV_ERR_UNSUPPORTED, "weight gradients in F32 or BF16");
        using T = __nv_bfloat16;
        const size_t rows = (size_t)n * h;
        auto al = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
        const size_t bg = al(4 * rows * w * L.cout * 2), bx = al(rows * w * L.cin * 2);
        NRV_TRY(net->layer_ws.ensure(bg + bx));
        char* ws = (char*)net->layer_ws.p;
        T *pg = (T*)ws, *px = (T*)(ws + bg);
        const RelayoutJob jobs[2] = {{dy, pg, 2 * rows, 2 * w, L.cout}, {x1, px, rows, w, L.cin}};
        NRV_TRY(relayout_in(jobs, 2, 2, s));
        Bwd<T> b(net, s, g, dgrad);
        return b.alone(l, [&] {
            return b.wgrad_up(l, TView<const T>{px, L.cin, 1}, TView<const T>{pg, L.cout, 1}, 0);
        });
    }
    if (L.kind != CONV3) return fail(NRV_ERR_ARG, "layer %s has no weight gradient here", L.name);
    int c1 = l == L_E0A ? net->c0p : L.cin, c2 = 0;
    if (l == L_D2A || l == L_D1A || l == L_D0A) c1 = c2 = L.cin / 2;
    if ((c2 > 0) != (x2 != nullptr))
        return fail(NRV_ERR_ARG, "layer %s: x2 must be %s", L.name, c2 ? "given" : "NULL");
    Geo g;
    memset(&g, 0, sizeof(g));
    g.n = n;
    g.h[0] = h;
    g.w[0] = w;
    if (prec == NRV_PREC_F32) {
        using T = float;
        Bwd<T> b(net, s, g, dgrad);
        return b.alone(l, [&] {
            return b.wgrad_conv(l, TView<const T>{(const T*)dy, L.cout}, TView<const T>{(const T*)x1, c1},
                                c1, TView<const T>{(const T*)x2, c2}, c2, 0);
        });
    }
    if (prec != NRV_PREC_BF16) return fail(NRV_ERR_UNSUPPORTED, "weight gradients in F32 or BF16");
    // BF16: row-planar copies, as the backward pass keeps its tensors
    using T = __nv_bfloat16;
    const size_t rows = (size_t)n * h;
    auto al = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
    const size_t bg = al(rows * w * L.cout * 2), b1 = al(rows * w * c1 * 2), b2 = al(rows * w * c2 * 2);
    NRV_TRY(net->layer_ws.ensure(bg + b1 + b2));
    char* ws = (char*)net->layer_ws.p;
    T *pg = (T*)ws, *p1 = (T*)(ws + bg), *p2 = c2 ? (T*)(ws + bg + b1) : nullptr;
    const RelayoutJob jobs[3] = {{dy, pg, rows, w, L.cout}, {x1, p1, rows, w, c1}, {x2, p2, rows, w, c2}};
    NRV_TRY(relayout_in(jobs, 3, 2, s));
    Bwd<T> b(net, s, g, dgrad);
    return b.alone(l, [&] {
        return b.wgrad_conv(l, TView<const T>{pg, L.cout, 1}, TView<const T>{p1, c1, 1}, c1,
                            TView<const T>{p2, c2, 1}, c2, 0);
    });
}

nrv_status net_layer_dgrad(Net* net, int l, const void* dy, const void* mask, int n, int h, int w,
                           nrv_prec prec, void* dx, cudaStream_t s) {
    const Layer& L = net->layers[l];
    if (L.kind == UPCONV2) {
        // transposed conv: dy at (n, 2h, 2w), mask and dx at (n, h, w)
        if (!mask) return fail(NRV_ERR_ARG, "layer %s: the mask (the layer's input) is required", L.name);
        Geo g;
        memset(&g, 0, sizeof(g));
        g.n = n;
        g.h[0] = h;
        g.w[0] = w;
        if (prec == NRV_PREC_F32) {
            using T = float;
            Bwd<T> b(net, s, g, nullptr);
            return b.dgrad_up(l, TView<const T>{(const T*)dy, L.cout}, TView<const T>{(const T*)mask, L.cin},
                              TView<T>{(T*)dx, L.cin}, 0);
        }
        if (prec != NRV_PREC_BF16) return fail(NRV_ERR_UNSUPPORTED, "data gradients in F32 or BF16");
        using T = __nv_bfloat16;
        const size_t rows = (size_t)n * h;
        auto al = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
        const size_t bg = al(4 * rows * w * L.cout * 2), bm = al(rows * w * L.cin * 2),
                     bo = al(rows * w * L.cin * 2);
        NRV_TRY(net->layer_ws.ensure(bg + bm + bo));
        char* ws = (char*)net->layer_ws.p;
        T *pg = (T*)ws, *pm = (T*)(ws + bg), *po = (T*)(ws + bg + bm);
        NRV_TRY(relayout(dy, pg, 2 * rows, 2 * w, L.cout, 2, true, s));
        {
            // the caller's NHWC mask and gradient read and written in place
            TcExtra direct;
            direct.nhwc = true;
            const nrv_status st = tc_updgrad(net, l, pg, L.cout, 0, mask, dx, n, h, w, s, &direct);
            if (st != NRV_ERR_UNSUPPORTED) return st;
            clear_error();
        }
        NRV_TRY(relayout(mask, pm, rows, w, L.cin, 2, true, s));
        Bwd<T> b(net, s, g, nullptr);
        NRV_TRY(b.dgrad_up(l, TView<const T>{pg, L.cout, 1}, TView<const T>{pm, L.cin, 1},
                           TView<T>{po, L.cin, 1}, 0));
        return relayout(po, dx, rows, w, L.cin, 2, false, s);
    }
    if (L.kind != CONV3 || l == L_E0A)
        return fail(NRV_ERR_ARG, "layer %s has no data gradient here", L.name);
    Geo g;
    memset(&g, 0, sizeof(g));
    g.n = n;
    g.h[0] = h;
    g.w[0] = w;
    if (prec == NRV_PREC_F32) {
        using T = float;
        Bwd<T> b(net, s, g, nullptr);
        return b.dgrad_conv(l, TView<const T>{(const T*)dy, L.cout}, TView<T>{(T*)dx, L.cin},
                            TView<const T>{(const T*)mask, mask ? L.cin : 0}, 0);
    }
    if (prec != NRV_PREC_BF16) return fail(NRV_ERR_UNSUPPORTED, "data gradients in F32 or BF16");
    using T = __nv_bfloat16;
    const size_t rows = (size_t)n * h;
    auto al = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
    const size_t bg = al(rows * w * L.cout * 2), bm = mask ? al(rows * w * L.cin * 2) : 0,
                 bo = al(rows * w * L.cin * 2);
    NRV_TRY(net->layer_ws.ensure(bg + bm + bo));
    char* ws = (char*)net->layer_ws.p;
    T *pg = (T*)ws, *pm = mask ? (T*)(ws + bg) : nullptr, *po = (T*)(ws + bg + bm);
    NRV_TRY(relayout(dy, pg, rows, w, L.cout, 2, true, s));
    {
        // the caller's NHWC mask and gradient read and written in place
        TcExtra direct;
        direct.nhwc = true;
        const nrv_status st = tc_dgrad(net, l, pg, dx, mask, n, h, w, s, &direct);
        if (st != NRV_ERR_UNSUPPORTED) return st;
        clear_error();
    }
    if (mask) NRV_TRY(relayout(mask, pm, rows, w, L.cin, 2, true, s));
    Bwd<T> b(net, s, g, nullptr);
    NRV_TRY(b.dgrad_conv(l, TView<const T>{pg, L.cout, 1}, TView<T>{po, L.cin, 1},
                         TView<const T>{pm, mask ? L.cin : 0, mask ? 1 : 0}, 0));
    return relayout(po, dx, rows, w, L.cin, 2, false, s);
}

nrv_status net_backward(Net* net, const float* drgb, float* dparams, cudaStream_t s) {
    if (!net->saved) return fail(NRV_ERR_STATE, "backward without a preceding training forward");
    const Geo& g = net->geo;
    const size_t es = elem_size(net->act_prec);
    size_t off[NUM_GRADS], tot = 0;
    for (int k = 0; k < NUM_GRADS; ++k) {
        off[k] = tot;
        tot += (g.px(kGradLevel[k]) * kGradC[k] * es + 1023) / 1024 * 1024;
    }
    NRV_TRY(net->grads.ensure(tot));
    if (net->act_prec == NRV_PREC_F32) {
        Bwd<float> b(net, s, g, dparams);
        for (int k = 0; k < NUM_GRADS; ++k) b.G[k] = (float*)((char*)net->grads.p + off[k]);
        return b.run(drgb, (const float*)net->saved_in);
    }
    if (net->act_prec == NRV_PREC_BF16) {
        Bwd<__nv_bfloat16> b(net, s, g, dparams);
        for (int k = 0; k < NUM_GRADS; ++k) b.G[k] = (__nv_bfloat16*)((char*)net->grads.p + off[k]);
        return b.run(drgb, (const __nv_bfloat16*)net->saved_in);
    }
    return fail(NRV_ERR_UNSUPPORTED, "backward is available for FP32 and BF16 only");
}

}  // namespace nrv
