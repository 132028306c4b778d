// The FP32 network's convolutions (Sec. 3.3) on the CUDA cores: 3x3 convs, 2x2 stride-2
// transposed convs and the data gradients of both, as one implicit GEMM over NHWC tensors.
//
//   out[pixel][n] = bias[n] + sum_k in[pixel, k] * B[k][n]
//   mode 0  3x3 conv (or its data gradient):  k = (tap, c),     B = [tap][c][n]
//   mode 1  transposed conv:                  k = c,            n = (ab, o) scattered to the
//                                             output pixel (2y + a, 2x + b), B = [ab][c][o]
//   mode 2  its data gradient:                k = (ab, o) read at pixel (2y + a, 2x + b),
//                                             B = [ab][o][c]
//
// Bound by the FP32 pipe (18.7 GFLOP for a 512 x 512 frame: 0.245 ms at the measured 76.4
// TFLOP/s), so the design keeps everything else off it:
//  * fma.rn.f32x2: two output channels per instruction.  Its rate in FMAs is the scalar one's
//    (measured: 36.8 T lane-FMAs/s either way) but it takes half the issue slots, which go to
//    the shared-memory reads.
//  * A thread makes 8 pixels of one row x 8 output channels: per input channel and kernel row
//    10 pixel words and 6 weight quads feed 96 paired FMAs.
//  * A block of 256 threads stages 8 input channels at a time (the halo tile and their weights)
//    with 16-byte cp.async into one of two buffers while it works on the other.  In a row the
//    pixels of a group of 8 sit 32 bytes apart and groups 16 bytes further, so that the eight
//    groups a quarter-warp reads lie in eight different bank quads.
//  * Where the tiles of one image are fewer than the SMs (the deep levels), the input
//    channels are split over a cluster of KS blocks, whose sums are added through distributed
//    shared memory in rank order (deterministic).  The split decides the order of the sums, so
//    it follows from the image's size alone: images computed together come out as they do alone.
#include <atomic>

#include <cooperative_groups.h>
#include <string.h>

#include "f32.h"
#include "project.cuh"

namespace nrv {

namespace {

constexpr int NT = 256;
constexpr int CK = 8;    // input channels per stage

struct F32Args {
    const float *x1, *x2;       // NHWC sources; x2: the second half of a concatenation
    int ld1, c1, ld2;           // channels per stored pixel, channels taken from x1
    int cin;                    // input channels (mode 2: 4 C_out)
    int cdiv;                   // mode 2: C_out (channels per kernel position)
    const float* b;             // weights (see above)
    int ncols;                  // columns (mode 1: 4 C_out)
    int cout;                   // mode 1: C_out
    const float* bias;
    const float* mask;          // shaped like the output: zero where not positive
    int relu;
    float* y;
    int ldy;
    int n, h, w;                // pixels the tiles cover (modes 1, 2: the lower level)
    int tiles_x, tiles_y;
};

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
}

template <int MODE, int OCB, int TW, int NB>   // NB threads
struct F32Tile {
    static constexpr int HALO = MODE == 0 ? 1 : 0;
    static constexpr int TAPS = MODE == 0 ? 9 : 1;
    static constexpr int OG = OCB / 8;                 // channel groups
    static constexpr int GX = TW / 8;                  // pixel groups per row
    static constexpr int RQ = 8 / GX;                  // rows of a quarter-warp
    static constexpr int RW = RQ * (4 / OG);           // rows of a warp
    static constexpr int TH = RW * (NB / 32);
    static constexpr int COLS = TW + 2 * HALO, ROWS = TH + 2 * HALO;
    static constexpr int RAW = (COLS - 1) * 32 + ((COLS - 1) / 8) * 16 + 32;
    // two rows per quarter-warp: the second one 64 bytes off in the banks
    static constexpr int RS = RQ == 1 ? RAW : (RAW + 63) / 128 * 128 + 64;
    static constexpr int IN_BYTES = ROWS * RS;
    static constexpr int W_BYTES = TAPS * CK * OCB * 4;
    static constexpr int STAGE = IN_BYTES + W_BYTES;
    static constexpr int RED = NB * 64 * 4;            // a block's sums, for the cluster
    static constexpr int SMEM1 = 2 * STAGE;
    static constexpr int SMEMK = SMEM1 > RED ? SMEM1 : RED;
    static_assert(RS >= RAW && RS % 16 == 0 && (RQ == 1 || RS % 128 == 64), "row stride");
};

template <int MODE, int OCB, int TW, int NB>
__global__ void __launch_bounds__(NB, 512 / NB) conv_f32_kernel(const __grid_constant__ F32Args a) {
    using T = F32Tile<MODE, OCB, TW, NB>;
    namespace cg = cooperative_groups;
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t s0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = (lane & 7) % T::GX, rq = (lane & 7) / T::GX, qd = lane >> 3;
    const int ocg = qd % T::OG, row = warp * T::RW + (qd / T::OG) * T::RQ + rq;
    const int nt = blockIdx.y * OCB;
    const int tile = blockIdx.x;
    const int tx = tile % a.tiles_x, ty = (tile / a.tiles_x) % a.tiles_y, img = tile / (a.tiles_x * a.tiles_y);
    const int x0 = tx * TW, y0 = ty * T::TH;
    const int nst = a.cin / CK, ks = gridDim.z, kr = blockIdx.z;
    const int st0 = nst * kr / ks, st1 = nst * (kr + 1) / ks;

    auto load = [&](int st, int buf) {
        const uint32_t base = s0 + buf * T::STAGE;
        const int ch = st * CK;
        const float* src;
        int ld, yo = 0, xo = 0, sc = 1, hh = a.h, ww = a.w;
        if (MODE == 2) {
            const int ab = ch / a.cdiv;
            src = a.x1 + (ch - ab * a.cdiv);
            ld = a.ld1;
            yo = ab >> 1;
            xo = ab & 1;
            sc = 2;
        } else if (ch < a.c1) {
            src = a.x1 + ch;
            ld = a.ld1;
        } else {
            src = a.x2 + (ch - a.c1);
            ld = a.ld2;
        }
        for (int i = tid; i < T::ROWS * T::COLS * 2; i += NB) {
            const int q = i & 1, pp = i >> 1, r = pp / T::COLS, p = pp - r * T::COLS;
            const int y = y0 + r - T::HALO, x = x0 + p - T::HALO;
            const bool ok = (unsigned)y < (unsigned)hh && (unsigned)x < (unsigned)ww;
            const float* s = src;
            if (ok) s += (((size_t)img * hh * sc + (y * sc + yo)) * ((size_t)ww * sc) + (x * sc + xo)) * ld + 4 * q;
            cp16(base + r * T::RS + p * 32 + (p >> 3) * 16 + q * 16, s, ok);
        }
        const uint32_t wb = base + T::IN_BYTES;
        for (int i = tid; i < T::TAPS * CK * (OCB / 4); i += NB) {
            const int n4 = i % (OCB / 4), kc = i / (OCB / 4);   // kc = tap * CK + c
            const float* s;
            if (MODE == 1) {
                const int col = nt + 4 * n4, ab = col / a.cout;
                s = a.b + ((size_t)ab * a.cin + ch + kc) * a.cout + (col - ab * a.cout);
            } else {
                const int tap = kc / CK, c = kc - tap * CK;
                s = a.b + ((size_t)tap * a.cin + ch + c) * a.ncols + nt + 4 * n4;
            }
            cp16(wb + i * 16, s, true);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    f2 acc[8][4];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[p][j] = 0ull;

    load(st0, 0);
    for (int st = st0; st < st1; ++st) {
        const int buf = (st - st0) & 1;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (st + 1 < st1) load(st + 1, buf ^ 1);
        const uint8_t* in = smem + buf * T::STAGE + row * T::RS + g * (8 * 32 + 16);
        const uint8_t* wt = smem + buf * T::STAGE + T::IN_BYTES + ocg * 32;
        constexpr int KY = MODE == 0 ? 3 : 1;
#pragma unroll 1
        for (int c = 0; c < CK; ++c) {
#pragma unroll
            for (int dy = 0; dy < KY; ++dy) {
                f2 xd[8 + 2 * T::HALO];
#pragma unroll
                for (int k = 0; k < 8 + 2 * T::HALO; ++k) {
                    const float v = *reinterpret_cast<const float*>(in + dy * T::RS + k * 32 + (k >> 3) * 16 + c * 4);
                    xd[k] = f2_pack(v, v);
                }
#pragma unroll
                for (int dx = 0; dx < KY; ++dx) {
                    const ulonglong2* wp = reinterpret_cast<const ulonglong2*>(wt + ((dy * 3 + dx) * CK + c) * OCB * 4);
                    const ulonglong2 w0 = wp[0], w1 = wp[1];
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        acc[p][0] = f2_fma(xd[p + dx], w0.x, acc[p][0]);
                        acc[p][1] = f2_fma(xd[p + dx], w0.y, acc[p][1]);
                        acc[p][2] = f2_fma(xd[p + dx], w1.x, acc[p][2]);
                        acc[p][3] = f2_fma(xd[p + dx], w1.y, acc[p][3]);
                    }
                }
            }
        }
    }

    // bias, activation, mask and store of pixel p's 8 channels
    const int yy = y0 + row, col = nt + 8 * ocg;
    auto emit = [&](int p, const float* v) {
        const int xx = x0 + 8 * g + p;
        if (yy >= a.h || xx >= a.w) return;
        float o[8];
        int ch = col, ab = 0;
        if (MODE == 1) {
            ab = col / a.cout;
            ch = col - ab * a.cout;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            o[j] = v[j] + (a.bias ? a.bias[ch + j] : 0.0f);
            if (a.relu) o[j] = fmaxf(o[j], 0.0f);
        }
        size_t at = ((size_t)img * a.h + yy) * a.w + xx;
        if (MODE == 1) at = ((size_t)img * 2 * a.h + 2 * yy + (ab >> 1)) * (2 * (size_t)a.w) + 2 * xx + (ab & 1);
        at = at * a.ldy + ch;
        if (a.mask) {
            const float4 m0 = *reinterpret_cast<const float4*>(a.mask + at);
            const float4 m1 = *reinterpret_cast<const float4*>(a.mask + at + 4);
            const float m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) o[j] = m[j] > 0.0f ? o[j] : 0.0f;
        }
        *reinterpret_cast<float4*>(a.y + at) = make_float4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<float4*>(a.y + at + 4) = make_float4(o[4], o[5], o[6], o[7]);
    };
    if (ks == 1) {
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) f2_unpack(acc[p][j], v[2 * j], v[2 * j + 1]);
            emit(p, v);
        }
        return;
    }
    // the cluster's sums: rank r makes the outputs of pixels r * 8 / ks ..
    __syncthreads();
    ulonglong2* red = reinterpret_cast<ulonglong2*>(smem);
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        red[(2 * p) * NB + tid] = make_ulonglong2(acc[p][0], acc[p][1]);
        red[(2 * p + 1) * NB + tid] = make_ulonglong2(acc[p][2], acc[p][3]);
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int np = 8 / ks;
    for (int p = kr * np; p < (kr + 1) * np; ++p) {
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int r = 0; r < ks; ++r) {
            const float4* q = reinterpret_cast<const float4*>(cl.map_shared_rank(smem, r));
            const float4 u0 = q[(2 * p) * NB + tid], u1 = q[(2 * p + 1) * NB + tid];
            v[0] += u0.x; v[1] += u0.y; v[2] += u0.z; v[3] += u0.w;
            v[4] += u1.x; v[5] += u1.y; v[6] += u1.z; v[7] += u1.w;
        }
        emit(p, v);
    }
    cl.sync();   // no block leaves while a peer reads its sums
}

// Allows `kern` `bytes` of dynamic shared memory on the current device, once per device.
template <typename K>
nrv_status allow_smem(K kern, int bytes, std::atomic<uint64_t>& done) {
    int dev = 0;
    NRV_CHECK_CUDA(cudaGetDevice(&dev));
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;
    if (done.load(std::memory_order_acquire) & bit) return NRV_OK;
    NRV_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    done.fetch_or(bit, std::memory_order_release);
    return NRV_OK;
}

// Blocks of 128 threads are for grids of at most two per SM of the chip's 152 (launch_block): they
// ask for the shared memory that keeps a third block out, because clusters are otherwise packed
// four blocks to an SM while SMs stay empty.  Blocks of 256 threads are not spread like that (one
// to an SM for grids of up to 152 blocks: a second wave, 39 us against 34.7).
template <int MODE, int OCB, int TW, int NB>
nrv_status launch_tile(F32Args& a, int ks, cudaStream_t s) {
    using T = F32Tile<MODE, OCB, TW, NB>;
    constexpr int SPREAD = NB == 128 ? 80 * 1024 : 0;
    a.tiles_x = (a.w + TW - 1) / TW;
    a.tiles_y = (a.h + T::TH - 1) / T::TH;
    const long long tiles = (long long)a.tiles_x * a.tiles_y * a.n;
    if (tiles > 0x7FFFFFFFll) return fail(NRV_ERR_UNSUPPORTED, "too many tiles");
    const int ob = a.ncols / OCB, nst = a.cin / CK;
    static std::atomic<uint64_t> attr{0};
    auto kern = conv_f32_kernel<MODE, OCB, TW, NB>;
    const nrv_status st = allow_smem(kern, T::SMEMK > SPREAD ? T::SMEMK : SPREAD, attr);
    if (st != NRV_OK) return st;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)tiles, ob, ks);
    cfg.blockDim = dim3(NB);
    cfg.dynamicSmemBytes = ks > 1 ? T::SMEMK : (nst > 1 ? T::SMEM1 : T::STAGE);
    if ((int)cfg.dynamicSmemBytes < SPREAD) cfg.dynamicSmemBytes = SPREAD;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = ks;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    NRV_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

// Blocks of 128 threads (half the tile) where 256-thread blocks split eight ways would not give
// every SM one. 128 channels at 2 x 32^2 pixels, 256 blocks of 128 against 128 of 256 threads:
// 21.4 us against 34.7 (64 channels in: 15.0 against 22.6).
template <int MODE, int OCB, int TW>
nrv_status launch_block(F32Args& a, cudaStream_t s) {
    constexpr int TH = F32Tile<MODE, OCB, TW, NT>::TH;
    const long long blocks = (long long)((a.w + TW - 1) / TW) * ((a.h + TH - 1) / TH) * (a.ncols / OCB);
    const int nst = a.cin / CK;
    // Split the input channels until one image has 128 blocks.  (256, two to an SM: 588 us against
    // 580 for a 512 x 512 frame, 1071 against 1027 for the 2 x 256^2 training step.  A split that
    // also counted the images took 1858 us for 16 x 256^2 against 2051 here, but then an image's
    // result depended on how many shared its call.)
    int ks = 1, most = 1;
    while (ks < 8 && blocks * ks < 128 && 2 * ks <= nst) ks *= 2;
    while (most < 8 && 2 * most <= nst) most *= 2;
    if (OCB == 32 && blocks * a.n * most <= 152) return launch_tile<MODE, OCB, TW, OCB == 32 ? 128 : NT>(a, ks, s);
    return launch_tile<MODE, OCB, TW, NT>(a, ks, s);
}

// The tile width that covers the image with the fewest pixels (64 where equal).
template <int MODE, int OCB>
nrv_status launch_width(F32Args& a, cudaStream_t s) {
    auto area = [&](int tw, int th) {
        return (long long)((a.w + tw - 1) / tw * tw) * ((a.h + th - 1) / th * th);
    };
    if (area(32, F32Tile<MODE, OCB, 32, NT>::TH) < area(64, F32Tile<MODE, OCB, 64, NT>::TH))
        return launch_block<MODE, OCB, 32>(a, s);
    return launch_block<MODE, OCB, 64>(a, s);
}

template <int MODE>
nrv_status launch_mode(F32Args& a, cudaStream_t s) {
    if (a.cin % CK || a.c1 % CK || a.ncols % 16 || (MODE == 2 && a.cdiv % CK) || (MODE == 1 && a.cout % 16))
        return fail(NRV_ERR_UNSUPPORTED, "FP32 conv: channel counts");
    return a.ncols % 32 == 0 ? launch_width<MODE, 32>(a, s) : launch_width<MODE, 16>(a, s);
}

// ------------------------------------------------------------------ weight gradients
// dW[(tap, c)][o] = sum over pixels of x[p + tap][c] g[p][o]: a block takes 16 input channels
// x 16 output channels x 9 taps over a contiguous run of 32 x 8 pixel tiles.  Thread (slice,
// dy, channel pair) walks one row of the tile with 3 dx x 2 c x 16 o sums: a window of three
// pixels slides along the row, so each step reads one new channel pair and 16 gradients for 48
// paired FMAs; the row is unrolled, so the window is register names and not moves.  The eight
// slices are added in order, through shared memory laid out [sum][thread]: with a thread's sums
// side by side the writes met in one bank (70% of all shared wavefronts).  16 x 16 channels over
// 2 x 256^2 pixels: 36 us before, 22 now (0.60 GFLOP: 8 us of the FP32 pipe).
constexpr int WT = 192;              // 8 slices x 3 kernel rows x 8 channel pairs
constexpr int WTW = 32, WTH = 8;     // tile
constexpr int WXRS = (WTW + 2) * 64 + 64;   // 64 bytes off per row in the banks
constexpr int WX_BYTES = (WTH + 2) * WXRS, WG_BYTES = WTH * WTW * 64;
constexpr int WSTAGE = WX_BYTES + WG_BYTES;
constexpr int WRLD = WT + 1;         // the odd pair count sets the two channels of a pair 16 banks apart
constexpr int WRED = 48 * WRLD * 8;
constexpr int WSMEM = 2 * WSTAGE > WRED ? 2 * WSTAGE : WRED;

struct F32Wgrad {
    const float* g;
    const float *x1, *x2;
    int c1, c2, cout;
    int n, h, w, tiles_x, tiles_y, ntiles, tiles_per_block;
    float *part, *partb;
};

__global__ void __launch_bounds__(WT, 2) wgrad_f32_kernel(const __grid_constant__ F32Wgrad a) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ float bred[12][16];
    const uint32_t s0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    const int t = threadIdx.x, slice = t / 24, u = t % 24, dy = u / 8, cp = u % 8;
    const int og = blockIdx.y * 16, cg = blockIdx.z * 16, cin = a.c1 + a.c2;
    const float* src = cg < a.c1 ? a.x1 + cg : a.x2 + (cg - a.c1);
    const int ld = cg < a.c1 ? a.c1 : a.c2;
    const int nc = cin - cg < 16 ? cin - cg : 16;      // real channels of the group
    const int t0 = blockIdx.x * a.tiles_per_block;
    const int t1 = t0 + a.tiles_per_block < a.ntiles ? t0 + a.tiles_per_block : a.ntiles;

    auto load = [&](int tile, int buf) {
        const int tx = tile % a.tiles_x, ty = (tile / a.tiles_x) % a.tiles_y, img = tile / (a.tiles_x * a.tiles_y);
        const int x0 = tx * WTW, y0 = ty * WTH;
        const uint32_t xb = s0 + buf * WSTAGE, gb = xb + WX_BYTES;
        for (int i = t; i < (WTH + 2) * (WTW + 2) * 4; i += WT) {
            const int q = i & 3, pp = i >> 2, r = pp / (WTW + 2), p = pp - r * (WTW + 2);
            const int y = y0 + r - 1, x = x0 + p - 1;
            const bool ok = (unsigned)y < (unsigned)a.h && (unsigned)x < (unsigned)a.w && 4 * q < nc;
            const float* sp = src;
            if (ok) sp += (((size_t)img * a.h + y) * a.w + x) * ld + 4 * q;
            cp16(xb + r * WXRS + p * 64 + q * 16, sp, ok);
        }
        for (int i = t; i < WTH * WTW * 4; i += WT) {
            const int q = i & 3, pp = i >> 2, r = pp / WTW, p = pp - r * WTW;
            const int y = y0 + r, x = x0 + p;
            const bool ok = y < a.h && x < a.w;
            const float* sp = a.g;
            if (ok) sp += (((size_t)img * a.h + y) * a.w + x) * a.cout + og + 4 * q;
            cp16(gb + pp * 64 + q * 16, sp, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    f2 acc[3][2][8];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[i][j][k] = 0ull;
    float bsum = 0.0f;
    if (t0 < t1) load(t0, 0);
    for (int tile = t0; tile < t1; ++tile) {
        const int buf = (tile - t0) & 1;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (tile + 1 < t1) load(tile + 1, buf ^ 1);
        const uint8_t* xs = smem + buf * WSTAGE + (slice + dy) * WXRS + cp * 8;
        const uint8_t* gs = smem + buf * WSTAGE + WX_BYTES;
        const uint8_t* gr = gs + slice * WTW * 64;
        f2 win[3][2];
        auto take = [&](int p, f2* d) {
            const float2 v = *reinterpret_cast<const float2*>(xs + p * 64);
            d[0] = f2_pack(v.x, v.x);
            d[1] = f2_pack(v.y, v.y);
        };
        take(0, win[0]);
        take(1, win[1]);
#pragma unroll
        for (int p = 0; p < WTW; ++p) {
            take(p + 2, win[(p + 2) % 3]);
            const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(gr + p * 64);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const ulonglong2 gv = gp[k];
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const f2 xv = win[(p + dx) % 3][c];
                        acc[dx][c][2 * k] = f2_fma(xv, gv.x, acc[dx][c][2 * k]);
                        acc[dx][c][2 * k + 1] = f2_fma(xv, gv.y, acc[dx][c][2 * k + 1]);
                    }
            }        }
        if (blockIdx.z == 0)
            for (int p = t >> 4; p < WTH * WTW; p += WT / 16)
                bsum += *reinterpret_cast<const float*>(gs + p * 64 + (t & 15) * 4);
    }
    __syncthreads();
    f2* red = reinterpret_cast<f2*>(smem);   // [sum][thread]: neighbouring threads in neighbouring banks
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int k = 0; k < 8; ++k)
                red[((dx * 2 + c) * 8 + k) * WRLD + t] = acc[dx][c][k];
    bred[t >> 4][t & 15] = bsum;
    __syncthreads();
    for (int i = t; i < 16 * 144; i += WT) {
        const int c = i & 15, tap = (i >> 4) % 9, o = i / 144;
        if (c >= nc) continue;
        const float* at = reinterpret_cast<const float*>(
            red + (((tap % 3) * 2 + (c & 1)) * 8 + o / 2) * WRLD + (tap / 3) * 8 + c / 2) + (o & 1);
        float v = at[0];
#pragma unroll
        for (int sl = 1; sl < 8; ++sl) v += at[sl * 48];
        a.part[((size_t)blockIdx.x * a.cout + og + o) * 9 * cin + tap * cin + cg + c] = v;
    }
    if (blockIdx.z == 0 && t < 16) {
        float v = bred[0][t];
        for (int k = 1; k < 12; ++k) v += bred[k][t];
        a.partb[(size_t)blockIdx.x * a.cout + og + t] = v;
    }
}

// Transposed conv: dW[c][(ab, o)] = sum over input pixels of x[p][c] g[out(p, ab)][o]: a block
// takes 32 c x 64 (ab, o) over a contiguous run of pixels, 64 per stage; a thread 8 x 8 sums,
// the eight warps every eighth pixel each, added in order at the end.
constexpr int UPX = 64;
constexpr int USTAGE = UPX * (32 + 64) * 4;
constexpr int URLD = NT + 1;
constexpr int URED = 64 * URLD * 4;
constexpr int USMEM = 2 * USTAGE > URED ? 2 * USTAGE : URED;

struct F32WgradUp {
    const float *x, *g;
    int cin, cout, ldg;
    int n, h, w;             // input level
    long long npx, px_per_block;
    float *part, *partb;
};

__global__ void __launch_bounds__(NT, 2) wgrad_up_f32_kernel(const __grid_constant__ F32WgradUp a) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ float bred[4][64];
    const uint32_t s0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, cq = lane & 3, nq = lane >> 2;
    const int cg = blockIdx.y * 32, ng = blockIdx.z * 64, K = 4 * a.cout;
    const long long q0 = blockIdx.x * a.px_per_block;
    const long long q1 = q0 + a.px_per_block < a.npx ? q0 + a.px_per_block : a.npx;

    auto load = [&](long long qb, int buf) {
        const uint32_t xb = s0 + buf * USTAGE, gb = xb + UPX * 128;
        for (int i = t; i < UPX * 8; i += NT) {
            const int q = i & 7, p = i >> 3;
            const bool ok = qb + p < q1;
            cp16(xb + i * 16, ok ? a.x + (size_t)(qb + p) * a.cin + cg + 4 * q : a.x, ok);
        }
        for (int i = t; i < UPX * 16; i += NT) {
            const int q = i & 15, p = i >> 4, col = ng + 4 * q, ab = col / a.cout, o = col - ab * a.cout;
            const long long px = qb + p;
            const bool ok = px < q1;
            const float* sp = a.g;
            if (ok) {
                const int X = (int)(px % a.w), r = (int)(px / a.w), Y = r % a.h, img = r / a.h;
                sp += (((size_t)img * 2 * a.h + 2 * Y + (ab >> 1)) * (2 * (size_t)a.w) + 2 * X + (ab & 1)) * a.ldg + o;
            }
            cp16(gb + i * 16, sp, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    f2 acc[4][8];   // channel pairs x columns
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
    float bsum = 0.0f;
    if (q0 < q1) load(q0, 0);
    int buf = 0;
    for (long long qb = q0; qb < q1; qb += UPX, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (qb + UPX < q1) load(qb + UPX, buf ^ 1);
        const uint8_t* xs = smem + buf * USTAGE;
        const uint8_t* gs = xs + UPX * 128;
#pragma unroll 2
        for (int p = warp; p < UPX; p += NT / 32) {
            const ulonglong2* xp = reinterpret_cast<const ulonglong2*>(xs + p * 128 + cq * 32);
            const ulonglong2 xa = xp[0], xb = xp[1];
            const f2 xv[4] = {xa.x, xa.y, xb.x, xb.y};
            const float4* gp = reinterpret_cast<const float4*>(gs + p * 256 + nq * 32);
            const float4 g0 = gp[0], g1 = gp[1];
            const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const f2 gd = f2_pack(gv[j], gv[j]);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][j] = f2_fma(xv[i], gd, acc[i][j]);
            }
        }
        if (blockIdx.y == 0)
            for (int p = t >> 6; p < UPX; p += 4) bsum += *reinterpret_cast<const float*>(gs + p * 256 + (t & 63) * 4);
    }
    __syncthreads();
    float* red = reinterpret_cast<float*>(smem);   // [channel 8][column 8][thread]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float lo, hi;
            f2_unpack(acc[i][j], lo, hi);
            red[((2 * i) * 8 + j) * URLD + t] = lo;
            red[((2 * i + 1) * 8 + j) * URLD + t] = hi;
        }
    bred[t >> 6][t & 63] = bsum;
    __syncthreads();
    for (int i = t; i < 32 * 64; i += NT) {
        const int col = i & 63, c = i >> 6;
        const int at = ((c & 7) * 8 + (col & 7)) * URLD + (col >> 3) * 4 + (c >> 3);
        float v = red[at];
#pragma unroll
        for (int wv = 1; wv < 8; ++wv) v += red[wv * 32 + at];
        a.part[((size_t)blockIdx.x * a.cin + cg + c) * K + ng + col] = v;
    }
    if (blockIdx.y == 0 && t < 64) {
        float v = bred[0][t];
        for (int k = 1; k < 4; ++k) v += bred[k][t];
        a.partb[(size_t)blockIdx.x * K + ng + t] = v;
    }
}

}  // namespace

// Blocks of one weight gradient: about two per SM over all channel groups.
static int split_blocks(long long units, int groups) {
    long long nb = (304 + groups - 1) / groups;
    if (nb > units) nb = units;
    if (nb < 1) nb = 1;
    const long long per = (units + nb - 1) / nb;
    return (int)((units + per - 1) / per);
}
int f32_wgrad_splits(int cin, int cout, int n, int h, int wd) {
    const long long tiles = (long long)((wd + WTW - 1) / WTW) * ((h + WTH - 1) / WTH) * n;
    return split_blocks(tiles, (cout / 16) * ((cin + 15) / 16));
}
int f32_wgrad_up_splits(int cin, int cout, int n, int h, int wd) {
    return split_blocks(((long long)n * h * wd + UPX - 1) / UPX, (cin / 32) * (cout / 16));
}

nrv_status f32_wgrad(const float* g, int cout, const float* x1, int c1, const float* x2, int c2, int n, int h,
                     int wd, float* part, float* partb, cudaStream_t s) {
    const int cin = c1 + c2;
    if (cout % 16 || (cin % 16 && cin != 8) || (c2 && c1 % 16))
        return fail(NRV_ERR_UNSUPPORTED, "weight gradient: channel groups");
    F32Wgrad a;
    memset(&a, 0, sizeof(a));
    a.g = g;
    a.x1 = x1;
    a.x2 = x2;
    a.c1 = c1;
    a.c2 = c2;
    a.cout = cout;
    a.n = n;
    a.h = h;
    a.w = wd;
    a.tiles_x = (wd + WTW - 1) / WTW;
    a.tiles_y = (h + WTH - 1) / WTH;
    if ((long long)a.tiles_x * a.tiles_y * n > 0x3FFFFFFF) return fail(NRV_ERR_UNSUPPORTED, "too many tiles");
    a.ntiles = a.tiles_x * a.tiles_y * n;
    const int nb = f32_wgrad_splits(cin, cout, n, h, wd);
    a.tiles_per_block = (a.ntiles + nb - 1) / nb;
    a.part = part;
    a.partb = partb;
    static std::atomic<uint64_t> attr{0};
    const nrv_status st = allow_smem(wgrad_f32_kernel, WSMEM, attr);
    if (st != NRV_OK) return st;
    wgrad_f32_kernel<<<dim3(nb, cout / 16, (cin + 15) / 16), WT, WSMEM, s>>>(a);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

nrv_status f32_wgrad_up(const float* x, int cin, const float* g, int ldg, int cout, int n, int h, int wd,
                        float* part, float* partb, cudaStream_t s) {
    if (cin % 32 || cout % 16) return fail(NRV_ERR_UNSUPPORTED, "weight gradient: channel groups");
    F32WgradUp a;
    memset(&a, 0, sizeof(a));
    a.x = x;
    a.g = g;
    a.cin = cin;
    a.cout = cout;
    a.ldg = ldg;
    a.n = n;
    a.h = h;
    a.w = wd;
    a.npx = (long long)n * h * wd;
    const int nb = f32_wgrad_up_splits(cin, cout, n, h, wd);
    const long long units = (a.npx + UPX - 1) / UPX;
    a.px_per_block = (units + nb - 1) / nb * UPX;
    a.part = part;
    a.partb = partb;
    static std::atomic<uint64_t> attr{0};
    const nrv_status st = allow_smem(wgrad_up_f32_kernel, USMEM, attr);
    if (st != NRV_OK) return st;
    wgrad_up_f32_kernel<<<dim3(nb, cin / 32, cout / 16), NT, USMEM, s>>>(a);
    NRV_CHECK_LAUNCH();
    return NRV_OK;
}

nrv_status f32_conv3(const float* x1, int c1, const float* x2, int c2, const float* w, const float* bias,
                     int relu, const float* mask, float* y, int cout, int n, int h, int wd, cudaStream_t s) {
    F32Args a;
    memset(&a, 0, sizeof(a));
    a.x1 = x1;
    a.x2 = x2;
    a.ld1 = a.c1 = c1;
    a.ld2 = c2;
    a.cin = c1 + c2;
    a.b = w;
    a.ncols = a.cout = cout;
    a.bias = bias;
    a.relu = relu;
    a.mask = mask;
    a.y = y;
    a.ldy = cout;
    a.n = n;
    a.h = h;
    a.w = wd;
    return launch_mode<0>(a, s);
}

nrv_status f32_upconv(const float* x, int cin, const float* w, const float* bias, float* y, int cout, int n,
                      int h, int wd, cudaStream_t s) {
    F32Args a;
    memset(&a, 0, sizeof(a));
    a.x1 = x;
    a.ld1 = a.c1 = a.cin = cin;
    a.b = w;
    a.ncols = 4 * cout;
    a.cout = cout;
    a.bias = bias;
    a.y = y;
    a.ldy = cout;
    a.n = n;
    a.h = h;
    a.w = wd;
    return launch_mode<1>(a, s);
}

nrv_status f32_upconv_dgrad(const float* g, int ldg, int cout, const float* wt, const float* mask, float* gx,
                            int cin, int n, int h, int wd, cudaStream_t s) {
    F32Args a;
    memset(&a, 0, sizeof(a));
    a.x1 = g;
    a.ld1 = ldg;
    a.cin = a.c1 = 4 * cout;
    a.cdiv = cout;
    a.b = wt;
    a.ncols = a.cout = cin;
    a.mask = mask;
    a.y = gx;
    a.ldy = cin;
    a.n = n;
    a.h = h;
    a.w = wd;
    return launch_mode<2>(a, s);
}

}  // namespace nrv
