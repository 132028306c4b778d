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
//  * Where the tiles of a layer are fewer than the SMs can hold (the deep levels), the input
//    channels are split over a cluster of KS blocks, whose sums are added through distributed
//    shared memory in rank order (deterministic).
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

template <int MODE, int OCB, int TW>
struct F32Tile {
    static constexpr int HALO = MODE == 0 ? 1 : 0;
    static constexpr int TAPS = MODE == 0 ? 9 : 1;
    static constexpr int OG = OCB / 8;                 // channel groups
    static constexpr int GX = TW / 8;                  // pixel groups per row
    static constexpr int RQ = 8 / GX;                  // rows of a quarter-warp
    static constexpr int RW = RQ * (4 / OG);           // rows of a warp
    static constexpr int TH = RW * (NT / 32);
    static constexpr int COLS = TW + 2 * HALO, ROWS = TH + 2 * HALO;
    static constexpr int RAW = (COLS - 1) * 32 + ((COLS - 1) / 8) * 16 + 32;
    // two rows per quarter-warp: the second one 64 bytes off in the banks
    static constexpr int RS = RQ == 1 ? RAW : (RAW + 63) / 128 * 128 + 64;
    static constexpr int IN_BYTES = ROWS * RS;
    static constexpr int W_BYTES = TAPS * CK * OCB * 4;
    static constexpr int STAGE = IN_BYTES + W_BYTES;
    static constexpr int RED = NT * 64 * 4;            // a block's sums, for the cluster
    static constexpr int SMEM1 = 2 * STAGE;
    static constexpr int SMEMK = SMEM1 > RED ? SMEM1 : RED;
    static_assert(RS >= RAW && RS % 16 == 0 && (RQ == 1 || RS % 128 == 64), "row stride");
};

template <int MODE, int OCB, int TW>
__global__ void __launch_bounds__(NT, 2) conv_f32_kernel(const __grid_constant__ F32Args a) {
    using T = F32Tile<MODE, OCB, TW>;
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
        for (int i = tid; i < T::ROWS * T::COLS * 2; i += NT) {
            const int q = i & 1, pp = i >> 1, r = pp / T::COLS, p = pp - r * T::COLS;
            const int y = y0 + r - T::HALO, x = x0 + p - T::HALO;
            const bool ok = (unsigned)y < (unsigned)hh && (unsigned)x < (unsigned)ww;
            const float* s = src;
            if (ok) s += (((size_t)img * hh * sc + (y * sc + yo)) * ((size_t)ww * sc) + (x * sc + xo)) * ld + 4 * q;
            cp16(base + r * T::RS + p * 32 + (p >> 3) * 16 + q * 16, s, ok);
        }
        const uint32_t wb = base + T::IN_BYTES;
        for (int i = tid; i < T::TAPS * CK * (OCB / 4); i += NT) {
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
        red[(2 * p) * NT + tid] = make_ulonglong2(acc[p][0], acc[p][1]);
        red[(2 * p + 1) * NT + tid] = make_ulonglong2(acc[p][2], acc[p][3]);
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int np = 8 / ks;
    for (int p = kr * np; p < (kr + 1) * np; ++p) {
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int r = 0; r < ks; ++r) {
            const float4* q = reinterpret_cast<const float4*>(cl.map_shared_rank(smem, r));
            const float4 u0 = q[(2 * p) * NT + tid], u1 = q[(2 * p + 1) * NT + tid];
            v[0] += u0.x; v[1] += u0.y; v[2] += u0.z; v[3] += u0.w;
            v[4] += u1.x; v[5] += u1.y; v[6] += u1.z; v[7] += u1.w;
        }
        emit(p, v);
    }
    cl.sync();   // no block leaves while a peer reads its sums
}

template <int MODE, int OCB, int TW>
nrv_status launch_tile(F32Args& a, cudaStream_t s) {
    using T = F32Tile<MODE, OCB, TW>;
    a.tiles_x = (a.w + TW - 1) / TW;
    a.tiles_y = (a.h + T::TH - 1) / T::TH;
    const long long tiles = (long long)a.tiles_x * a.tiles_y * a.n;
    if (tiles > 0x7FFFFFFFll) return fail(NRV_ERR_UNSUPPORTED, "too many tiles");
    const int ob = a.ncols / OCB, nst = a.cin / CK;
    // split the input channels while the blocks do not fill the SMs (two blocks each)
    int ks = 1;
    while (ks < 8 && tiles * ob * ks < 256 && 2 * ks <= nst) ks *= 2;
    static bool attr = false;
    auto kern = conv_f32_kernel<MODE, OCB, TW>;
    if (!attr) {
        NRV_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, T::SMEMK));
        attr = true;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)tiles, ob, ks);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = ks > 1 ? T::SMEMK : (nst > 1 ? T::SMEM1 : T::STAGE);
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

// The tile width that covers the image with the fewest pixels (64 where equal).
template <int MODE, int OCB>
nrv_status launch_width(F32Args& a, cudaStream_t s) {
    auto area = [&](int tw, int th) {
        return (long long)((a.w + tw - 1) / tw * tw) * ((a.h + th - 1) / th * th);
    };
    if (area(32, F32Tile<MODE, OCB, 32>::TH) < area(64, F32Tile<MODE, OCB, 64>::TH))
        return launch_tile<MODE, OCB, 32>(a, s);
    return launch_tile<MODE, OCB, 64>(a, s);
}

template <int MODE>
nrv_status launch_mode(F32Args& a, cudaStream_t s) {
    if (a.cin % CK || a.c1 % CK || a.ncols % 16 || (MODE == 2 && a.cdiv % CK) || (MODE == 1 && a.cout % 16))
        return fail(NRV_ERR_UNSUPPORTED, "FP32 conv: channel counts");
    return a.ncols % 32 == 0 ? launch_width<MODE, 32>(a, s) : launch_width<MODE, 16>(a, s);
}

}  // namespace

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
