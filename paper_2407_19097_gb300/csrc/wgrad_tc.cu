// Weight gradient of a 3x3 convolution on the tensor cores (the backward pass of
// Sec. 3.3's network, trained with Adam as in Sec. 4.1):
//
//   dW[o][c][tap] = sum over pixels p of  g[p][o] * x[p + shift(tap)][c]
//
// as a GEMM with M = output channel o (padded to the 128 lanes of TMEM), K = pixels and
// N = (tap, c) for a group of 16 input channels: N = 9 x 16 = 144, so one MMA of K = 16
// pixels serves all nine taps.  Both operands come straight from the row-planar BF16
// layout ([row][plane][pixel][8 channels]), which is the MN-major no-swizzle operand
// layout: a core matrix is 8 consecutive pixels (K) x 16 bytes (8 channels of M or N),
// K-adjacent core matrices 128 bytes apart (LBO), MN-adjacent ones one plane apart
// (SBO).  A tile is 128 pixels x0..x0+127 of one row (64 or 32 where the image is narrow: at
// level 3 of 256-pixel crops three quarters of a 128-pixel tile were padding, loaded and
// multiplied): its A block is the output gradient
// (all C_out planes), its B block nine shifted copies of the group's two input planes --
// rows y-1, y, y+1 at pixel offsets -1, 0, +1 -- loaded by TMA, so the nine taps are
// nine consecutive N blocks and zero padding is TMA's out-of-bounds fill.
//
// The 2x2 stride-2 transposed conv's weight gradient,
//
//   dW[c][o][a][b] = sum over input pixels (i, j) of  x[i][j][c] * g[2i + a][2j + b][o],
//
// runs through the same kernel with the roles turned: M = (a, b, o) -- four kernel
// positions of C_out channels, split over CTAs by a where 4 C_out > 128 -- K = input
// pixels j of one row and N = C_in.  A 5-D TMA view of the output gradient (8-byte half,
// pixel parity b, j, plane, row) loads the pixels of one parity as a dense tile, so each
// (a, b) block is again an MN-major operand; the input row is the B block.
//
// The bias gradient comes out of the same MMAs: two constant planes of BF16 ones follow
// each B block, so 16 more accumulator columns hold sum_p g[p][row].
//
// Each CTA takes a channel group and a contiguous range of tiles (a split of K), sums
// its MMAs in one TMEM accumulator and writes its partial dW; partials are added in a
// fixed order afterwards (deterministic).  Warp 0 issues TMA into two to eight stages, warp 1
// owns TMEM and issues the MMAs, warps 2-5 read the accumulator at the end.  Waits are
// bounded: on timeout the kernel sets STATUS_TIMEOUT, drains its copies, frees TMEM and
// returns.
#include <algorithm>

#include "net.h"
#include "tcgen05.cuh"

namespace nrv {

namespace {

constexpr int WG_NT = 192;           // producer, MMA issuer, 4 epilogue warps
constexpr int WG_STAGES = 8;         // at most
constexpr int WG_N = 144;            // 9 taps x 16 channels
constexpr int WG_COLS = 256;         // TMEM columns allocated (>= WG_N)

struct WgParams {
    int mode;              // 0: 3x3 conv; 1: 2x2 stride-2 transposed conv
    int n, h, w;           // input level geometry
    int tpx;               // pixels of a tile: 128, 64 or 32
    uint32_t plane;        // bytes of one plane of a tile (tpx x 16)
    int nst;               // stages
    int tiles_x, ntiles;   // t = (img * h + y) * tiles_x + xt
    int nsplit;            // CTAs per channel group (blockIdx.x)
    int cout, cin;         // channels of the output gradient and of the whole input
    int groups1;           // channel groups that read source 1 (the rest read source 2)
    int n_ab;              // mode 1: kernel positions (a, b) per CTA (4, or 2 when split by a)
    int g_plane0;          // mode 1: first plane of the output gradient's channels
    int m_real;            // mode 1: A rows that hold data (n_ab * C_out)
    int ncols;             // weight columns of the accumulator (144, or C_in); the bias
                           // column follows
    int b_planes;          // mode 0: planes per tap loaded (2, or 1 for an 8-channel input)
    uint32_t b_bytes;      // bytes TMA brings into the B block per stage
    uint32_t b_bytes_span; // B block size in shared memory (the ones planes follow it)
    uint32_t a_bytes;      // output-gradient block of a stage (C_out / 8 planes)
    uint32_t stage_bytes;  // a_bytes + the nine input blocks
    uint32_t idesc;
    float* part;           // [split][o][tap][c] (mode 0) or [split][c][ab * C_out + o]
    float* partb;          // bias: [split][o] (mode 0) or [split][ab * C_out + o]
    unsigned* status;
};

__device__ __forceinline__ uint64_t wg_desc(uint32_t saddr, uint32_t plane) {
    // start address, LBO = 128 bytes (K), SBO = one plane (M / N), version 1, no swizzle
    const uint64_t lo = ((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16);
    const uint64_t hi = (uint64_t)((plane >> 4) | (1u << 14));
    return lo | (hi << 32);
}

__global__ void __launch_bounds__(WG_NT, 1)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap tg, const __grid_constant__ CUtensorMap t1,
                    const __grid_constant__ CUtensorMap t2, const __grid_constant__ WgParams P) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bars[2 * WG_STAGES + 1];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = warp_number(), lane = threadIdx.x % 32;
    const uint32_t s0 = smem_u32(smem);
    auto b_full = [&](int i) { return smem_u32(&bars[i]); };
    auto b_empty = [&](int i) { return smem_u32(&bars[WG_STAGES + i]); };
    const uint32_t b_done = smem_u32(&bars[2 * WG_STAGES]);

    const int split = blockIdx.x, grp = blockIdx.y;
    const int t_begin = (int)(((long long)split * P.ntiles) / P.nsplit);
    const int t_end = (int)(((long long)(split + 1) * P.ntiles) / P.nsplit);
    const CUtensorMap* tx = grp < P.groups1 ? &t1 : &t2;
    const int plane0 = P.b_planes * (grp < P.groups1 ? grp : grp - P.groups1);   // in its source
    const int ab0 = grp * P.n_ab;   // mode 1: first kernel position of this CTA

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < P.nst; ++i) {
            mbar_init(b_full(i), 1);
            mbar_init(b_empty(i), 1);
        }
        mbar_init(b_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    {
        // constant parts of both stages: the ones planes (BF16 1.0), and for a one-plane
        // input the unused second plane of every tap (zero)
        const uint4 one = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
        for (int st = 0; st < P.nst; ++st) {
            uint8_t* b = smem + (size_t)st * P.stage_bytes + P.a_bytes;
            uint4* ones = reinterpret_cast<uint4*>(b + P.b_bytes_span);
            for (int i = threadIdx.x; i < 2 * P.tpx; i += WG_NT) ones[i] = one;
            if (P.mode == 0 && P.b_planes == 1)
                for (int i = threadIdx.x; i < 9 * P.tpx; i += WG_NT) {
                    const int tap = i / P.tpx, r = i % P.tpx;
                    reinterpret_cast<uint4*>(b + (size_t)(2 * tap + 1) * P.plane)[r] =
                        make_uint4(0u, 0u, 0u, 0u);
                }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"(WG_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = uniform(tmem_slot);

    if (warp == 0) {
        {
            int nloads = 0, st = 0;
            uint32_t ph = 1;
            for (int t = t_begin; t < t_end; ++t) {
                if (!warp_wait(b_empty(st), ph, &abort_flag, P.status)) break;
                const int xt = t % P.tiles_x;
                const int row = t / P.tiles_x;
                const int y = row % P.h, img = row / P.h;
                const int x0 = xt * P.tpx;
                const uint32_t sa = s0 + (uint32_t)st * P.stage_bytes;
                const uint32_t sb = sa + P.a_bytes;
                if (elect_one()) {
                    mbar_expect_tx(b_full(st), P.a_bytes + P.b_bytes);
                    if (P.mode == 0) {
                        tma_load_4d(sa, &tg, 2 * x0, 0, y, img, b_full(st));
                        for (int dy = 0; dy < 3; ++dy)
                            for (int dx = 0; dx < 3; ++dx)
                                tma_load_4d(sb + (uint32_t)(3 * dy + dx) * 2 * P.plane, tx,
                                            2 * (x0 - 1 + dx), plane0, y + dy - 1, img, b_full(st));
                    } else {
                        // kernel position (a, b): output row 2y + a, output pixels 2j + b
                        const uint32_t ab_bytes = P.a_bytes / (uint32_t)P.n_ab;
                        for (int k = 0; k < P.n_ab; ++k) {
                            const int ab = ab0 + k;
                            tma_load_5d(sa + (uint32_t)k * ab_bytes, &tg, 0, ab & 1, x0, P.g_plane0,
                                        (img * P.h + y) * 2 + (ab >> 1), b_full(st));
                        }
                        tma_load_4d(sb, &t1, 2 * x0, 0, y, img, b_full(st));
                    }
                }
                ++nloads;
                if (++st == P.nst) {
                    st = 0;
                    ph ^= 1u;
                }
            }
            // the last loads issued must land before the CTA may exit
            for (int i = nloads - P.nst < 0 ? 0 : nloads - P.nst; i < nloads; ++i)
                warp_wait(b_full(i % P.nst), (i / P.nst) & 1, &abort_flag, P.status, false);
        }
    } else if (warp == 1) {
        if (t_end > t_begin) {
            int st = 0;
            uint32_t ph = 0;
            for (int t = t_begin; t < t_end; ++t) {
                if (!warp_wait(b_full(st), ph, &abort_flag, P.status)) break;
                tc_fence_after();
                const uint32_t sa = s0 + (uint32_t)st * P.stage_bytes;
                const uint32_t sb = sa + P.a_bytes;
                if (elect_one()) {
                    // 16 pixels per K-step
                    const uint64_t da = wg_desc(sa, P.plane), db = wg_desc(sb, P.plane);
                    if (P.tpx == 128) {
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            mma_bf16(tmem, da + 16u * ks, db + 16u * ks, P.idesc,
                                     (t > t_begin || ks > 0) ? 1u : 0u);
                    } else {
                        for (int ks = 0; ks < P.tpx / 16; ++ks)
                            mma_bf16(tmem, da + 16u * ks, db + 16u * ks, P.idesc,
                                     (t > t_begin || ks > 0) ? 1u : 0u);
                    }
                    mma_commit(b_empty(st));
                }
                if (++st == P.nst) {
                    st = 0;
                    ph ^= 1u;
                }
            }
            if (elect_one()) mma_commit(b_done);
            warp_wait(b_done, 0, &abort_flag, P.status, false);
        }
    } else {
        // epilogue: TMEM lane o (warp quadrant q = warp % 4) holds dW[o][tap][16 channels]
        const int q = warp & 3;
        const int o = 32 * q + lane;
        bool ok = true;
        if (t_end > t_begin) {
            int r = 1;
            if (lane == 0) r = mbar_wait(b_done, 0, &abort_flag, P.status) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, r, 0) != 0;
            tc_fence_after();
        }
        if (ok && P.mode == 1 && 32 * q < P.m_real) {
            // row m = (ab - ab0) * C_out + o; column c -> part[split][c][ab * C_out + o]
            const int k4 = 4 * P.cout;
            float* dst = P.part + (size_t)split * P.cin * k4 + ab0 * P.cout + o;
            for (int c0 = 0; c0 < P.ncols; c0 += 16) {
                uint32_t v[16];
                if (t_end > t_begin) {
                    tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, v);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0u;
                }
                if (o < P.m_real) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) dst[(size_t)(c0 + j) * k4] = __uint_as_float(v[j]);
                }
            }
            // bias column: sum of the output gradient at this row's kernel position
            uint32_t v[16];
            if (t_end > t_begin) {
                tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)P.ncols, v);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = 0u;
            }
            if (o < P.m_real) P.partb[(size_t)split * k4 + ab0 * P.cout + o] = __uint_as_float(v[0]);
        }
        if (ok && P.mode == 0 && 32 * q < P.cout) {
            float* dst = P.part + ((size_t)split * P.cout + o) * 9 * P.cin + 8 * P.b_planes * grp;
            for (int tap = 0; tap < 9; ++tap) {
                uint32_t v[16];
                if (t_end > t_begin) {
                    tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(16 * tap), v);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0u;   // an empty split adds nothing
                }
                if (o < P.cout) {
                    // 16 channels of the group (8 with a one-plane input)
                    float4* d = reinterpret_cast<float4*>(dst + (size_t)tap * P.cin);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (j < 2 * P.b_planes) d[j] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                           __uint_as_float(v[4 * j + 2]),
                                           __uint_as_float(v[4 * j + 3]));
                }
            }
            if (grp == 0) {
                // bias column (every channel group computes it; the first one writes it)
                uint32_t v[16];
                if (t_end > t_begin) {
                    tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)P.ncols, v);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0u;
                }
                if (o < P.cout) P.partb[(size_t)split * P.cout + o] = __uint_as_float(v[0]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(WG_COLS)
                     : "memory");
    }
}

}  // namespace

// Planes of a stage whose A and B blocks hold `planes`: the ones planes after them, and at least the
// 16 planes (M = 128) that the A descriptor spans from its block.
static uint32_t stage_planes(uint32_t planes) { return planes + 2 < 16 ? 16 : planes + 2; }
// CTAs per SM (TMEM: 256 columns each): two where two stages of 128 pixels fit twice; the stages
// of narrower tiles then share that space.
static int wg_per_sm(uint32_t planes) { return 2 * stage_planes(planes) * 2048 <= 110 * 1024 ? 2 : 1; }
// Splits of K over the CTAs of one channel group, at most one per tile.
static nrv_status wg_splits(int per_sm, int groups, int ntiles, long long* ns) {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        NRV_CHECK_CUDA(cudaGetDevice(&dev));
        NRV_CHECK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (sms <= 0) sms = 148;
    }
    *ns = (long long)sms * per_sm / groups;
    if (*ns < 1) *ns = 1;
    if (*ns > ntiles) *ns = ntiles;
    return NRV_OK;
}

// Launch: grid (splits, groups), stages of (A block, B block), partials in `part`.
static nrv_status wg_launch(WgParams& P, int groups, const CUtensorMap& mg, const CUtensorMap& m1,
                            const CUtensorMap& m2, size_t per_split, float* part,
                            size_t part_floats, float* partb, int* nsplit, cudaStream_t s) {
    P.status = status_word();
    if (!P.status) return fail(NRV_ERR_CUDA, "status word unavailable");
    const uint32_t planes = (P.a_bytes + P.b_bytes_span) / P.plane;
    P.stage_bytes = stage_planes(planes) * P.plane;
    const int per_sm = wg_per_sm(planes);
    const uint32_t room = per_sm == 2 ? 110 * 1024 : 215 * 1024;
    P.nst = (int)(room / P.stage_bytes);
    if (P.nst > WG_STAGES) P.nst = WG_STAGES;
    if (P.nst < 2) return fail(NRV_ERR_UNSUPPORTED, "stages do not fit");
    if (P.tpx == 128) P.nst = 2;
    const uint32_t smem = P.nst * P.stage_bytes;
    static bool attr = false;
    if (!attr) {
        NRV_CHECK_CUDA(cudaFuncSetAttribute(wgrad_tc_kernel,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, 215 * 1024));
        attr = true;
    }
    long long ns = 0;
    NRV_TRY(wg_splits(per_sm, groups, P.ntiles, &ns));
    if ((size_t)ns * per_split > part_floats) ns = (long long)(part_floats / per_split);
    if (ns < 1) return fail(NRV_ERR_ARG, "partial buffer too small");
    P.nsplit = (int)ns;
    P.part = part;
    P.partb = partb;
    wgrad_tc_kernel<<<dim3((unsigned)ns, (unsigned)groups), WG_NT, smem, s>>>(mg, m1, m2, P);
    NRV_CHECK_LAUNCH();
    *nsplit = (int)ns;
    return NRV_OK;
}

static nrv_status wg_geometry(WgParams& P, int n, int H, int W) {
    if (n <= 0 || H <= 0 || W <= 0) return fail(NRV_ERR_ARG, "empty tensor");
    P.n = n;
    P.h = H;
    P.w = W;
    // The widest tile within a tenth of the fewest padded pixels: rows of 64 and 32 pixels in tiles
    // of 128 load and multiply 50 and 75% padding (16 x 64 x 64 pixels, 128 -> 64 channels: 46 us in
    // tiles of 128, 28 in tiles of 64; 16 x 32 x 32, 128 -> 128: 30 and 19.5), while a wide row in
    // narrow tiles pays the hand-off of a tile more often.
    auto padded = [&](long long t) { return (W + t - 1) / t * t; };
    const long long least = std::min(padded(128), std::min(padded(64), padded(32)));
    P.tpx = 10 * padded(128) <= 11 * least ? 128 : 10 * padded(64) <= 11 * least ? 64 : 32;
    P.plane = (uint32_t)P.tpx * 16;
    P.tiles_x = (W + P.tpx - 1) / P.tpx;
    const long long ntiles = (long long)P.tiles_x * H * n;
    if (ntiles > 0x3FFFFFFFll) return fail(NRV_ERR_UNSUPPORTED, "too many tiles");
    P.ntiles = (int)ntiles;
    return NRV_OK;
}

// Channel groups of a transposed conv: all four kernel positions in one CTA while 4 C_out rows fit
// in M = 128, else two groups (by a).
static int up_groups(int cout) { return 4 * cout <= 128 ? 1 : 2; }

// instruction descriptor: FP32 accumulator, A and B BF16 MN-major, M = 128
static uint32_t wg_idesc(int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

nrv_status tc_wgrad_splits(const Net* net, int l, int n, int H, int W, int* splits) {
    const Layer& L = net->layers[l];
    WgParams P;
    memset(&P, 0, sizeof(P));
    *splits = 0;
    const nrv_status st = wg_geometry(P, n, H, W);
    if (st == NRV_ERR_UNSUPPORTED) {
        clear_error();
        return NRV_OK;
    }
    NRV_TRY(st);
    long long ns = 0;
    if (L.kind == CONV3) {
        const int cin = l == L_E0A ? net->c0p : L.cin;
        NRV_TRY(wg_splits(wg_per_sm(L.cout / 8 + 18), cin == 8 ? 1 : cin / 16, P.ntiles, &ns));
    } else {
        const int groups = up_groups(L.cout);
        NRV_TRY(wg_splits(wg_per_sm(4 / groups * (L.cout / 8) + L.cin / 8), groups, P.ntiles, &ns));
    }
    *splits = (int)ns;
    return NRV_OK;
}

nrv_status tc_wgrad(const Net* net, int l, const void* g, const void* x1, int c1, const void* x2,
                    int c2, int n, int H, int W, float* part, size_t part_floats, float* partb,
                    int* nsplit, cudaStream_t s) {
    const Layer& L = net->layers[l];
    const int cin = c1 + c2;
    // channel groups of 16 (two planes per tap), or one group of 8 (the packed input)
    const int bp = (c1 % 16 == 0 && c2 % 16 == 0) ? 2 : (c1 == 8 && c2 == 0 ? 1 : 0);
    if (L.kind != CONV3 || !bp || L.cout % 8 || L.cout > 128 || (bp == 2 && cin != L.cin))
        return fail(NRV_ERR_UNSUPPORTED, "tensor-core weight gradient: channel counts");
    WgParams P;
    memset(&P, 0, sizeof(P));
    P.mode = 0;
    NRV_TRY(wg_geometry(P, n, H, W));
    P.cout = L.cout;
    P.cin = cin;
    P.groups1 = c1 / (8 * bp);
    P.n_ab = 1;
    P.m_real = L.cout;
    P.ncols = WG_N;
    P.b_planes = bp;
    P.a_bytes = (uint32_t)(L.cout / 8) * P.plane;
    P.b_bytes = 9u * bp * P.plane;
    P.b_bytes_span = 9u * 2 * P.plane;
    P.idesc = wg_idesc(WG_N + 16);
    CUtensorMap mg, m1, m2;
    NRV_TRY(tc_planar_map(&mg, g, n, H, W, L.cout / 8, L.cout / 8, P.tpx));
    NRV_TRY(tc_planar_map(&m1, x1, n, H, W, c1 / 8, bp, P.tpx));
    if (c2) NRV_TRY(tc_planar_map(&m2, x2, n, H, W, c2 / 8, bp, P.tpx));
    else m2 = m1;
    return wg_launch(P, cin / (8 * bp), mg, m1, m2, (size_t)L.cout * 9 * cin, part, part_floats,
                     partb, nsplit, s);
}

nrv_status tc_wgrad_up(const Net* net, int l, const void* g, int g_ld, int g_off, const void* x,
                       int n, int H, int W, float* part, size_t part_floats, float* partb,
                       int* nsplit, cudaStream_t s) {
    const Layer& L = net->layers[l];
    if (L.kind != UPCONV2 || L.cin % 16 || L.cin > 128 || L.cout % 8 || L.cout > 64 || g_ld % 8 ||
        g_off % 8 || g_off + L.cout > g_ld)
        return fail(NRV_ERR_UNSUPPORTED, "tensor-core weight gradient: channel counts");
    WgParams P;
    memset(&P, 0, sizeof(P));
    P.mode = 1;
    NRV_TRY(wg_geometry(P, n, H, W));
    P.cout = L.cout;
    P.cin = L.cin;
    P.groups1 = 0;
    const int groups = up_groups(L.cout);
    P.n_ab = 4 / groups;
    P.m_real = P.n_ab * L.cout;
    P.ncols = L.cin;
    P.b_planes = 2;
    P.a_bytes = (uint32_t)P.n_ab * (L.cout / 8) * P.plane;
    P.b_bytes = (uint32_t)(L.cin / 8) * P.plane;
    P.b_bytes_span = P.b_bytes;
    P.idesc = wg_idesc(L.cin + 16);
    CUtensorMap mg, m1;
    P.g_plane0 = g_off / 8;
    NRV_TRY(tc_parity_map(&mg, g, n * 2 * H, 2 * W, g_ld / 8, L.cout / 8, P.tpx));
    NRV_TRY(tc_planar_map(&m1, x, n, H, W, L.cin / 8, L.cin / 8, P.tpx));
    return wg_launch(P, groups, mg, m1, m1, (size_t)L.cin * 4 * L.cout, part, part_floats, partb,
                     nsplit, s);
}

}  // namespace nrv
