"""The four-point projection of the render pass against the scalar IEEE sequence, bit for bit.

A small kernel built from the library's own header (csrc/project.cuh) compares, on the GPU:
the negated reciprocal with __frcp_rn for every mantissa at the ends and the middle of the
depth range, the corrected quotient with __fdiv_rn on random operands whose quotient is near
the screen (and on the hardest ones, next to a pixel edge), and project4 with the scalar
projection on random views and points, among them NaN, infinities, huge and tiny values.
"""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_19097_gb300", "csrc")

SOURCE = r"""
#include "project.cuh"
using namespace nrv;
__device__ __forceinline__ uint32_t rnd(uint64_t& s) {
    s += 0x9E3779B97F4A7C15ull;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)((z ^ (z >> 31)) >> 32);
}
__device__ __forceinline__ float lo(f2 v) { float a, b; f2_unpack(v, a, b); return a; }
__global__ void rcp_k(uint32_t exponent, unsigned long long* bad) {
    const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;      // 2^23 threads
    const float w = __uint_as_float((exponent << 23) | m);
    const float n = lo(f2_neg_rcp(f2_pack(w, w)));
    if (__float_as_uint(n) != __float_as_uint(-__frcp_rn(w))) atomicAdd(bad, 1ull);
}
__global__ void div_k(uint64_t seed, int iters, unsigned long long* bad) {
    uint64_t s = seed + 0x632BE59BD9B4E019ull * (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x);
    for (int i = 0; i < iters; ++i) {
        const uint32_t e = 67 + rnd(s) % 180;                      // 2^-60 .. 2^119
        const float w = __uint_as_float((e << 23) | (rnd(s) & 0x7FFFFFu));
        float q = __uint_as_float(((127u - rnd(s) % 12u) << 23) | (rnd(s) & 0x7FFFFFu));
        if (rnd(s) & 1) {                                          // a quotient at a pixel edge
            const float W = (float)(1 + rnd(s) % 4096);
            q = __fsub_rn(__fdiv_rn((float)(rnd(s) % 4097), 0.5f * W), 1.0f);
        }
        float c = __fmul_rn(q, w);
        c = __uint_as_float(__float_as_uint(c) + (rnd(s) % 5u) - 2u);
        if (rnd(s) & 1) c = -c;
        const f2 W2 = f2_pack(w, w), C = f2_pack(c, c);
        const float a = lo(f2_neg_quot(C, W2, f2_neg_rcp(W2))), b = -__fdiv_rn(c, w);
        // infinite or NaN: NaN here (off screen either way); below 2^-40 the last bits do not matter
        const bool same = !(fabsf(b) <= 3.4028234e38f) ? a != a
                          : fabsf(b) < 0x1p-40f        ? fabsf(a) < 0x1p-39f
                                                       : __float_as_uint(a) == __float_as_uint(b);
        if (!same) atomicAdd(bad, 1ull);
    }
}
__global__ void proj_k(uint64_t seed, int iters, unsigned long long* bad) {
    uint64_t s = seed + 0x632BE59BD9B4E019ull * (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x);
    const float special[8] = {0.0f, -0.0f, INFINITY, -INFINITY, NAN, 3e38f, 1e-42f, -3e38f};
    auto val = [&](float scale) {
        const uint32_t r = rnd(s);
        if (r % 97 == 0) return special[rnd(s) & 7];
        return scale * ((float)(int)rnd(s) * 0x1p-31f);
    };
    for (int i = 0; i < iters; ++i) {
        RView v;
        const float sc = rnd(s) % 7 ? 1.0f : __uint_as_float((60 + rnd(s) % 130) << 23);
        for (int k = 0; k < 12; ++k) {
            v.m[k] = sc * ((float)(int)rnd(s) * 0x1p-31f);
            if (rnd(s) % 3 == 0) v.m[k] = 0.0f;
        }
        v.m[11] += 2.0f * sc;
        v.width = 1 + rnd(s) % (rnd(s) % 3 ? 2048 : 16384);
        v.height = 1 + rnd(s) % (rnd(s) % 3 ? 2048 : 16384);
        v.hw = 0.5f * v.width; v.hh = 0.5f * v.height; v.fw = v.width; v.fh = v.height;
        v.znear = rnd(s) % 5 ? 0.1f * sc : 1e-40f;
        v.zfar = rnd(s) % 5 ? 1e3f * sc : INFINITY;
        if (!(v.znear > 0.0f) || !(v.zfar >= v.znear)) continue;
        v.key = nullptr;
        FView f;
        fview_init(f, v);
        float x[4], y[4], z[4];
        for (int j = 0; j < 4; ++j) { x[j] = val(2.0f); y[j] = val(2.0f); z[j] = val(2.0f); }
        const f2 X[2] = {f2_pack(x[0], x[1]), f2_pack(x[2], x[3])};
        const f2 Y[2] = {f2_pack(y[0], y[1]), f2_pack(y[2], y[3])};
        const f2 Z[2] = {f2_pack(z[0], z[1]), f2_pack(z[2], z[3])};
        uint32_t pix[4], db[4];
        bool ok[4];
        project4(f, X, Y, Z, pix, db, ok);
        for (int j = 0; j < 4; ++j) {
            auto row = [&](int r) {
                const float* m = v.m + 4 * r;
                return __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(m[0], x[j]), __fmul_rn(m[1], y[j])),
                                           __fmul_rn(m[2], z[j])), m[3]);
            };
            const float cw = row(2);
            bool want = cw >= v.znear && cw <= v.zfar;
            const uint32_t b = __float_as_uint(cw);
            if (want && (b < FAST_W_LO || b > FAST_W_HI)) {       // the wide path's
                if (ok[j] || !f.wide) atomicAdd(bad, 1ull);
                continue;
            }
            const float sx = __fmul_rn(__fadd_rn(__fdiv_rn(row(0), cw), 1.0f), v.hw);
            const float sy = __fmul_rn(__fsub_rn(1.0f, __fdiv_rn(row(1), cw)), v.hh);
            want = want && sx >= 0.0f && sx < v.fw && sy >= 0.0f && sy < v.fh;
            if (want != ok[j]) { atomicAdd(bad, 1ull); continue; }
            if (want && (db[j] != b || pix[j] != (uint32_t)__float2int_rz(sy) * (uint32_t)v.width +
                                                     (uint32_t)__float2int_rz(sx)))
                atomicAdd(bad, 1ull);
            if (want) atomicAdd(bad + 1, 1ull);
        }
    }
}
static int done(unsigned long long* d, unsigned long long* out) {
    const int e = cudaDeviceSynchronize() != cudaSuccess ||
                  cudaMemcpy(out, d, 16, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(d);
    return e;
}
#define START unsigned long long* d; if (cudaMalloc(&d, 16) != cudaSuccess || cudaMemset(d, 0, 16) != cudaSuccess) return 1
extern "C" int t_rcp(unsigned e, unsigned long long* out) { START; rcp_k<<<32768, 256>>>(e, d); return done(d, out); }
extern "C" int t_div(uint64_t seed, int it, unsigned long long* out) { START; div_k<<<1216, 256>>>(seed, it, d); return done(d, out); }
extern "C" int t_proj(uint64_t seed, int it, unsigned long long* out) { START; proj_k<<<1216, 256>>>(seed, it, d); return done(d, out); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2407_19097_gb300.build_lib import ARCH, _nvcc
    d = tmp_path_factory.mktemp("project")
    src, so = d / "t.cu", d / "t.so"
    src.write_text(SOURCE)
    subprocess.check_call([_nvcc(), *ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
                           "-shared", "-I" + CSRC, str(src), "-o", str(so)])
    return ctypes.CDLL(str(so))


def _run(fn, *args):
    out = (ctypes.c_uint64 * 2)()
    assert fn(*args, out) == 0
    return out[0], out[1]


@pytest.mark.parametrize("exponent", [67, 68, 120, 126, 127, 128, 140, 200, 250, 251])
def test_reciprocal_every_mantissa(lib, exponent):
    assert _run(lib.t_rcp, ctypes.c_uint(exponent))[0] == 0


def test_quotient_is_ieee(lib):
    for seed in (1, 2):
        assert _run(lib.t_div, ctypes.c_uint64(seed), 4000)[0] == 0


def test_projection_matches_scalar(lib):
    bad, hits = _run(lib.t_proj, ctypes.c_uint64(5), 2000)
    assert bad == 0 and hits > 1_000_000
