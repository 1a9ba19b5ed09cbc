// Surrogate network kernels (include/lbm_nn.h) other than the convolutions
// (nn_conv.cu): weight flipping, bias gradient, the MSE loss, Adam, and the
// packing between solver fields and network states.
#include "lbm.h"
#include "lbm_nn.h"
#include "nn_internal.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

namespace {

// ---------------------------------------------------------------- helpers --
int launch_status() {
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

// -------------------------------------------------------- small kernels --
__global__ void flip_kernel(const __nv_bfloat16* __restrict__ w, int CI, int CO, __nv_bfloat16* __restrict__ wt) {
    const int n = 9 * CI * CO;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int o = i % CO, t = (i / CO) % 9, c = i / (9 * CO);  // wt[c][t][o]
        wt[i] = w[((size_t)o * 9 + (8 - t)) * CI + c];
    }
}

constexpr int RED_BLOCKS = 1024;

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Sums of the channels of dy over pixels, one partial per block.  HBM-bound: a
// thread takes 8 channels of a pixel in one 16-byte load and keeps 8 sums, the
// block's threads lie over consecutive bytes, and 4 loads per thread are in
// flight.  16 x 256 x 256 pixels of 48 channels (100.7 MB, dy written before it):
// 37 us with one 2-byte load per thread and iteration, 26 us so (cold L2).
// aligned: dy on a 16-byte boundary (else the same sums from 2-byte loads).
template <int CO>
__global__ void __launch_bounds__(256)
    bias_grad_partials(const __nv_bfloat16* __restrict__ dy, long long P, float* __restrict__ part, bool aligned) {
    constexpr int NC = CO / 8;                // 16-byte chunks per pixel
    constexpr int ROWS = 256 / NC;            // pixels per pass of a block
    __shared__ float s[ROWS][CO];
    const int j = threadIdx.x % NC, r = threadIdx.x / NC;
    float a[8] = {};
    if (r < ROWS) {
        const long long stride = (long long)gridDim.x * ROWS;
        auto add = [&](uint4 v) {
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                a[2 * k] += bf16_lo(w[k]);
                a[2 * k + 1] += bf16_hi(w[k]);
            }
        };
        long long p = (long long)blockIdx.x * ROWS + r;
        if (aligned) {
            const uint4* src = reinterpret_cast<const uint4*>(dy) + j;
            for (; p + 3 * stride < P; p += 4 * stride) {
                uint4 v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = __ldg(src + (p + k * stride) * NC);
#pragma unroll
                for (int k = 0; k < 4; ++k) add(v[k]);
            }
            for (; p < P; p += stride) add(__ldg(src + p * NC));
        } else {
            for (; p < P; p += stride)
#pragma unroll
                for (int k = 0; k < 8; ++k) a[k] += __bfloat162float(dy[p * CO + 8 * j + k]);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) s[r][8 * j + k] = a[k];
    }
    __syncthreads();
    if (threadIdx.x < CO) {
        float t = 0.0f;
#pragma unroll 4
        for (int k = 0; k < ROWS; ++k) t += s[k][threadIdx.x];
        part[(size_t)blockIdx.x * CO + threadIdx.x] = t;
    }
}

// out[o] = sum over nb partials of channel o, one block per channel and a tree in
// a fixed order: latency-bound (58 us when one thread per channel added them in
// turn, 3.6 us so at nb = 1024).
__global__ void __launch_bounds__(256)
    sum_partials(const float* __restrict__ part, int nb, int CO, float* __restrict__ out) {
    __shared__ float s[256];
    const int o = blockIdx.x;
    float t = 0.0f;
    for (int b = threadIdx.x; b < nb; b += 256) t += part[(size_t)b * CO + o];
    s[threadIdx.x] = t;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[o] = s[0];
}

// One pixel of the loss per thread.  The FP64 pipe (2 lanes per clock and SM on
// GB300) bounds a version that forms every square in double: 208 us at 16 x 256 x
// 256 pixels, over the 16 channels of which 5 are used.  Here the difference is
// split exactly into two floats, s + e = pred - target (Knuth's two-sum), its
// square into h + l + p + q + e^2 (a fused multiply-add gives a product's rounding
// error), and the pixel's squares are added as triples of floats H + M + L; only
// the pixel's sum is converted and added in double.  L is 2^-48 of the sum and
// carries 24 bits, so a pixel's sum is exact to better than 2^-60, where adding the
// squares in double rounded once per channel.  (As pairs, without L: 2^-46.)
// Squares that would leave the float range take the double form.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// A pixel's squares and gradient formed in double throughout (a call, so that the
// common path holds none of it: predicated off, it kept the FP64 pipe busy).
__device__ __noinline__ double pixel_in_double(const float* __restrict__ x, const float* __restrict__ y, int U,
                                               double two_inv, __nv_bfloat16* __restrict__ out) {
    double a = 0.0;
    for (int c = 0; c < 16; ++c) {
        const double d = c < U ? (double)x[c] - (double)y[c] : 0.0;
        a += d * d;
        if (out) out[c] = __float2bfloat16_rn((float)(two_inv * d));
    }
    return a;
}

// VEC: pred, target and dpred on 16-byte boundaries (else scalar accesses).
// dpred = 2 inv d: the FP32 product with 2 inv = khi + klo, accurate to 2^-46 before
// its one rounding to float, then rounded to bfloat16.
// NV: groups of 4 channels in use.  Each thread has the loads of two pixels in
// flight before it uses either.
template <bool VEC, int NV>
__global__ void __launch_bounds__(256)
    mse_partials(const float* __restrict__ pred, const float* __restrict__ target, int U, long long P,
                 __nv_bfloat16* __restrict__ dpred, double* __restrict__ part, double inv, float khi, float klo) {
    __shared__ double sh[8];
    double a = 0.0;
    auto fetch = [&](const float* __restrict__ src, long long p, float (&x)[4 * NV]) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            if constexpr (VEC) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(src + p * 16) + q);
                x[4 * q] = v.x;
                x[4 * q + 1] = v.y;
                x[4 * q + 2] = v.z;
                x[4 * q + 3] = v.w;
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) x[4 * q + c] = __ldg(src + p * 16 + 4 * q + c);
            }
        }
    };
    auto pixel = [&](long long p, const float (&x)[4 * NV], const float (&y)[4 * NV]) {
        float g[16] = {};
        float H = 0.0f, M = 0.0f, L = 0.0f;
        bool odd = false;  // a difference whose square leaves the float range
#pragma unroll
        for (int c = 0; c < 4 * NV; ++c) {
            if (c >= U) continue;
            float s, e;
            two_sum(x[c], -y[c], s, e);
            const float m = fabsf(s);
            odd |= !(m == 0.0f || (m > 1e-14f && m < 1e18f));  // also NaN
            // (s + e)^2 = h + l + p + q + e^2
            const float h = __fmul_rn(s, s), l = __fmaf_rn(s, s, -h);
            const float s2 = 2.0f * s, p = __fmul_rn(s2, e), q = __fmaf_rn(s2, e, -p);
            float r0, r1, r2, r3;
            two_sum(H, h, H, r0);
            two_sum(M, r0, M, r1);
            two_sum(M, l, M, r2);
            two_sum(M, p, M, r3);
            L = __fadd_rn(L, __fadd_rn(__fadd_rn(__fadd_rn(r1, r2), r3), __fmaf_rn(e, e, q)));
            g[c] = __fmaf_rn(khi, s, __fmaf_rn(khi, e, __fmul_rn(klo, s)));
        }
        if (odd) {
            a += pixel_in_double(pred + p * 16, target + p * 16, U, 2.0 * inv, dpred ? dpred + p * 16 : nullptr);
            return;
        }
        a += (double)H + ((double)M + (double)L);
        if (!dpred) return;
        if constexpr (VEC) {
            uint32_t out[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const __nv_bfloat162 w = __floats2bfloat162_rn(g[2 * k], g[2 * k + 1]);
                out[k] = *reinterpret_cast<const uint32_t*>(&w);
            }
            uint4* o = reinterpret_cast<uint4*>(dpred + p * 16);
            o[0] = make_uint4(out[0], out[1], out[2], out[3]);
            o[1] = make_uint4(out[4], out[5], out[6], out[7]);
        } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) dpred[p * 16 + c] = __float2bfloat16_rn(g[c]);
        }
    };
    const long long stride = (long long)gridDim.x * 256;
    for (long long p = (long long)blockIdx.x * 256 + threadIdx.x; p < P; p += 2 * stride) {
        const bool two = p + stride < P;
        float x0[4 * NV], y0[4 * NV], x1[4 * NV], y1[4 * NV];
        fetch(pred, p, x0);
        fetch(target, p, y0);
        if (two) {
            fetch(pred, p + stride, x1);
            fetch(target, p + stride, y1);
        }
        pixel(p, x0, y0);
        if (two) pixel(p + stride, x1, y1);
    }
    for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += sh[w];
        part[blockIdx.x] = t * inv;
    }
}

// The loss from the block partials, in a fixed order (67 us when one thread added
// the 1024 of them in turn, 3.7 us so).
__global__ void __launch_bounds__(256) mse_final(const double* __restrict__ part, int nb, double* __restrict__ loss) {
    __shared__ double s[256];
    double t = 0.0;
    for (int b = threadIdx.x; b < nb; b += 256) t += part[b];
    s[threadIdx.x] = t;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = s[0];
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                            const uint8_t* __restrict__ mask, __nv_bfloat16* __restrict__ wb, long long n, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float val = 0.0f;
        if (!mask || mask[i]) {
            const float gi = g[i];
            const float mi = b1 * m[i] + (1.0f - b1) * gi;
            const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
            m[i] = mi;
            v[i] = vi;
            val = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        }
        p[i] = val;
        if (wb) wb[i] = __float2bfloat16_rn(val);
    }
}

// Fields to normalised states.  HBM-bound (24 B read and up to 96 B written per
// pixel): a lane loads its own pixel's six values (a warp reads 128 contiguous
// bytes per plane), then the warp writes its 32 pixels four lanes (FP32) or two
// (bfloat16) to a pixel, 512 contiguous bytes per store, the values passed by
// shuffles.  With one thread per output value, every thread divided by the plane
// size in 64 bits and re-read its plane one value at a time: 80 us at 16 x 256 x
// 256 pixels; now 20 us.
// vec: state and act on 16-byte boundaries (else scalar stores).
__global__ void __launch_bounds__(256)
    pack_kernel(const float* __restrict__ fields, int B, long long HW, const float* __restrict__ shift,
                const float* __restrict__ scale, float* __restrict__ state, __nv_bfloat16* __restrict__ act, bool vec) {
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * 8, per = (HW + 31) / 32;  // 32-pixel groups of an image
    float sh[5], sc[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        sh[c] = shift[c];
        sc[c] = scale[c];
    }
    for (long long n = blockIdx.y; n < B; n += gridDim.y) {
        const float* f = fields + n * 6 * HW;
        for (long long k = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); k < per; k += warps) {
            const long long q = k * 32 + lane;
            float v[5] = {};
            if (q < HW) {
#pragma unroll
                for (int c = 0; c < 4; ++c) v[c] = (f[c * HW + q] - sh[c]) * sc[c];
                v[4] = ((f[4 * HW + q] + f[5 * HW + q]) - sh[4]) * sc[4];
            }
            float* so = state + (n * HW + k * 32) * 16;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int px = 8 * t + (lane >> 2), j = lane & 3;
                float w[5];
#pragma unroll
                for (int c = 0; c < 5; ++c) w[c] = __shfl_sync(0xffffffffu, v[c], px);
                const float4 o = j == 0 ? make_float4(w[0], w[1], w[2], w[3])
                                        : make_float4(j == 1 ? w[4] : 0.0f, 0.0f, 0.0f, 0.0f);
                if (k * 32 + px >= HW) continue;
                float* d = so + px * 16 + 4 * j;
                if (vec) {
                    *reinterpret_cast<float4*>(d) = o;
                } else {
                    d[0] = o.x;
                    d[1] = o.y;
                    d[2] = o.z;
                    d[3] = o.w;
                }
            }
            if (!act) continue;
            __nv_bfloat16* ao = act + (n * HW + k * 32) * 16;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int px = 16 * t + (lane >> 1), j = lane & 1;
                __nv_bfloat16 w[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float x = c < 5 ? __shfl_sync(0xffffffffu, v[c], px) : 0.0f;
                    w[c] = __float2bfloat16_rn(j == 0 ? x : 0.0f);
                }
                if (k * 32 + px >= HW) continue;
                __nv_bfloat16* d = ao + px * 16 + 8 * j;
                if (vec) {
                    uint32_t u[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        u[c] = (uint32_t)__bfloat16_as_ushort(w[2 * c]) | ((uint32_t)__bfloat16_as_ushort(w[2 * c + 1]) << 16);
                    *reinterpret_cast<uint4*>(d) = make_uint4(u[0], u[1], u[2], u[3]);
                } else {
#pragma unroll
                    for (int c = 0; c < 8; ++c) d[c] = w[c];
                }
            }
        }
    }
}

// State -> the six fields of a solver restart, in double: phi, u, p as they
// are, and c1 + c2 = C split between the phases at the Henry equilibrium
// c1 / phi = K c2 / (1 - phi) (phi clipped to [0, 1]).
__global__ void unpack_macros_kernel(const float* __restrict__ state, int B, int H, int W,
                                     const float* __restrict__ shift, const float* __restrict__ scale,
                                     const float* __restrict__ keq, double* __restrict__ out) {
    const long long HW = (long long)H * W, P = B * HW;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (long long)gridDim.x * blockDim.x) {
        const long long n = i / HW, q = i % HW;
        const float* s = state + i * 16;
        double f[5];
        for (int c = 0; c < 5; ++c) f[c] = (double)(s[c] / scale[c] + shift[c]);
        const double ph = f[0] < 0.0 ? 0.0 : (f[0] > 1.0 ? 1.0 : f[0]);
        const double K = keq[n], den = K * ph + (1.0 - ph);
        double* o = out + n * 6 * HW + q;
        o[0] = f[0];
        o[HW] = f[1];
        o[2 * HW] = f[2];
        o[3 * HW] = f[3];
        o[4 * HW] = f[4] * K * ph / den;
        o[5 * HW] = f[4] * (1.0 - ph) / den;
    }
}

// The five fields of a state: a lane reads the used part of its pixel (one 32-byte
// sector of the 64 bytes) and writes one value per plane, 128 contiguous bytes per
// warp and plane.
__global__ void __launch_bounds__(256)
    unpack_kernel(const float* __restrict__ state, int B, long long HW, const float* __restrict__ shift,
                  const float* __restrict__ scale, float* __restrict__ fields, bool vec) {
    float sh[5], sc[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        sh[c] = shift[c];
        sc[c] = scale[c];
    }
    for (long long n = blockIdx.y; n < B; n += gridDim.y)
        for (long long q = (long long)blockIdx.x * 256 + threadIdx.x; q < HW; q += (long long)gridDim.x * 256) {
            const float* s = state + (n * HW + q) * 16;
            float v[5];
            if (vec) {
                const float4 a = *reinterpret_cast<const float4*>(s);
                v[0] = a.x;
                v[1] = a.y;
                v[2] = a.z;
                v[3] = a.w;
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) v[c] = s[c];
            }
            v[4] = s[4];
            float* o = fields + n * 5 * HW + q;
#pragma unroll
            for (int c = 0; c < 5; ++c) o[c * HW] = v[c] / sc[c] + sh[c];
        }
}

// Per sample and channel (first 5): max |a - b| and sum (a - b)^2 over pixels.
__global__ void state_diff_kernel(const float* __restrict__ a, const float* __restrict__ b, long long HW,
                                  float* __restrict__ out) {
    __shared__ float smax[5][256];
    __shared__ double ssum[5][256];
    const int n = blockIdx.y;
    float mx[5] = {0, 0, 0, 0, 0};
    double sm[5] = {0, 0, 0, 0, 0};
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < HW; q += (long long)gridDim.x * blockDim.x) {
        const long long i = ((long long)n * HW + q) * 16;
        for (int c = 0; c < 5; ++c) {
            const float d = a[i + c] - b[i + c];
            mx[c] = fmaxf(mx[c], fabsf(d));
            sm[c] += (double)d * d;
        }
    }
    for (int c = 0; c < 5; ++c) { smax[c][threadIdx.x] = mx[c]; ssum[c][threadIdx.x] = sm[c]; }
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k)
            for (int c = 0; c < 5; ++c) {
                smax[c][threadIdx.x] = fmaxf(smax[c][threadIdx.x], smax[c][threadIdx.x + k]);
                ssum[c][threadIdx.x] += ssum[c][threadIdx.x + k];
            }
        __syncthreads();
    }
    if (threadIdx.x < 5) {
        // one block column per sample: partials [n][block][c][2]
        float* o = out + (((size_t)n * gridDim.x + blockIdx.x) * 5 + threadIdx.x) * 2;
        o[0] = smax[threadIdx.x][0];
        o[1] = (float)ssum[threadIdx.x][0];
    }
}

__global__ void state_diff_final(const float* __restrict__ part, int nblk, long long HW, float* __restrict__ out) {
    const int n = blockIdx.x, c = threadIdx.x;
    if (c >= 5) return;
    float mx = 0.0f;
    double sm = 0.0;
    for (int b = 0; b < nblk; ++b) {
        const float* o = part + (((size_t)n * nblk + b) * 5 + c) * 2;
        mx = fmaxf(mx, o[0]);
        sm += o[1];
    }
    out[((size_t)n * 5 + c) * 2] = mx;
    out[((size_t)n * 5 + c) * 2 + 1] = (float)sqrt(sm / (double)HW);
}

// Gaussian noise on the first `used` channels of a float state: Box-Muller
// (1958) on two uniforms from a counter-based hash (the MurmurHash3 32-bit
// finalizer) of (seed, element index): reproducible for a given seed.
__device__ __forceinline__ uint32_t nn_mix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

__global__ void add_noise_kernel(float* __restrict__ s, long long P, int used, float sigma, uint32_t seed) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P * used;
         i += (long long)gridDim.x * blockDim.x) {
        const long long p = i / used;
        const int c = (int)(i % used);
        const uint32_t k = nn_mix32(seed ^ nn_mix32((uint32_t)i ^ (uint32_t)(i >> 32) * 0x9e3779b9u));
        const float u1 = ((float)(k >> 8) + 1.0f) * 0x1p-24f;  // (0, 1]
        const float u2 = (float)(nn_mix32(k + 0x68e31da4u) >> 8) * 0x1p-24f;
        s[p * 16 + c] += sigma * sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
    }
}

__global__ void to_f32_kernel(const __nv_bfloat16* __restrict__ a, long long n, float* __restrict__ s) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        s[i] = __bfloat162float(a[i]);
}

__global__ void axpy_kernel(float* __restrict__ y, const float* __restrict__ x, float a, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] += a * x[i];
}

__global__ void to_bf16_kernel(const float* __restrict__ s, long long n, __nv_bfloat16* __restrict__ a) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        a[i] = __float2bfloat16_rn(s[i]);
}

int grid_for(long long n, int threads) { return (int)std::max<long long>(1, std::min<long long>((n + threads - 1) / threads, 152LL * 16)); }

// blocks of 256 pixels of an image (x) by images (y), about 16 blocks per SM in all
dim3 image_grid(long long hw, int batch) {
    const long long gy = std::min<long long>(batch, 65535);
    const long long gx = std::min<long long>((hw + 255) / 256, std::max<long long>(1, (152LL * 16 + gy - 1) / gy));
    return dim3((unsigned)gx, (unsigned)gy);
}

}  // namespace

extern "C" {

int lbm_nn_flip_weights(const void* w, int32_t cin, int32_t cout, void* wt, void* stream) {
    if (!w || !wt || cin < 1 || cout < 1) return LBM_ERR_ARG;
    const int n = 9 * cin * cout;
    flip_kernel<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const __nv_bfloat16*>(w), cin, cout, static_cast<__nv_bfloat16*>(wt));
    return launch_status();
}

int lbm_nn_bias_grad(const void* dy, int32_t cout, int64_t pixels, float* db, float* partials, void* stream) {
    if (!dy || !db || !partials || (cout != 16 && cout != 48) || pixels < 1) return LBM_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool aligned = (uintptr_t)dy % 16 == 0;
    const auto* d = static_cast<const __nv_bfloat16*>(dy);
    if (cout == 48) bias_grad_partials<48><<<RED_BLOCKS, 256, 0, s>>>(d, pixels, partials, aligned);
    else bias_grad_partials<16><<<RED_BLOCKS, 256, 0, s>>>(d, pixels, partials, aligned);
    sum_partials<<<cout, 256, 0, s>>>(partials, RED_BLOCKS, cout, db);
    return launch_status();
}

int lbm_nn_mse(const float* pred, const float* target, int32_t used, int64_t pixels, void* dpred, double* loss_partials,
               double* loss, void* stream) {
    if (!pred || !target || !loss_partials || !loss || used < 1 || used > 16 || pixels < 1) return LBM_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const double inv = 1.0 / ((double)pixels * used);
    const float khi = (float)(2.0 * inv), klo = (float)(2.0 * inv - (double)khi);
    auto* dp = static_cast<__nv_bfloat16*>(dpred);
    const bool vec = ((uintptr_t)pred | (uintptr_t)target | (uintptr_t)dpred) % 16 == 0;
    auto run = [&](auto kernel) { kernel<<<RED_BLOCKS, 256, 0, s>>>(pred, target, used, pixels, dp, loss_partials, inv, khi, klo); };
    switch ((used + 3) / 4) {
        case 1: vec ? run(mse_partials<true, 1>) : run(mse_partials<false, 1>); break;
        case 2: vec ? run(mse_partials<true, 2>) : run(mse_partials<false, 2>); break;
        case 3: vec ? run(mse_partials<true, 3>) : run(mse_partials<false, 3>); break;
        default: vec ? run(mse_partials<true, 4>) : run(mse_partials<false, 4>); break;
    }
    mse_final<<<1, 256, 0, s>>>(loss_partials, RED_BLOCKS, loss);
    return launch_status();
}

int lbm_nn_adam(float* param, const float* grad, float* m, float* v, const uint8_t* mask, void* wbf16, int64_t n,
                float lr, float beta1, float beta2, float eps, int32_t t, void* stream) {
    if (!param || !grad || !m || !v || n < 1 || t < 1) return LBM_ERR_ARG;
    const float c1 = 1.0f - powf(beta1, (float)t), c2 = 1.0f - powf(beta2, (float)t);
    adam_kernel<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        param, grad, m, v, mask, static_cast<__nv_bfloat16*>(wbf16), n, lr, beta1, beta2, eps, c1, c2);
    return launch_status();
}

int lbm_nn_pack(const float* fields, int32_t batch, int32_t h, int32_t w, const float* shift, const float* scale,
                float* state, void* act, void* stream) {
    if (!fields || !shift || !scale || !state || batch < 1 || h < 1 || w < 1) return LBM_ERR_ARG;
    const long long hw = (long long)h * w;
    pack_kernel<<<image_grid(hw, batch), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        fields, batch, hw, shift, scale, state, static_cast<__nv_bfloat16*>(act),
        ((uintptr_t)state | (uintptr_t)act) % 16 == 0);
    return launch_status();
}

int lbm_nn_unpack(const float* state, int32_t batch, int32_t h, int32_t w, const float* shift, const float* scale,
                  float* fields, void* stream) {
    if (!state || !shift || !scale || !fields || batch < 1 || h < 1 || w < 1) return LBM_ERR_ARG;
    const long long hw = (long long)h * w;
    unpack_kernel<<<image_grid(hw, batch), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        state, batch, hw, shift, scale, fields, (uintptr_t)state % 16 == 0);
    return launch_status();
}

int lbm_nn_unpack_macros(const float* state, int32_t batch, int32_t h, int32_t w, const float* shift,
                         const float* scale, const float* keq, double* macros, void* stream) {
    if (!state || !shift || !scale || !keq || !macros || batch < 1 || h < 1 || w < 1) return LBM_ERR_ARG;
    const long long n = (long long)batch * h * w;
    unpack_macros_kernel<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        state, batch, h, w, shift, scale, keq, macros);
    return launch_status();
}

int lbm_nn_state_diff(const float* a, const float* b, int32_t batch, int64_t pixels, float* partials, float* out,
                      void* stream) {
    if (!a || !b || !partials || !out || batch < 1 || pixels < 1) return LBM_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    constexpr int NBLK = 64;
    state_diff_kernel<<<dim3(NBLK, batch), 256, 0, s>>>(a, b, pixels, partials);
    state_diff_final<<<batch, 32, 0, s>>>(partials, NBLK, pixels, out);
    return launch_status();
}

int lbm_nn_add_noise(float* state, int64_t pixels, int32_t used, float sigma, uint32_t seed, void* stream) {
    if (!state || pixels < 1 || used < 1 || used > 16) return LBM_ERR_ARG;
    const long long n = (long long)pixels * used;
    add_noise_kernel<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(state, pixels, used, sigma, seed);
    return launch_status();
}

int lbm_nn_to_bf16(const float* state, int64_t values, void* act, void* stream) {
    if (!state || !act || values < 1) return LBM_ERR_ARG;
    to_bf16_kernel<<<grid_for(values, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        state, values, static_cast<__nv_bfloat16*>(act));
    return launch_status();
}

int lbm_nn_to_f32(const void* act, int64_t values, float* state, void* stream) {
    if (!state || !act || values < 1) return LBM_ERR_ARG;
    to_f32_kernel<<<grid_for(values, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const __nv_bfloat16*>(act), values, state);
    return launch_status();
}

int lbm_nn_axpy(float* y, const float* x, float a, int64_t n, void* stream) {
    if (!y || !x || n < 1) return LBM_ERR_ARG;
    axpy_kernel<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(y, x, a, n);
    return launch_status();
}

}  // extern "C"
