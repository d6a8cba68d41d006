// Learned plane proposals: a small U-Net that maps the reference image and an
// early PatchMatch state to K = 4 plane hypotheses per pixel, trained on the
// depth maps the plain pipeline produces.  (No counterpart in the paper; the
// proposals only add candidates to the propagation step, the ZNCC cost of
// Eq. 4/5 still decides.)
//
// Tensors are channels-last bfloat16 (pixel-major, channels contiguous, a
// multiple of 16 channels); convolutions are implicit GEMMs on the
// fifth-generation tensor cores (conv_tc.cu: TMA-staged operands,
// tcgen05.mma bf16 x bf16 -> fp32 in tensor memory): M = pixels, N = output
// channels, K = taps x input channels.  The data gradient is the same kernel
// run on the output gradient with flipped, transposed weights; the weight
// gradient is a tensor-core reduction over pixels.  Master weights, gradients
// and Adam moments are fp32.
#include <atomic>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/mvs.h"
#include "conv_tc.h"
#include "mvs_internal.h"
#include "pm_device.cuh"

namespace {

typedef __nv_bfloat16 bf16;

struct Mat3 {
    float m[9];
};

// Weight gradient: dw[co][tap][ci] += sum_p dy[p][co] * x[p + tap][ci],
// db[co] += sum_p dy[p][co]: a contraction over pixels with both operands
// channels-last, i.e. pixel-major.  A warp owns 16 output x 16 input channels
// and all taps (72 fp32 accumulators per lane) and takes 16 pixels of a row per
// step with mma.m16n8k16 (bf16 products are exact, sums fp32); a tap is only
// another row of the staged input, so one fragment of dy serves the nine taps.
// mma.sync and not tcgen05: the layers' 16..128 output channels would fill at
// most one 128-row tile, mostly padding, and the transposed fragment loads come
// with ldmatrix.  A block covers kWgSeg pixels x `rows` image rows and up to 16
// warps of channel tiles; input rows pass through a ring of four (each is read
// once per block and used by three output rows), the next row arriving by
// cp.async while the current one is multiplied.  Bound by the latency of the
// chain fragment load, product, product with 4 to 16 warps per multiprocessor
// (128 registers; full-resolution layers: 30 % of the issue slots, 24 to 43 % of
// the shared-memory pipe) and, on the small levels, by the atomic sums of few
// blocks.  512 x 384, all ten layers: 184 us against 1730 us for the fp32 SIMT
// reduction it replaces; the tensor core's fp32 sums differ from its one rounded
// multiply-add per product by about 2e-6 relative.
constexpr int kWgSeg = 64;
struct WgradArgs {
    const bf16* x;
    const bf16* dy;
    int Cin, Cout, W, H, taps, rows;
    int ct, it;               // channel tiles of 16 per block: output, input
    float *dw, *db;
};

__device__ __forceinline__ void ldsm_t(uint32_t a, uint32_t r[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// 16 bytes from global to shared memory in the background, or zeros
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// bytes of a staged pixel: an odd number of 16-byte groups, so that the eight
// rows of a fragment load fall on different banks
__host__ __device__ inline uint32_t wg_pixel_bytes(int ch) { return (uint32_t)ch * 2u + 16u; }
inline size_t wg_smem(int ct, int it, int taps) {
    return (size_t)(taps == 9 ? 4 * (kWgSeg + 2) : 2 * kWgSeg) * wg_pixel_bytes(16 * it) +
           (size_t)2 * kWgSeg * wg_pixel_bytes(16 * ct);
}

template <int TAPS>
__global__ void __launch_bounds__(512, 1) k_conv_wgrad(const __grid_constant__ WgradArgs a) {
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int HALO = TAPS == 9 ? 1 : 0, RING = TAPS == 9 ? 4 : 2, SEGX = kWgSeg + 2 * HALO;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int segs = (a.W + kWgSeg - 1) / kWgSeg;
    const int x0 = (blockIdx.x % segs) * kWgSeg, y0 = (blockIdx.x / segs) * a.rows, y1 = min(a.H, y0 + a.rows);
    const int ci0 = blockIdx.y * a.it * 16, nci = min(a.it * 16, a.Cin - ci0), nco = a.ct * 16;
    const int seg = min(kWgSeg, a.W - x0);
    const uint32_t xb = wg_pixel_bytes(16 * a.it), yb = wg_pixel_bytes(nco);
    const uint32_t xs = (uint32_t)__cvta_generic_to_shared(sm), ys = xs + RING * SEGX * xb;
    auto load_x = [&](int y) {        // row y of the input with its halo, zero outside the image
        const int v = nci / 8;
        const uint32_t d = xs + (uint32_t)((y + RING) % RING) * SEGX * xb;
        const bool in = y >= 0 && y < a.H;
        for (int i = threadIdx.x; i < SEGX * v; i += blockDim.x) {
            const int p = i / v, c = i - p * v, px = x0 + p - HALO;
            const bool ok = in && px >= 0 && px < a.W;
            copy16(d + (uint32_t)p * xb + 16u * c, a.x + (ok ? ((long long)y * a.W + px) * a.Cin + ci0 + 8 * c : 0), ok);
        }
    };
    auto load_dy = [&](int y) {       // zero past the end of the row
        const int v = nco / 8;
        const uint32_t d = ys + (uint32_t)(y & 1) * kWgSeg * yb;
        for (int i = threadIdx.x; i < kWgSeg * v; i += blockDim.x) {
            const int p = i / v, c = i - p * v;
            const bool ok = p < seg;
            copy16(d + (uint32_t)p * yb + 16u * c, a.dy + (ok ? ((long long)y * a.W + x0 + p) * a.Cout + 8 * c : 0), ok);
        }
    };
    const int wc = warp % a.ct, wi = warp / a.ct;
    const bool active = wi * 16 < nci;
    const bool bias = a.db && blockIdx.y == 0 && wi == 0;
    float acc[TAPS][2][4] = {}, bacc[4] = {0.f, 0.f, 0.f, 0.f};
    // fragment rows of this lane (see mma.m16n8k16): A is dy transposed, B the input
    const uint32_t ya = (uint32_t)((lane & 7) + (lane >> 4) * 8) * yb + (uint32_t)(wc * 32 + ((lane >> 3) & 1) * 16);
    const uint32_t xa = (uint32_t)((lane & 7) + ((lane >> 3) & 1) * 8) * xb + (uint32_t)(wi * 32 + (lane >> 4) * 16);

    if (HALO) {
        load_x(y0 - 1);
        load_x(y0);
    }
    load_x(y0 + HALO);
    load_dy(y0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int y = y0; y < y1; ++y) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();              // row y (and its halo) has arrived; row y - 1's buffers are free
        if (y + 1 < y1) {
            load_x(y + 1 + HALO);
            load_dy(y + 1);
        }
        if (active) {
            for (int k = 0; k < seg; k += 16) {
                uint32_t fa[4];
                ldsm_t(ys + (uint32_t)(y & 1) * kWgSeg * yb + (uint32_t)k * yb + ya, fa);
#pragma unroll
                for (int r = 0; r < (TAPS == 9 ? 3 : 1); ++r) {
                    const uint32_t row = xs + (uint32_t)((y + r - HALO + RING) % RING) * SEGX * xb + xa;
#pragma unroll
                    for (int c = 0; c < (TAPS == 9 ? 3 : 1); ++c) {
                        uint32_t fb[4];
                        ldsm_t(row + (uint32_t)(k + c) * xb, fb);
                        mma16816(acc[3 * r + c][0], fa, fb[0], fb[1]);
                        mma16816(acc[3 * r + c][1], fa, fb[2], fb[3]);
                    }
                }
                if (bias) mma16816(bacc, fa, 0x3F803F80u, 0x3F803F80u);   // bf16 ones: the sum over pixels
            }
        }
    }
    if (!active) return;
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int tap = 0; tap < TAPS; ++tap)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int co = wc * 16 + g + 8 * h, ci = ci0 + wi * 16 + 8 * n + 2 * t;
                atomicAdd(reinterpret_cast<float2*>(a.dw + ((long long)co * TAPS + tap) * a.Cin + ci),
                          make_float2(acc[tap][n][2 * h], acc[tap][n][2 * h + 1]));
            }
    if (bias && t == 0) {
        atomicAdd(a.db + wc * 16 + g, bacc[0]);
        atomicAdd(a.db + wc * 16 + g + 8, bacc[2]);
    }
}

// ---------------------------------------------------------------------------
// elementwise pieces
// ---------------------------------------------------------------------------
// Eight bf16 channels as floats, and back (rounded)
__device__ __forceinline__ void unpack8(uint4 q, float f[8]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t w = (&q.x)[k];
        const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
        f[2 * k] = v.x;
        f[2 * k + 1] = v.y;
    }
}
__device__ __forceinline__ uint4 pack8(const float f[8]) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
        w[k] = *reinterpret_cast<uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// g where the activation is positive, else zero (the gradient through ReLU)
__device__ __forceinline__ void relu_mask8(float g[8], uint4 y) {
    float a[8];
    unpack8(y, a);
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (!(a[k] > 0.0f)) g[k] = 0.0f;
}

// Backward data movement, 8 channels (16 bytes) per thread, each level's
// gradient written once: the split of the concatenation, the sum with the
// pooling's gradient and the ReLU mask were passes of their own.
// Gradient of an encoder level l < 4: mask(e) * (skip channels of gc + 1/4 of
// gp at the parent pixel), the sum rounded to bf16.
__global__ void k_enc_grad(const uint4* __restrict__ gc, int gc_v, int off_v, const uint4* __restrict__ gp,
                           const uint4* __restrict__ e, int W, int H, int cv, uint4* __restrict__ ge) {
    const int n = W * H * cv;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int p = i / cv, c = i - p * cv, y = p / W, x = p - y * W;
        float a[8], b[8];
        unpack8(gc[(long long)p * gc_v + off_v + c], a);
        unpack8(gp[((long long)(y / 2) * (W / 2) + x / 2) * cv + c], b);
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = __fadd_rn(0.25f * b[k], a[k]);
        relu_mask8(a, e[i]);
        ge[i] = pack8(a);
    }
}

// Gradient through the up-sampling and the ReLU below it: mask(act) * (sum of
// the four children of channels [0, 8 cv) of gc (W x H)), for W/2 x H/2
__global__ void k_up_grad(const uint4* __restrict__ gc, int gc_v, const uint4* __restrict__ act, int W, int H, int cv,
                          uint4* __restrict__ out) {
    const int Wo = W / 2, n = Wo * (H / 2) * cv;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int p = i / cv, c = i - p * cv, y = p / Wo, x = p - y * Wo;
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float a[8];
                unpack8(gc[((long long)(2 * y + j) * W + 2 * x + q) * gc_v + c], a);
#pragma unroll
                for (int k = 0; k < 8; ++k) s[k] += a[k];
            }
        relu_mask8(s, act[i]);
        out[i] = pack8(s);
    }
}

// gradient through ReLU: g *= (y > 0)
__global__ void k_relu_mask(uint4* __restrict__ g, const uint4* __restrict__ y, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float a[8];
        unpack8(g[i], a);
        relu_mask8(a, y[i]);
        g[i] = pack8(a);
    }
}

// Forward-pass data movement in 16-byte vectors (8 channels per thread,
// channel counts are multiples of 16, rows of pixels at most 8192 wide).
// 2 x 2 average pooling: out (W/2 x H/2, C) from in (W x H, C), summed in
// the order (0,0), (0,1), (1,0), (1,1) and scaled by 1/4 in fp32.
__global__ void k_pool_fwd_v(const uint4* __restrict__ in, int W, int H, int C, uint4* __restrict__ out) {
    const int cv = C / 8, Wo = W / 2;
    const long long n = (long long)Wo * (H / 2) * cv;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % cv);
        const int p = (int)(i / cv), x = p % Wo, y = p / Wo;
        const uint4 q[4] = {in[((long long)(2 * y) * W + 2 * x) * cv + c], in[((long long)(2 * y) * W + 2 * x + 1) * cv + c],
                            in[((long long)(2 * y + 1) * W + 2 * x) * cv + c],
                            in[((long long)(2 * y + 1) * W + 2 * x + 1) * cv + c]};
        uint32_t r[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t w = (&q[j].x)[k];
                const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
                s.x += f.x;
                s.y += f.y;
            }
            __nv_bfloat162 h = __floats2bfloat162_rn(0.25f * s.x, 0.25f * s.y);
            r[k] = *reinterpret_cast<uint32_t*>(&h);
        }
        out[i] = make_uint4(r[0], r[1], r[2], r[3]);
    }
}

__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       long long n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float gi = g[i];
        float mi = b1 * m[i] + (1.0f - b1) * gi, vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// ---------------------------------------------------------------------------
// proposal head: 16 outputs per pixel = 4 x (a, nx, ny, nz); inverse depth
// rho = 1/d_hi + (1/d_lo - 1/d_hi) sigmoid(a), normal = (nx, ny, nz) / norm
// ---------------------------------------------------------------------------
struct HeadConst {
    float rho_lo, rho_hi;   // 1/d_hi, 1/d_lo
    float lambda_n;         // weight of the normal term
};

__device__ __forceinline__ void decode(const float* o, const HeadConst& hc, float& rho, float n[3], float& len,
                                       float& sig) {
    sig = 1.0f / (1.0f + expf(-o[0]));
    rho = hc.rho_lo + (hc.rho_hi - hc.rho_lo) * sig;
    len = sqrtf(o[1] * o[1] + o[2] * o[2] + o[3] * o[3]) + 1e-12f;
    n[0] = o[1] / len; n[1] = o[2] / len; n[2] = o[3] / len;
}

// per pixel with a target: loss = min_k |rho_k - rho_t| / (rho_hi - rho_lo)
// + lambda (1 - |n_k . n_t|), rho_t = 1 / target depth; the first k wins
// ties.  L = scale * sum over target pixels; writes dL/d out rounded to bf16
// and adds L to *loss_sum.
__global__ void k_proposal_loss(const float* __restrict__ out, const float4* __restrict__ target,
                                const uint8_t* __restrict__ mask, long long npix, HeadConst hc, float scale,
                                uint4* __restrict__ grad, float* __restrict__ loss_sum) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    float lsum = 0.0f;
    if (i < npix) {
        uint4 q[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
        if (mask[i]) {
            // the head's 16 outputs in 16-byte loads
            alignas(16) float outv[16];
#pragma unroll
            for (int k = 0; k < 4; ++k) reinterpret_cast<float4*>(outv)[k] = reinterpret_cast<const float4*>(out)[4 * i + k];
            const float4 t4 = target[i];
            const float tp[4] = {1.0f / t4.w, t4.x, t4.y, t4.z};
            const float span = hc.rho_hi - hc.rho_lo;
            int best = 0;
            float bl = 3.0e38f, o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float rho, n[3], len, sig;
                decode(outv + 4 * k, hc, rho, n, len, sig);
                float l = fabsf(rho - tp[0]) / span + hc.lambda_n * (1.0f - fabsf(n[0] * tp[1] + n[1] * tp[2] + n[2] * tp[3]));
                if (l < bl) {
                    bl = l;
                    best = k;
#pragma unroll
                    for (int c = 0; c < 4; ++c) o[c] = outv[4 * k + c];
                }
            }
            float rho, n[3], len, sig, gp[4];
            decode(o, hc, rho, n, len, sig);
            float sgn = rho > tp[0] ? 1.0f : (rho < tp[0] ? -1.0f : 0.0f);
            gp[0] = scale * sgn * sig * (1.0f - sig);
            float dot = n[0] * tp[1] + n[1] * tp[2] + n[2] * tp[3];
            float sd = dot > 0.0f ? 1.0f : (dot < 0.0f ? -1.0f : 0.0f);
#pragma unroll
            for (int c = 0; c < 3; ++c) gp[1 + c] = scale * hc.lambda_n * (-sd) * (tp[1 + c] - dot * n[c]) / len;
            const __nv_bfloat162 h0 = __floats2bfloat162_rn(gp[0], gp[1]), h1 = __floats2bfloat162_rn(gp[2], gp[3]);
            const uint32_t w0 = *reinterpret_cast<const uint32_t*>(&h0), w1 = *reinterpret_cast<const uint32_t*>(&h1);
            uint4& b = q[best >> 1];
            if (best & 1) { b.z = w0; b.w = w1; } else { b.x = w0; b.y = w1; }
            lsum = bl * scale;
        }
        grad[2 * i] = q[0];
        grad[2 * i + 1] = q[1];
    }
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if ((threadIdx.x & 31) == 0 && lsum != 0.0f) atomicAdd(loss_sum, lsum);
}

// decode the head into K = 4 planes per pixel (n facing the camera, depth),
// one proposal per thread (one 16-byte load and store)
__global__ void k_decode_proposals(const float4* __restrict__ out, long long npix, int W, HeadConst hc, Mat3 Kinv,
                                   float4* __restrict__ props) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= 4 * npix) return;
    const int i = (int)(t >> 2), y = i / W, x = i - y * W;   // at most 8192 x 8192 pixels
    float r0 = Kinv.m[0] * x + Kinv.m[1] * y + Kinv.m[2], r1 = Kinv.m[3] * x + Kinv.m[4] * y + Kinv.m[5];
    float r2 = Kinv.m[6] * x + Kinv.m[7] * y + Kinv.m[8];
    const float4 v = out[t];
    const float o[4] = {v.x, v.y, v.z, v.w};
    float rho, n[3], len, sig;
    decode(o, hc, rho, n, len, sig);
    if (n[0] * r0 + n[1] * r1 + n[2] * r2 > 0.0f) { n[0] = -n[0]; n[1] = -n[1]; n[2] = -n[2]; }
    props[t] = make_float4(n[0], n[1], n[2], 1.0f / rho);
}

// network input (16 channels, bf16): image / 255, normalised inverse depth,
// normal (3), cost / 2, zeros
__global__ void k_make_input(const uint8_t* __restrict__ img, const float4* __restrict__ plane,
                             const float* __restrict__ cost, long long npix, HeadConst hc, bf16* __restrict__ in) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= npix) return;
    float4 p = plane[i];
    float rho = p.w > 0.0f ? 1.0f / p.w : hc.rho_lo;
    float v[6] = {img[i] / 255.0f, (rho - hc.rho_lo) / (hc.rho_hi - hc.rho_lo), p.x, p.y, p.z, cost[i] * 0.5f};
    uint32_t w[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * c], v[2 * c + 1]);
        w[c] = *reinterpret_cast<uint32_t*>(&h);
    }
    uint4* o = reinterpret_cast<uint4*>(in + 16 * i);
    o[0] = make_uint4(w[0], w[1], w[2], 0u);
    o[1] = make_uint4(0u, 0u, 0u, 0u);
}

unsigned blocks(long long n, int b = 256) {
    long long g = (n + b - 1) / b;
    return (unsigned)(g > 152LL * 32 ? 152LL * 32 : (g < 1 ? 1 : g));
}

}  // namespace

// ===========================================================================
// host side: the network, its buffers and the C ABI
// ===========================================================================
namespace {

struct Layer {
    int cin, cout, taps;
    bool relu;
    size_t nw;                     // cout * taps * cin
    float *w, *b, *gw, *gb;
    bf16 *wt, *wtf;                // bf16 B operands of the tensor-core convolution: forward, data gradient
};

// channel plan (level l has 1/2^l resolution)
enum { E0, E1, E2, E3, E4, D3, D2, D1, D0, HEAD, NL };
const int kLayerCin[NL] = {16, 32, 48, 64, 96, 224, 160, 112, 80, 32};
const int kLayerCout[NL] = {32, 48, 64, 96, 128, 96, 64, 48, 32, 16};

cudaError_t g_cnn_err = cudaSuccess;

// widest level-0 image that training takes (the widest that the layer tests
// check; no kernel needs the limit)
constexpr int kMaxTrainWidth = 768;

}  // namespace

struct mvs_cnn {
    int maxW = 0, maxH = 0;
    cudaStream_t stream = nullptr;
    HeadConst hc;
    Layer L[NL];
    // activations (bf16, channels last)
    bf16 *x = nullptr, *e[5] = {}, *p[4] = {}, *c[4] = {}, *d[4] = {};
    float* y = nullptr;            // head output, 16 channels fp32
    // gradients
    bf16 *gyb = nullptr, *gd[4] = {}, *gc[4] = {}, *ge[5] = {}, *gp[4] = {};
    // parameters, gradients and Adam moments, layer by layer: weights then biases
    float *theta = nullptr, *grad = nullptr, *mom = nullptr, *var = nullptr;
    size_t n_theta = 0;
    float* loss = nullptr;
    int* status = nullptr;         // device word: MVS_DEV_TIMEOUT once a bounded wait of a convolution ran out
    int steps = 0;
    int lastW = 0, lastH = 0;      // size of the last forward pass
    std::string err;
    std::vector<void*> allocs;
};

namespace {

template <typename T>
cudaError_t cnn_alloc(mvs_cnn* n, T** p, size_t count) {
    cudaError_t e = cudaMalloc((void**)p, count * sizeof(T) + 256);
    if (e == cudaSuccess) n->allocs.push_back((void*)*p);
    return e;
}

// wait limit of the convolutions' mbarriers (polls, with a 64 ns back-off):
// about a second
constexpr unsigned kConvWaitLimit = 1u << 24;

// One tensor-core convolution; `status` collects a timed-out wait.
cudaError_t conv_launch(mvs_cnn* n, const bf16* in, int Cin, int W, int H, const bf16* wt, const float* bias,
                        int taps, int Cout, bool relu, bool out_f32, void* out, int out_ch, int out_off,
                        cudaStream_t s, const ConvExtra& extra = ConvExtra());

cudaError_t wgrad_launch(const bf16* x, int Cin, const bf16* dy, int Cout, int W, int H, int taps, float* dw, float* db,
                         cudaStream_t s) {
    WgradArgs a{x, dy, Cin, Cout, W, H, taps, 0, Cout / 16, 0, dw, db};
    // input-channel tiles per block: as even a split as gives at most 16 warps
    const int nit = Cin / 16, most = std::max(1, 16 / a.ct), gy = (nit + most - 1) / most;
    a.it = (nit + gy - 1) / gy;
    const int warps = a.ct * a.it, segs = (W + kWgSeg - 1) / kWgSeg;
    // image rows per block: enough blocks for about 16 warps per SM, since every
    // block re-reads two halo rows and adds its sums to the whole gradient
    const long long want = 152LL * std::max(1, 16 / warps);
    a.rows = (int)std::max<long long>(2, ((long long)H * segs * gy + want - 1) / want);
    const dim3 grid((unsigned)(segs * ((H + a.rows - 1) / a.rows)), (unsigned)gy);
    const size_t smem = wg_smem(a.ct, a.it, taps);
    const void* fn = taps == 9 ? (const void*)k_conv_wgrad<9> : (const void*)k_conv_wgrad<1>;
    // the shared-memory opt-in is a property of the current device
    static std::atomic<bool> attr[128][2];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
    if (!attr[dev][taps == 9].load()) {
        if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024)) != cudaSuccess)
            return e;
        attr[dev][taps == 9].store(true);
    }
    if (taps == 9) k_conv_wgrad<9><<<grid, 32 * warps, smem, s>>>(a);
    else k_conv_wgrad<1><<<grid, 32 * warps, smem, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

#define CUK(call)                         \
    do {                                  \
        cudaError_t _e = (call);          \
        if (_e != cudaSuccess) return _e; \
    } while (0)

cudaError_t refresh_bf16(mvs_cnn* n) {
    for (int i = 0; i < NL; ++i) {
        Layer& L = n->L[i];
        CUK(conv_tc_weights(L.w, L.cout, L.taps, L.cin, 0, L.wt, n->stream));
        CUK(conv_tc_weights(L.w, L.cout, L.taps, L.cin, 1, L.wtf, n->stream));
    }
    return cudaGetLastError();
}

cudaError_t conv_launch(mvs_cnn* n, const bf16* in, int Cin, int W, int H, const bf16* wt, const float* bias,
                        int taps, int Cout, bool relu, bool out_f32, void* out, int out_ch, int out_off,
                        cudaStream_t s, const ConvExtra& extra) {
    return conv_tc_launch(in, Cin, W, H, wt, bias, taps, Cout, relu, out_f32, out, out_ch, out_off, extra, n->status, 0,
                          kConvWaitLimit, s);
}

// forward pass; x must hold the 16-channel input of a W x H image
cudaError_t cnn_forward(mvs_cnn* n, int W, int H) {
    cudaStream_t s = n->stream;
    auto C = [&](int l) -> const Layer& { return n->L[l]; };
    int Ws[5], Hs[5];
    for (int l = 0; l < 5; ++l) { Ws[l] = W >> l; Hs[l] = H >> l; }
    // decoder input of level l: c[l] = [up(d[l + 1] or e[4]) | e[l]], each part
    // written by the convolution that computes it
    auto cat_ch = [&](int l) { return C(D3 + (3 - l)).cin; };
    // encoder
    const bf16* in = n->x;
    for (int l = 0; l <= 4; ++l) {
        const Layer& L = C(E0 + l);
        ConvExtra x;
        if (l < 4) {
            x.skip = n->c[l];
            x.skip_ch = cat_ch(l);
            x.skip_off = cat_ch(l) - L.cout;
            if (conv_tc_can_pool(9, L.cout, Ws[l], Hs[l])) x.pool = n->p[l];
        } else {
            x.up = n->c[3];
            x.up_ch = cat_ch(3);
        }
        CUK(conv_launch(n, in, L.cin, Ws[l], Hs[l], L.wt, L.b, 9, L.cout, true, false, n->e[l], L.cout, 0, s, x));
        if (l < 4) {
            if (!x.pool) {
                k_pool_fwd_v<<<blocks((long long)Ws[l + 1] * Hs[l + 1] * L.cout / 8), 256, 0, s>>>(
                    reinterpret_cast<const uint4*>(n->e[l]), Ws[l], Hs[l], L.cout, reinterpret_cast<uint4*>(n->p[l]));
                count_launch();
            }
            in = n->p[l];
        }
    }
    // decoder: level l = 3..0
    for (int l = 3; l >= 0; --l) {
        const Layer& L = C(D3 + (3 - l));
        ConvExtra x;
        if (l > 0) {
            x.up = n->c[l - 1];
            x.up_ch = cat_ch(l - 1);
        }
        CUK(conv_launch(n, n->c[l], L.cin, Ws[l], Hs[l], L.wt, L.b, 9, L.cout, true, false, n->d[l], L.cout, 0, s, x));
    }
    const Layer& Hd = C(HEAD);
    CUK(conv_launch(n, n->d[0], Hd.cin, W, H, Hd.wt, Hd.b, 1, Hd.cout, false, true, n->y, Hd.cout, 0, s));
    return cudaGetLastError();
}

// backward pass from gyb (bf16, 16 channels); fills every layer's gw / gb
cudaError_t cnn_backward(mvs_cnn* n, int W, int H) {
    cudaStream_t s = n->stream;
    int Ws[5], Hs[5];
    for (int l = 0; l < 5; ++l) { Ws[l] = W >> l; Hs[l] = H >> l; }
    CUK(cudaMemsetAsync(n->grad, 0, n->n_theta * sizeof(float), s));
    auto v = [](const bf16* p) { return reinterpret_cast<const uint4*>(p); };
    auto vw = [](bf16* p) { return reinterpret_cast<uint4*>(p); };
    const long long np0 = (long long)W * H;
    Layer& Hd = n->L[HEAD];
    CUK(wgrad_launch(n->d[0], Hd.cin, n->gyb, Hd.cout, W, H, 1, Hd.gw, Hd.gb, s));
    CUK(conv_launch(n, n->gyb, Hd.cout, W, H, Hd.wtf, nullptr, 1, Hd.cin, false, false, n->gd[0], Hd.cin, 0, s));
    {
        const int nv = (int)(np0 * Hd.cin / 8);
        k_relu_mask<<<blocks(nv), 256, 0, s>>>(vw(n->gd[0]), v(n->d[0]), nv);
        count_launch();
    }
    // decoder levels 0..3: gd[l] is the gradient of d[l]
    for (int l = 0; l <= 3; ++l) {
        Layer& L = n->L[D3 + (3 - l)];
        CUK(wgrad_launch(n->c[l], L.cin, n->gd[l], L.cout, Ws[l], Hs[l], 9, L.gw, L.gb, s));
        CUK(conv_launch(n, n->gd[l], L.cout, Ws[l], Hs[l], L.wtf, nullptr, 9, L.cin, false, false, n->gc[l], L.cin, 0,
                        s));
        // gc[l] = [g up(prev) | g e[l] (skip)]: the first part goes on to the
        // level below, the second waits for the encoder
        const int up_v = (L.cin - n->L[E0 + l].cout) / 8;
        k_up_grad<<<blocks((long long)Ws[l + 1] * Hs[l + 1] * up_v), 256, 0, s>>>(
            v(n->gc[l]), L.cin / 8, v(l < 3 ? n->d[l + 1] : n->e[4]), Ws[l], Hs[l], up_v,
            vw(l < 3 ? n->gd[l + 1] : n->ge[4]));
        count_launch();
    }
    // encoder levels 4..0: ge[l] is the gradient of e[l]
    for (int l = 4; l >= 0; --l) {
        Layer& L = n->L[E0 + l];
        const bf16* in = l > 0 ? n->p[l - 1] : n->x;
        CUK(wgrad_launch(in, L.cin, n->ge[l], L.cout, Ws[l], Hs[l], 9, L.gw, L.gb, s));
        if (l > 0) {
            CUK(conv_launch(n, n->ge[l], L.cout, Ws[l], Hs[l], L.wtf, nullptr, 9, L.cin, false, false, n->gp[l - 1],
                            L.cin, 0, s));
            const int cat = n->L[D3 + (3 - (l - 1))].cin, cv = L.cin / 8;
            k_enc_grad<<<blocks((long long)Ws[l - 1] * Hs[l - 1] * cv), 256, 0, s>>>(
                v(n->gc[l - 1]), cat / 8, cat / 8 - cv, v(n->gp[l - 1]), v(n->e[l - 1]), Ws[l - 1], Hs[l - 1], cv,
                vw(n->ge[l - 1]));
            count_launch();
        }
    }
    return cudaGetLastError();
}

uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

mvs_status cnn_fail(mvs_cnn* n, mvs_status st, const char* msg, cudaError_t e = cudaSuccess) {
    if (n) n->err = std::string(msg) + (e != cudaSuccess ? std::string(": ") + cudaGetErrorString(e) : "");
    return st;
}

#define CNK(n, call)                                                                        \
    do {                                                                                    \
        cudaError_t _e = (call);                                                            \
        if (_e != cudaSuccess)                                                              \
            return cnn_fail((n), _e == cudaErrorMemoryAllocation ? MVS_ENOMEM : MVS_ECUDA, #call, _e); \
    } while (0)

bool shape_ok(const mvs_cnn* n, int W, int H) {
    return W >= 16 && H >= 16 && W % 16 == 0 && H % 16 == 0 && W <= n->maxW && H <= n->maxH;
}

}  // namespace

// network input from a PatchMatch state, forward pass, decode (the steps
// mvs_propose in mvs_api.cu runs on a context's view)
cudaError_t cnn_propose(mvs_cnn* n, const uint8_t* img, const float4* plane, const float* cost, int W, int H,
                        const double Kinv[9], float4* props, cudaStream_t s) {
    cudaStream_t keep = n->stream;
    n->stream = s;
    const long long np = (long long)W * H;
    k_make_input<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(img, plane, cost, np, n->hc, n->x);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cnn_forward(n, W, H);
    if (e == cudaSuccess) {
        Mat3 K;
        for (int i = 0; i < 9; ++i) K.m[i] = (float)Kinv[i];
        k_decode_proposals<<<(unsigned)((4 * np + 255) / 256), 256, 0, s>>>(reinterpret_cast<const float4*>(n->y), np, W,
                                                                           n->hc, K, props);
        count_launch();
        e = cudaGetLastError();
    }
    n->stream = keep;
    return e;
}

bool cnn_shape_ok(const mvs_cnn* n, int W, int H) { return shape_ok(n, W, H); }

extern "C" {

mvs_status mvs_cnn_create(int32_t max_width, int32_t max_height, float d_lo, float d_hi, uint64_t seed,
                          void* cuda_stream, mvs_cnn** out) {
    if (!out) return MVS_EINVAL;
    *out = nullptr;
    if (max_width < 16 || max_height < 16 || max_width % 16 || max_height % 16 || max_width > 8192 ||
        max_height > 8192 || !(d_lo > 0) || !(d_hi > d_lo))
        return MVS_EINVAL;
    mvs_cnn* n = new (std::nothrow) mvs_cnn();
    if (!n) return MVS_ENOMEM;
    n->maxW = max_width;
    n->maxH = max_height;
    n->stream = (cudaStream_t)cuda_stream;
    n->hc.rho_lo = 1.0f / d_hi;
    n->hc.rho_hi = 1.0f / d_lo;
    n->hc.lambda_n = 0.1f;
    const long long np = (long long)max_width * max_height;
    cudaError_t e = cudaSuccess;
    uint64_t rs = seed ^ 0x6A09E667F3BCC909ULL;
    for (int i = 0; i < NL; ++i) n->n_theta += (size_t)kLayerCout[i] * (i == HEAD ? 1 : 9) * kLayerCin[i] + kLayerCout[i];
    if (e == cudaSuccess) e = cnn_alloc(n, &n->theta, n->n_theta);
    if (e == cudaSuccess) e = cnn_alloc(n, &n->grad, n->n_theta);
    if (e == cudaSuccess) e = cnn_alloc(n, &n->mom, n->n_theta);
    if (e == cudaSuccess) e = cnn_alloc(n, &n->var, n->n_theta);
    if (e == cudaSuccess) e = cudaMemset(n->theta, 0, n->n_theta * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(n->mom, 0, n->n_theta * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(n->var, 0, n->n_theta * sizeof(float));
    size_t at = 0;
    for (int i = 0; i < NL && e == cudaSuccess; ++i) {
        Layer& L = n->L[i];
        L.cin = kLayerCin[i];
        L.cout = kLayerCout[i];
        L.taps = i == HEAD ? 1 : 9;
        L.relu = i != HEAD;
        L.nw = (size_t)L.cout * L.taps * L.cin;
        // layer i's part of the flat arrays (sizes are multiples of 16 floats)
        L.w = n->theta + at;
        L.gw = n->grad + at;
        L.b = L.w + L.nw;
        L.gb = L.gw + L.nw;
        at += L.nw + L.cout;
        e = cnn_alloc(n, &L.wt, L.nw);
        if (e == cudaSuccess) e = cnn_alloc(n, &L.wtf, L.nw);
        if (e != cudaSuccess) break;
        // He initialisation (Box-Muller on a splitmix64 stream); the first
        // layer's padding channels (6..15) and the head start small
        std::vector<float> hw(L.nw);
        const int fan_in = L.taps * (i == E0 ? 6 : L.cin);
        const float sd = (i == HEAD ? 0.1f : 1.0f) * sqrtf(2.0f / fan_in);
        for (size_t k = 0; k < L.nw; ++k) {
            double u1 = ((splitmix(rs) >> 11) + 1.0) * (1.0 / 9007199254740993.0);
            double u2 = (splitmix(rs) >> 11) * (1.0 / 9007199254740992.0);
            float v = (float)(sqrt(-2.0 * log(u1)) * cos(2.0 * 3.14159265358979323846 * u2)) * sd;
            if (i == E0 && (int)(k % L.cin) >= 6) v = 0.0f;
            hw[k] = v;
        }
        e = cudaMemcpy(L.w, hw.data(), L.nw * sizeof(float), cudaMemcpyHostToDevice);
    }
    // activations and gradients at the maximum size
    for (int l = 0; l < 5 && e == cudaSuccess; ++l) {
        long long npl = np >> (2 * l);
        e = cnn_alloc(n, &n->e[l], npl * kLayerCout[E0 + l]);
        if (e == cudaSuccess) e = cnn_alloc(n, &n->ge[l], npl * kLayerCout[E0 + l]);
        if (e == cudaSuccess && l < 4) e = cnn_alloc(n, &n->p[l], (npl / 4) * kLayerCout[E0 + l]);
        if (e == cudaSuccess && l < 4) e = cnn_alloc(n, &n->gp[l], (npl / 4) * kLayerCout[E0 + l]);
        if (e == cudaSuccess && l < 4) e = cnn_alloc(n, &n->c[l], npl * kLayerCin[D3 + (3 - l)]);
        if (e == cudaSuccess && l < 4) e = cnn_alloc(n, &n->gc[l], npl * kLayerCin[D3 + (3 - l)]);
        if (e == cudaSuccess && l < 4) e = cnn_alloc(n, &n->d[l], npl * kLayerCout[D3 + (3 - l)]);
        if (e == cudaSuccess && l < 4) e = cnn_alloc(n, &n->gd[l], npl * kLayerCout[D3 + (3 - l)]);
    }
    if (e == cudaSuccess) e = cnn_alloc(n, &n->x, np * 16);
    if (e == cudaSuccess) e = cnn_alloc(n, &n->y, np * 16);
    if (e == cudaSuccess) e = cnn_alloc(n, &n->gyb, np * 16);
    if (e == cudaSuccess) e = cnn_alloc(n, &n->loss, 1);
    if (e == cudaSuccess) e = cnn_alloc(n, &n->status, 1);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->status, 0, sizeof(int), n->stream);
    if (e == cudaSuccess) e = refresh_bf16(n);
    if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
    if (e != cudaSuccess) {
        g_cnn_err = e;
        mvs_cnn_destroy(n);
        return e == cudaErrorMemoryAllocation ? MVS_ENOMEM : MVS_ECUDA;
    }
    *out = n;
    return MVS_OK;
}

void mvs_cnn_destroy(mvs_cnn* n) {
    if (!n) return;
    cudaStreamSynchronize(n->stream);
    for (void* p : n->allocs) cudaFree(p);
    delete n;
}

const char* mvs_cnn_last_error(const mvs_cnn* n) {
    return n ? n->err.c_str() : (g_cnn_err != cudaSuccess ? cudaGetErrorString(g_cnn_err) : "");
}

mvs_status mvs_cnn_n_params(const mvs_cnn* n, int64_t* count) {
    if (!n || !count) return MVS_EINVAL;
    int64_t t = 0;
    for (int i = 0; i < NL; ++i) t += (int64_t)n->L[i].nw + n->L[i].cout;
    *count = t;
    return MVS_OK;
}

// MVS_ETIMEOUT once a convolution's bounded wait ran out since the last
// check (the status word is cleared); call after synchronising the stream
static mvs_status check_status(mvs_cnn* n) {
    int st = 0;
    CNK(n, cudaMemcpyAsync(&st, n->status, sizeof st, cudaMemcpyDeviceToHost, n->stream));
    CNK(n, cudaStreamSynchronize(n->stream));
    if (st == 0) return MVS_OK;
    CNK(n, cudaMemsetAsync(n->status, 0, sizeof(int), n->stream));
    return cnn_fail(n, MVS_ETIMEOUT, "a tensor-core convolution gave up waiting for its operands");
}

static mvs_status copy_params(mvs_cnn* n, float* host, bool grads, bool set) {
    float* dev = grads ? n->grad : n->theta;
    const size_t bytes = n->n_theta * sizeof(float);
    if (set) CNK(n, cudaMemcpyAsync(dev, host, bytes, cudaMemcpyHostToDevice, n->stream));
    else CNK(n, cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, n->stream));
    if (set) CNK(n, refresh_bf16(n));
    CNK(n, cudaStreamSynchronize(n->stream));
    return check_status(n);
}

mvs_status mvs_cnn_get_params(mvs_cnn* n, float* host_out) {
    if (!n || !host_out) return MVS_EINVAL;
    return copy_params(n, host_out, false, false);
}

mvs_status mvs_cnn_set_params(mvs_cnn* n, const float* host_in) {
    if (!n || !host_in) return MVS_EINVAL;
    return copy_params(n, const_cast<float*>(host_in), false, true);
}

mvs_status mvs_cnn_get_grads(mvs_cnn* n, float* host_out) {
    if (!n || !host_out) return MVS_EINVAL;
    return copy_params(n, host_out, true, false);
}

static mvs_status run_forward(mvs_cnn* n, const uint8_t* img, const float4* plane, const float* cost, int W, int H) {
    if (!shape_ok(n, W, H))
        return cnn_fail(n, MVS_EINVAL, "width and height must be multiples of 16 within the capacity");
    if (((uintptr_t)plane & 15u) || ((uintptr_t)cost & 3u))
        return cnn_fail(n, MVS_EINVAL, "plane must be 16-byte and cost 4-byte aligned");
    const long long np = (long long)W * H;
    k_make_input<<<(unsigned)((np + 255) / 256), 256, 0, n->stream>>>(img, plane, cost, np, n->hc, n->x);
    count_launch();
    CNK(n, cudaGetLastError());
    CNK(n, cnn_forward(n, W, H));
    n->lastW = W;
    n->lastH = H;
    return MVS_OK;
}

mvs_status mvs_cnn_forward(mvs_cnn* n, const uint8_t* img, const float* plane, const float* cost, int32_t W,
                           int32_t H, float* out) {
    if (!n || !img || !plane || !cost || !out) return MVS_EINVAL;
    mvs_status st = run_forward(n, img, (const float4*)plane, cost, W, H);
    if (st != MVS_OK) return st;
    CNK(n, cudaMemcpyAsync(out, n->y, (size_t)W * H * 16 * sizeof(float), cudaMemcpyDeviceToDevice, n->stream));
    return MVS_OK;
}

mvs_status mvs_cnn_backward(mvs_cnn* n, const uint8_t* img, const float* plane, const float* cost, int32_t W,
                            int32_t H, const float* target, const uint8_t* mask, float* loss_out) {
    if (!n || !img || !plane || !cost || !target || !mask) return MVS_EINVAL;
    if (W > kMaxTrainWidth) return cnn_fail(n, MVS_EINVAL, "training takes images up to 768 pixels wide");
    if ((uintptr_t)target & 15u) return cnn_fail(n, MVS_EINVAL, "target must be 16-byte aligned");
    mvs_status st = run_forward(n, img, (const float4*)plane, cost, W, H);
    if (st != MVS_OK) return st;
    const long long np = (long long)W * H;
    CNK(n, cudaMemsetAsync(n->loss, 0, sizeof(float), n->stream));
    k_proposal_loss<<<(unsigned)((np + 255) / 256), 256, 0, n->stream>>>(
        n->y, (const float4*)target, mask, np, n->hc, 1.0f / (float)np, reinterpret_cast<uint4*>(n->gyb), n->loss);
    count_launch();
    CNK(n, cudaGetLastError());
    CNK(n, cnn_backward(n, W, H));
    if (loss_out) {
        CNK(n, cudaMemcpyAsync(loss_out, n->loss, sizeof(float), cudaMemcpyDeviceToHost, n->stream));
        CNK(n, cudaStreamSynchronize(n->stream));
        return check_status(n);
    }
    return MVS_OK;
}

mvs_status mvs_cnn_propose(mvs_cnn* n, const uint8_t* img, const float* plane, const float* cost, int32_t W,
                           int32_t H, const double Kinv[9], float* proposals) {
    if (!n || !img || !plane || !cost || !Kinv || !proposals) return MVS_EINVAL;
    if (!shape_ok(n, W, H))
        return cnn_fail(n, MVS_EINVAL, "width and height must be multiples of 16 within the capacity");
    if (((uintptr_t)plane & 15u) || ((uintptr_t)cost & 3u) || ((uintptr_t)proposals & 15u))
        return cnn_fail(n, MVS_EINVAL, "plane and proposals must be 16-byte, cost 4-byte aligned");
    CNK(n, cnn_propose(n, img, (const float4*)plane, cost, W, H, Kinv, (float4*)proposals, n->stream));
    return MVS_OK;
}

mvs_status mvs_cnn_read(mvs_cnn* n, int32_t tensor, int32_t level, void* host_out, int64_t bytes) {
    if (!n || !host_out) return MVS_EINVAL;
    if (!n->lastW) return cnn_fail(n, MVS_EINVAL, "no forward pass yet");
    const void* src = nullptr;
    int ch = 0, lv = level;
    size_t elem = sizeof(bf16);
    auto in_range = [&](int hi) { return level >= 0 && level <= hi; };
    switch (tensor) {
        case MVS_CNN_T_INPUT: if (level == 0) { src = n->x; ch = 16; } break;
        case MVS_CNN_T_ENC: if (in_range(4)) { src = n->e[level]; ch = kLayerCout[E0 + level]; } break;
        case MVS_CNN_T_POOL: if (in_range(3)) { src = n->p[level]; ch = kLayerCout[E0 + level]; lv = level + 1; } break;
        case MVS_CNN_T_CAT: if (in_range(3)) { src = n->c[level]; ch = kLayerCin[D3 + (3 - level)]; } break;
        case MVS_CNN_T_DEC: if (in_range(3)) { src = n->d[level]; ch = kLayerCout[D3 + (3 - level)]; } break;
        case MVS_CNN_T_HEAD: if (level == 0) { src = n->y; ch = 16; elem = sizeof(float); } break;
        case MVS_CNN_T_GRAD_HEAD: if (level == 0) { src = n->gyb; ch = 16; } break;
        case MVS_CNN_T_GRAD_DEC: if (in_range(3)) { src = n->gd[level]; ch = kLayerCout[D3 + (3 - level)]; } break;
        case MVS_CNN_T_GRAD_CAT: if (in_range(3)) { src = n->gc[level]; ch = kLayerCin[D3 + (3 - level)]; } break;
        case MVS_CNN_T_GRAD_ENC: if (in_range(4)) { src = n->ge[level]; ch = kLayerCout[E0 + level]; } break;
        case MVS_CNN_T_GRAD_POOL:
            if (in_range(3)) { src = n->gp[level]; ch = kLayerCout[E0 + level]; lv = level + 1; }
            break;
        default: break;
    }
    if (!src) return cnn_fail(n, MVS_EINVAL, "no such tensor");
    const size_t need = (size_t)(n->lastW >> lv) * (size_t)(n->lastH >> lv) * ch * elem;
    if ((int64_t)need != bytes) return cnn_fail(n, MVS_EINVAL, "size mismatch");
    CNK(n, cudaMemcpyAsync(host_out, src, need, cudaMemcpyDeviceToHost, n->stream));
    CNK(n, cudaStreamSynchronize(n->stream));
    return check_status(n);
}

mvs_status mvs_cnn_test_timeout(mvs_cnn* n) {
    if (!n) return MVS_EINVAL;
    // one 16 x 16 convolution of the input buffer whose first wait targets a
    // barrier that nothing completes, with a wait limit of about 0.1 ms
    CNK(n, conv_tc_launch(n->x, 16, 16, 16, n->L[E0].wt, n->L[E0].b, 9, n->L[E0].cout, true, false, n->e[0],
                          n->L[E0].cout, 0, ConvExtra(), n->status, 1, 1500u, n->stream));
    CNK(n, cudaStreamSynchronize(n->stream));
    return check_status(n);
}

mvs_status mvs_cnn_adam_step(mvs_cnn* n, float lr) {
    if (!n || !(lr > 0)) return MVS_EINVAL;
    n->steps++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)n->steps), c2 = 1.0f - powf(b2, (float)n->steps);
    k_adam<<<blocks((long long)n->n_theta), 256, 0, n->stream>>>(n->theta, n->grad, n->mom, n->var,
                                                                (long long)n->n_theta, lr, b1, b2, 1e-8f, c1, c2);
    count_launch();
    CNK(n, cudaGetLastError());
    CNK(n, refresh_bf16(n));
    return MVS_OK;
}

}  // extern "C"
