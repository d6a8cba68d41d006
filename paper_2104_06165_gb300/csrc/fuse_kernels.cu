// Depth-map fusion (Sec. III-F): the depth maps of several views are merged
// into one point cloud.  Views are taken in the given order; every pixel of
// view a that is still present (depth > 0, kept, not merged before) is
// back-projected to X, projected into each later view b, and when the pixel
// it lands on is present and its back-projection X' differs from X by less
// than tol times the depth of X, that pixel is merged into X's point and
// removed from view b.
//
// The sequential statement is order dependent only through which pixel of
// view a takes a pixel of view b first (the lowest in raster order), so view
// a is processed in parallel in two passes: every pixel claims its
// consistent targets with an atomicMin of its index, then every pixel
// averages the targets it won and removes them.  Every claimed target is
// removed, so the claim arrays are reset once for the whole fusion.  The points of view a are
// written in raster order after those of the earlier views (a block count,
// a one-block scan, a block-local rank).
//
// The decisions are integers and the paper fixes no precision, so they are
// taken in single precision with every operation rounded on its own
// (__fmul_rn / __fadd_rn / __fsub_rn / __fdiv_rn, no contraction):
//   back-projection of pixel (x, y) with depth d (pinhole K, x_cam = R X + t):
//     yc = (y - cy) / fy, xc = ((x - cx) - s yc) / fx,
//     X = R^T ((d xc, d yc, d) - t), component k = ((R0k e0 + R1k e1) + R2k e2)
//   projection: c = R X + t, component k = ((Rk0 X0 + Rk1 X1) + Rk2 X2) + tk,
//     u = ((fx c0 + s c1) + cx c2) / c2, v = (fy c1 + cy c2) / c2,
//     pixel (floor(u + 1/2), floor(v + 1/2)) when c2 > 0 and inside the image
//   agreement: ((e0 e0 + e1 e1) + e2 e2) < (tol d)^2 with e = X - X'
//   point: (X + X'_b1 + X'_b2 + ...) / count, summed in view order.
//
// What bounds it: the latency of the gathers from the later views (the claim
// pass of a 2048 x 1365 view issues in 54 % of its slots at 4 % of the DRAM's
// rate; its warps wait for gathers and, at the count's barrier, for the slowest
// warp of the block) and the launches of the small views.  A view's depth and whether a pixel is still present share one
// compact float array (zero = absent), so that a gather touches 4 bytes of a
// 32-byte sector that the neighbours use too instead of a flag and 4 of a
// plane's 16 bytes.  One launch prepares all views; the claim pass notes which
// views a pixel claimed from, so that the merge projects into those only; its
// blocks also count their pixels and the last of them to finish scans the
// counts, so a view takes two launches instead of four (8 views, 13.5 M
// pixels: 796 us against 1005).
#include <algorithm>

#include "mvs_internal.h"

namespace {

constexpr int kFuseBlock = 256;
// views whose reads a claiming thread keeps in flight (8 views, 13.5 M pixels:
// one 839 us, two 798, four 796, eight 904)
constexpr int kFuseBatch = 4;

__device__ __forceinline__ void fuse_backproject(const FuseView& c, int x, int y, float d, float X[3]) {
    const float yc = __fdiv_rn(__fsub_rn((float)y, c.cy), c.fy);
    const float xc = __fdiv_rn(__fsub_rn(__fsub_rn((float)x, c.cx), __fmul_rn(c.sk, yc)), c.fx);
    const float e0 = __fsub_rn(__fmul_rn(d, xc), c.t[0]);
    const float e1 = __fsub_rn(__fmul_rn(d, yc), c.t[1]);
    const float e2 = __fsub_rn(d, c.t[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        X[k] = __fadd_rn(__fadd_rn(__fmul_rn(c.R[k], e0), __fmul_rn(c.R[3 + k], e1)), __fmul_rn(c.R[6 + k], e2));
}

// pixel (x, y) of the projection of X into view c; false outside the image
__device__ __forceinline__ bool fuse_project(const FuseView& c, const float X[3], int& x, int& y) {
    float q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        q[k] = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(c.R[3 * k], X[0]), __fmul_rn(c.R[3 * k + 1], X[1])),
                                   __fmul_rn(c.R[3 * k + 2], X[2])),
                         c.t[k]);
    if (!(q[2] > 0.0f)) return false;
    const float u = __fdiv_rn(__fadd_rn(__fadd_rn(__fmul_rn(c.fx, q[0]), __fmul_rn(c.sk, q[1])), __fmul_rn(c.cx, q[2])),
                              q[2]);
    const float v = __fdiv_rn(__fadd_rn(__fmul_rn(c.fy, q[1]), __fmul_rn(c.cy, q[2])), q[2]);
    const float fu = floorf(__fadd_rn(u, 0.5f)), fv = floorf(__fadd_rn(v, 0.5f));
    if (!(fu >= 0.0f && fu <= (float)(c.W - 1) && fv >= 0.0f && fv <= (float)(c.H - 1))) return false;
    x = (int)fu;
    y = (int)fv;
    return true;
}

__device__ __forceinline__ bool fuse_agree(const float X[3], const float Y[3], float thr) {
    const float e0 = __fsub_rn(X[0], Y[0]), e1 = __fsub_rn(X[1], Y[1]), e2 = __fsub_rn(X[2], Y[2]);
    const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(e0, e0), __fmul_rn(e1, e1)), __fmul_rn(e2, e2));
    return d2 < __fmul_rn(thr, thr);
}

// every view (blockIdx.y): present pixels (depth > 0 and kept) keep their
// depth, nothing claimed (0x7f7f7f7f, above every pixel index), owner -1
__global__ void __launch_bounds__(kFuseBlock) k_fuse_init(const FuseView* __restrict__ views) {
    const FuseView& v = views[blockIdx.y];
    const int n = v.W * v.H;   // at most 2^30
    for (int i = blockIdx.x * kFuseBlock + threadIdx.x; i < n; i += gridDim.x * kFuseBlock) {
        const float d = v.plane[i].w;
        v.depth[i] = d > 0.0f && (!v.keep || v.keep[i]) ? d : 0.0f;
        v.claim[i] = 0x7f7f7f7f;
        if (v.owner) v.owner[i] = -1;
    }
}

// exclusive scan of the block counts by one block (any number of counts),
// offset by the points already written; the running total is updated
__device__ __forceinline__ void fuse_scan(const int* block_count, long long* __restrict__ block_off, int nblk,
                                          long long* __restrict__ total) {
    __shared__ long long part[kFuseBlock];
    const int per = (nblk + kFuseBlock - 1) / kFuseBlock;
    const int lo = min(nblk, (int)threadIdx.x * per), hi = min(nblk, lo + per);
    long long s = 0;
    for (int k = lo; k < hi; ++k) s += __ldcg(block_count + k);
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < kFuseBlock; o <<= 1) {   // inclusive Hillis-Steele scan
        long long v = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    long long base = *total + (threadIdx.x ? part[threadIdx.x - 1] : 0);
    for (int k = lo; k < hi; ++k) {
        block_off[k] = base;
        base += __ldcg(block_count + k);
    }
    __syncthreads();
    if (threadIdx.x == 0) *total += part[kFuseBlock - 1];
}

// pass 1: every present pixel of view a claims the pixels of later views it
// agrees with (the lowest index wins, as in the raster-order statement) and
// notes the views in `hits`; each block counts its present pixels and the last
// block to finish scans the counts
__global__ void __launch_bounds__(kFuseBlock) k_fuse_claim(const FuseView* __restrict__ views, int n, int a, float tol,
                                                           int* block_count, long long* __restrict__ block_off,
                                                           long long* __restrict__ total, unsigned* finished) {
    const FuseView& va = views[a];
    const int i = blockIdx.x * kFuseBlock + threadIdx.x;
    const float d = i < va.W * va.H ? va.depth[i] : 0.0f;
    if (d > 0.0f) {
        const int y = i / va.W, x = i - y * va.W;
        float X[3];
        fuse_backproject(va, x, y, d, X);
        const float thr = __fmul_rn(tol, d);
        uint32_t hits = 0;
        for (int b0 = a + 1; b0 < n; b0 += kFuseBatch) {
            int tx[kFuseBatch], ty[kFuseBatch];
            float e[kFuseBatch];
#pragma unroll
            for (int k = 0; k < kFuseBatch; ++k) {
                e[k] = 0.0f;
                if (b0 + k < n && fuse_project(views[b0 + k], X, tx[k], ty[k]))
                    e[k] = views[b0 + k].depth[ty[k] * views[b0 + k].W + tx[k]];
            }
#pragma unroll
            for (int k = 0; k < kFuseBatch; ++k) {
                if (!(e[k] > 0.0f)) continue;
                const FuseView& vb = views[b0 + k];
                float Y[3];
                fuse_backproject(vb, tx[k], ty[k], e[k], Y);
                if (fuse_agree(X, Y, thr)) {
                    atomicMin(vb.claim + ty[k] * vb.W + tx[k], i);
                    hits |= 1u << min(b0 + k - a - 1, 31);
                }
            }
        }
        va.hits[i] = hits;
    }
    const int c = __syncthreads_count(d > 0.0f);
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __stcg(block_count + blockIdx.x, c);
        __threadfence();
        last = atomicAdd(finished, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    fuse_scan(block_count, block_off, (int)gridDim.x, total);
    if (threadIdx.x == 0) *finished = 0;   // for the next view
}

// pass 2: every present pixel of view a averages the pixels it won, removes
// them from their views and writes its point at its raster rank
__global__ void __launch_bounds__(kFuseBlock) k_fuse_merge(const FuseView* __restrict__ views, int n, int a,
                                                           const long long* __restrict__ block_off,
                                                           float4* __restrict__ points, int2* __restrict__ src,
                                                           long long cap) {
    __shared__ int warp_count[kFuseBlock / 32];
    const FuseView& va = views[a];
    const int i = blockIdx.x * kFuseBlock + threadIdx.x;
    const float d = i < va.W * va.H ? va.depth[i] : 0.0f;
    const bool p = d > 0.0f;
    // rank of this pixel among the present pixels of the block
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned m = __ballot_sync(0xffffffffu, p);
    if (lane == 0) warp_count[warp] = __popc(m);
    __syncthreads();
    int rank = __popc(m & ((1u << lane) - 1u));
    for (int w = 0; w < warp; ++w) rank += warp_count[w];
    if (!p) return;
    const int y = i / va.W, x = i - y * va.W;
    float X[3], sum[3];
    fuse_backproject(va, x, y, d, X);
    sum[0] = X[0]; sum[1] = X[1]; sum[2] = X[2];
    int cnt = 1;
    // only the views this pixel claimed from (bit 31: any of the 32nd and later)
    const uint32_t hits = va.hits[i];
    for (int b = a + 1; b < n; ++b) {
        const int hb = b - a - 1;
        if (hb < 31 && !((hits >> hb) & 1u)) continue;
        if (hb == 31 && !(hits >> 31)) break;
        const FuseView& vb = views[b];
        int tx, ty;
        if (!fuse_project(vb, X, tx, ty)) continue;
        const int t = ty * vb.W + tx;
        // a claim won in this view's pass implies a present, agreeing pixel;
        // claims left from earlier views sit on pixels already removed
        if (vb.claim[t] != i) continue;
        const float e = vb.depth[t];
        if (!(e > 0.0f)) continue;
        float Y[3];
        fuse_backproject(vb, tx, ty, e, Y);
        sum[0] = __fadd_rn(sum[0], Y[0]);
        sum[1] = __fadd_rn(sum[1], Y[1]);
        sum[2] = __fadd_rn(sum[2], Y[2]);
        cnt++;
        vb.depth[t] = 0.0f;
        if (vb.owner) vb.owner[t] = block_off[blockIdx.x] + rank;
    }
    const long long k = block_off[blockIdx.x] + rank;
    if (va.owner) va.owner[i] = k;
    if (k < cap) {
        const float fc = (float)cnt;
        points[k] = make_float4(__fdiv_rn(sum[0], fc), __fdiv_rn(sum[1], fc), __fdiv_rn(sum[2], fc), fc);
        if (src) src[k] = make_int2(va.index, i);
    }
}

unsigned blocks_of(long long n, int block) { return (unsigned)((n + block - 1) / block); }

}  // namespace

cudaError_t launch_fuse(const FuseView* host_views, FuseView* dev_views, int n, float tol, int* block_count,
                        long long* block_off, long long* total, float4* points, int2* src, long long cap,
                        cudaStream_t s) {
    cudaError_t e = cudaMemcpyAsync(dev_views, host_views, sizeof(FuseView) * n, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    // the running total and, behind it, the counter of finished blocks
    if ((e = cudaMemsetAsync(total, 0, 2 * sizeof(long long), s)) != cudaSuccess) return e;
    unsigned* finished = reinterpret_cast<unsigned*>(total + 1);
    long long most = 1;
    for (int a = 0; a < n; ++a) most = std::max(most, (long long)host_views[a].W * host_views[a].H);
    for (int a0 = 0; a0 < n; a0 += 32768) {
        const dim3 grid((unsigned)std::min<long long>(blocks_of(most, kFuseBlock), 152LL * 8),
                        (unsigned)std::min(n - a0, 32768));
        k_fuse_init<<<grid, kFuseBlock, 0, s>>>(dev_views + a0);
        count_launch();
    }
    for (int a = 0; a < n; ++a) {
        const unsigned nb = blocks_of((long long)host_views[a].W * host_views[a].H, kFuseBlock);
        k_fuse_claim<<<nb, kFuseBlock, 0, s>>>(dev_views, n, a, tol, block_count, block_off, total, finished);
        k_fuse_merge<<<nb, kFuseBlock, 0, s>>>(dev_views, n, a, block_off, points, src, cap);
        count_launch(2);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaGetLastError();
}
