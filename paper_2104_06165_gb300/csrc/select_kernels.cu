// Kernels on the sparse points of a structure-from-motion step: neighbouring-
// image selection (Sec. III-A) and the depth initialisation from sparse
// features (Sec. III-B, at the end of this file).
//
// Neighbouring-image selection (Sec. III-A, Eqs. 1-3).  For every ordered
// pair (reference i, source j) one block walks the sparse points: a point
// visible in both counts towards N_A, and Eq. 1 moves it along the ray from
// the reference centre, X^ = (1 + eps) X - eps C_i, so that Eq. 2 averages
// the displacement |x^'_j - x'_j| of its projection into j (FP64, block
// reduction in a fixed order).  Then one thread per reference image scores
// the sources with Eq. 3, zeta = (1 / N_A) min(b_ij, 0.1) min(theta_ij, 0.05)
// (baselines and principal-axis angles are FP64 per-pair constants from the
// host), removes those with tau < t_tau or no shared point and keeps the k
// smallest (tie: lower index).
#include <algorithm>
#include <cmath>

#include "mvs_internal.h"

namespace {

constexpr int kNbrBlock = 256;

__device__ __forceinline__ void proj(const NbrView& v, const double X[3], double& u, double& w) {
    double c[3], q[3];
    for (int a = 0; a < 3; ++a) c[a] = v.R[3 * a] * X[0] + v.R[3 * a + 1] * X[1] + v.R[3 * a + 2] * X[2] + v.t[a];
    for (int a = 0; a < 3; ++a) q[a] = v.K[3 * a] * c[0] + v.K[3 * a + 1] * c[1] + v.K[3 * a + 2] * c[2];
    u = q[0] / q[2];
    w = q[1] / q[2];
}

__global__ void __launch_bounds__(kNbrBlock) k_nbr_pairs(const NbrView* __restrict__ views, int n,
                                                        const double* __restrict__ X,
                                                        const unsigned long long* __restrict__ vis, long long n_pts,
                                                        double eps, double* __restrict__ tau, int* __restrict__ na) {
    const int i = blockIdx.x / n, j = blockIdx.x % n;
    __shared__ double s_sum[kNbrBlock / 32];
    __shared__ long long s_cnt[kNbrBlock / 32];
    double sum = 0.0;
    long long cnt = 0;
    if (i != j) {
        const NbrView& vi = views[i];
        const NbrView& vj = views[j];
        const double Ci[3] = {vi.C[0], vi.C[1], vi.C[2]};
        const unsigned long long both = (1ULL << i) | (1ULL << j);
        for (long long p = threadIdx.x; p < n_pts; p += blockDim.x) {
            if ((vis[p] & both) != both) continue;
            const double Xp[3] = {X[3 * p], X[3 * p + 1], X[3 * p + 2]};
            double Xh[3];
            for (int a = 0; a < 3; ++a) Xh[a] = (1.0 + eps) * Xp[a] - eps * Ci[a];
            double u, w, uh, wh;
            proj(vj, Xp, u, w);
            proj(vj, Xh, uh, wh);
            const double du = uh - u, dv = wh - w;
            sum += sqrt(du * du + dv * dv);
            cnt++;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_down_sync(0xffffffffu, sum, o);
        cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s_sum[threadIdx.x >> 5] = sum;
        s_cnt[threadIdx.x >> 5] = cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        long long c = 0;
        for (int w = 0; w < kNbrBlock / 32; ++w) {
            s += s_sum[w];
            c += s_cnt[w];
        }
        na[blockIdx.x] = (int)c;
        tau[blockIdx.x] = c ? s / (double)c : 0.0;
    }
}

// one thread per reference image: Eq. 3 scores and the k smallest
__global__ void k_nbr_select(int n, int k, const double* __restrict__ base, const double* __restrict__ angle,
                             const int* __restrict__ na, const double* __restrict__ tau, double t_tau,
                             double* __restrict__ zeta, int* __restrict__ nbr) {
    const int i = threadIdx.x;
    if (i >= n) return;
    int cand[MVS_MAX_VIEWS_SELECT];
    double zc[MVS_MAX_VIEWS_SELECT];
    int nc = 0;
    for (int j = 0; j < n; ++j) {
        const long long e = (long long)i * n + j;
        double z = INFINITY;
        if (j != i && na[e] > 0 && tau[e] >= t_tau) {
            z = (1.0 / (double)na[e]) * fmin(base[e], 0.1) * fmin(angle[e], 0.05);
            // insertion by (zeta, index)
            int b = nc - 1;
            while (b >= 0 && zc[b] > z) {
                cand[b + 1] = cand[b];
                zc[b + 1] = zc[b];
                b--;
            }
            cand[b + 1] = j;
            zc[b + 1] = z;
            nc++;
        }
        if (zeta) zeta[e] = z;
    }
    for (int r = 0; r < k; ++r) nbr[(long long)i * k + r] = r < nc ? cand[r] : -1;
}

}  // namespace

cudaError_t launch_select_neighbors(const NbrView* dev_views, int n, const double* X, const unsigned long long* vis,
                                    long long n_pts, double eps, double t_tau, int k, const double* base,
                                    const double* angle, double* tau, int* na, double* zeta, int* nbr,
                                    cudaStream_t s) {
    k_nbr_pairs<<<n * n, kNbrBlock, 0, s>>>(dev_views, n, X, vis, n_pts, eps, tau, na);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_nbr_select<<<1, 64, 0, s>>>(n, k, base, angle, na, tau, t_tau, zeta, nbr);
    count_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Depth initialisation from sparse features (Sec. III-B).  Features of the
// reference view: the sparse points visible in it whose re-projection error
// is below max_reproj and that are visible in at least floor(v - 1) images
// (v = mean images per point); each keeps its observation in the reference
// and its z-depth there (FP64, rounded to float).  Per pixel, the closest
// feature in each of four quadrants within W / 10 px gives [d_min, d_max],
// clamped to the depth range; the closest-feature choice is taken in single
// precision, each operation rounded on its own, the first feature winning a
// tie.
//
// With many tiles and points the features are binned into cells and a warp
// looks at the cells in rings around its pixels until no farther feature can
// matter, so that what is left is about the features nearby (3072 x 2048, 20 k
// points: 0.39 ms for the whole call; 3.8 ms with every tile scanning every
// point, which is the faster way for the small calls, see all_features).
// ---------------------------------------------------------------------------
namespace {

// pixels of a block: 16 x 16, a warp covers 16 x 2 (inside one cell)
constexpr int kRangeTile = 16;

__global__ void k_sparse_count(const unsigned long long* __restrict__ vis, long long n_pts,
                               unsigned long long views_mask, unsigned long long* __restrict__ total) {
    unsigned long long s = 0;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n_pts; p += (long long)gridDim.x * blockDim.x)
        s += __popcll(vis[p] & views_mask);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(total, s);
}

__global__ void k_sparse_features(const double* __restrict__ X, const unsigned long long* __restrict__ vis,
                                  const double* __restrict__ reproj, const double* __restrict__ obs, long long n_pts,
                                  unsigned long long views_mask, const unsigned long long* __restrict__ total,
                                  int ref, double R6, double R7, double R8, double t2, double max_reproj,
                                  int cell, int ncx, int ncy, float4* __restrict__ feat, int* __restrict__ cell_of,
                                  unsigned* __restrict__ cell_n) {
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= n_pts) return;
    const double vbar = (double)*total / (double)n_pts;
    const int min_views = (int)floor(__dsub_rn(vbar, 1.0));
    const unsigned long long m = vis[p];
    const bool keep = ((m >> ref) & 1ULL) && reproj[p] < max_reproj && __popcll(m & views_mask) >= min_views;
    double z = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(R6, X[3 * p]), __dmul_rn(R7, X[3 * p + 1])),
                                   __dmul_rn(R8, X[3 * p + 2])),
                         t2);
    const float u = (float)obs[2 * p], v = (float)obs[2 * p + 1], zf = (float)z;
    // a feature without a depth is none
    const bool feature = keep && isfinite(u) && isfinite(v) && zf == zf;
    feat[p] = make_float4(u, v, feature ? zf : __int_as_float(0x7fc00000), __uint_as_float((uint32_t)p));
    if (!cell_of) return;
    int c = -1;
    if (feature) {
        // features outside the image go to the cells at its edge
        const int cx = (int)fminf(fmaxf(u, 0.0f), (float)(ncx * cell - 1)) / cell;
        const int cy = (int)fminf(fmaxf(v, 0.0f), (float)(ncy * cell - 1)) / cell;
        c = cy * ncx + cx;
        atomicAdd(cell_n + c, 1u);
    }
    cell_of[p] = c;
}

// exclusive scan of the cell counts (one block), counts cleared for the filling
__global__ void __launch_bounds__(1024) k_sparse_scan(unsigned* __restrict__ cell_n, unsigned* __restrict__ cell_start,
                                                      int n) {
    __shared__ unsigned part[1024];
    const int per = (n + 1023) / 1024, lo = min(n, (int)threadIdx.x * per), hi = min(n, lo + per);
    unsigned s = 0;
    for (int k = lo; k < hi; ++k) s += cell_n[k];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const unsigned v = threadIdx.x >= o ? part[threadIdx.x - o] : 0u;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    unsigned base = threadIdx.x ? part[threadIdx.x - 1] : 0u;
    for (int k = lo; k < hi; ++k) {
        cell_start[k] = base;
        base += cell_n[k];
        cell_n[k] = 0;
    }
    if (threadIdx.x == 1023) cell_start[n] = part[1023];
}

// (the order within a cell does not matter: ties go by the point's index)
__global__ void k_sparse_fill(const float4* __restrict__ feat, const int* __restrict__ cell_of, long long n_pts,
                              const unsigned* __restrict__ cell_start, unsigned* __restrict__ cell_n,
                              float4* __restrict__ binned) {
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= n_pts) return;
    const int c = cell_of[p];
    if (c >= 0) binned[cell_start[c] + atomicAdd(cell_n + c, 1u)] = feat[p];
}

__device__ __forceinline__ float2 span(const float best[4], const float bd[4], float d_lo, float d_hi) {
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (best[q] < INFINITY) {
            lo = bd[q] < lo ? bd[q] : lo;
            hi = bd[q] > hi ? bd[q] : hi;
        }
    const float nan = __int_as_float(0x7fc00000);
    return lo <= hi ? make_float2(fminf(fmaxf(lo, d_lo), d_hi), fminf(fmaxf(hi, d_lo), d_hi)) : make_float2(nan, nan);
}

__global__ void __launch_bounds__(kRangeTile * kRangeTile) k_sparse_range(
    const float4* __restrict__ binned, const unsigned* __restrict__ cell_start, int cell, int ncx, int ncy, int W, int H,
    float d_lo, float d_hi, float2* __restrict__ range) {
    const int x = blockIdx.x * kRangeTile + (threadIdx.x % kRangeTile);
    const int y = blockIdx.y * kRangeTile + (threadIdx.x / kRangeTile);
    const float r = __fdiv_rn((float)W, 10.0f), r2 = __fmul_rn(r, r);
    const int cx = blockIdx.x * kRangeTile / cell, cy = blockIdx.y * kRangeTile / cell;
    // quadrants: 0 right / lower, 1 left / lower, 2 left / upper, 3 right / upper
    float best[4] = {INFINITY, INFINITY, INFINITY, INFINITY}, bd[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t bi[4] = {0u, 0u, 0u, 0u};
    const float fx = (float)x, fy = (float)y;
    auto scan = [&](unsigned lo, unsigned hi) {        // features [lo, hi) of the binned list, the same for the whole warp
#pragma unroll 4
        for (unsigned k = lo; k < hi; ++k) {
            const float4 f = __ldg(binned + k);
            const float dx = __fsub_rn(f.x, fx), dy = __fsub_rn(f.y, fy);
            const float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
            const bool right = dx >= 0.0f, lower = dy >= 0.0f;
            const float cur = right ? (lower ? best[0] : best[3]) : (lower ? best[1] : best[2]);
            if (d2 < r2 && d2 <= cur) {
                const uint32_t id = __float_as_uint(f.w);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (right == (q == 0 || q == 3) && lower == (q < 2) && (d2 < best[q] || id < bi[q])) {
                        best[q] = d2;
                        bd[q] = f.z;
                        bi[q] = id;
                    }
            }
        }
    };
    for (int k = 0;; ++k) {
        // ring k: its upper and lower row of cells are contiguous in the list,
        // the cells between them at its two sides are not
        const int xa = max(cx - k, 0), xb = min(cx + k, ncx - 1);
        if (cy - k >= 0) scan(__ldg(cell_start + (cy - k) * ncx + xa), __ldg(cell_start + (cy - k) * ncx + xb + 1));
        if (k > 0) {
            if (cy + k < ncy) scan(__ldg(cell_start + (cy + k) * ncx + xa), __ldg(cell_start + (cy + k) * ncx + xb + 1));
            for (int yy = max(cy - k + 1, 0); yy <= min(cy + k - 1, ncy - 1); ++yy) {
                const unsigned* row = cell_start + yy * ncx;
                if (cx - k >= 0) scan(__ldg(row + cx - k), __ldg(row + cx - k + 1));
                if (cx + k < ncx) scan(__ldg(row + cx + k), __ldg(row + cx + k + 1));
            }
        }
        // distance of the features not seen yet: beyond the square of cells
        // looked at (to infinity where it has reached the edge of the grid);
        // 0.01 px covers the rounding of the compared distances
        const float el = cx - k > 0 ? fx - (float)((cx - k) * cell) : INFINITY;
        const float er = cx + k < ncx - 1 ? (float)((cx + k + 1) * cell) - fx : INFINITY;
        const float eu = cy - k > 0 ? fy - (float)((cy - k) * cell) : INFINITY;
        const float ed = cy + k < ncy - 1 ? (float)((cy + k + 1) * cell) - fy : INFINITY;
        bool done = true;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float side = fminf(q == 0 || q == 3 ? er : el, q < 2 ? ed : eu) - 0.01f;
            done = done && (side > r + 0.01f || (side > 0.0f && best[q] < side * side));
        }
        if (__all_sync(0xffffffffu, done || x >= W || y >= H)) break;
    }
    if (x < W && y < H) range[(long long)y * W + x] = span(best, bd, d_lo, d_hi);
}

// Every feature against every tile: 1024 features per step are compacted to
// those within the radius of the tile, in the order of the points, so a
// strict comparison keeps the first of a tie.
__global__ void __launch_bounds__(kRangeTile * kRangeTile) k_sparse_range_all(
    const float4* __restrict__ feat, long long n_pts, int W, int H, float d_lo, float d_hi, float2* __restrict__ range) {
    constexpr int NT = kRangeTile * kRangeTile, NW = NT / 32, U = 4;
    __shared__ float2 s_uv[U * NT];
    __shared__ float s_d[U * NT];
    __shared__ int s_wc[U * NW];
    const int x = blockIdx.x * kRangeTile + (threadIdx.x % kRangeTile);
    const int y = blockIdx.y * kRangeTile + (threadIdx.x / kRangeTile);
    const float r = __fdiv_rn((float)W, 10.0f), r2 = __fmul_rn(r, r);
    const float bx0 = (float)(blockIdx.x * kRangeTile) - r, bx1 = (float)(blockIdx.x * kRangeTile + kRangeTile - 1) + r;
    const float by0 = (float)(blockIdx.y * kRangeTile) - r, by1 = (float)(blockIdx.y * kRangeTile + kRangeTile - 1) + r;
    float best[4] = {INFINITY, INFINITY, INFINITY, INFINITY}, bd[4] = {0.f, 0.f, 0.f, 0.f};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long base = 0; base < n_pts; base += U * NT) {
        float4 f[U];
        unsigned m[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const long long p = base + i * NT + threadIdx.x;
            f[i] = p < n_pts ? __ldg(feat + p) : make_float4(0.f, 0.f, __int_as_float(0x7fc00000), 0.f);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            m[i] = __ballot_sync(0xffffffffu, f[i].z == f[i].z && f[i].x >= bx0 && f[i].x <= bx1 && f[i].y >= by0 &&
                                                  f[i].y <= by1);
            if (lane == 0) s_wc[i * NW + warp] = __popc(m[i]);
        }
        __syncthreads();
        static_assert(U * NW == 32, "one count per lane");
        int incl = s_wc[lane];
        const int own = incl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int cnt = __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int off = __shfl_sync(0xffffffffu, incl - own, i * NW + warp) + __popc(m[i] & ((1u << lane) - 1u));
            if ((m[i] >> lane) & 1u) {
                s_uv[off] = make_float2(f[i].x, f[i].y);
                s_d[off] = f[i].z;
            }
        }
        __syncthreads();
        for (int k = 0; k < cnt; ++k) {
            const float dx = __fsub_rn(s_uv[k].x, (float)x), dy = __fsub_rn(s_uv[k].y, (float)y);
            const float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
            if (!(d2 < r2)) continue;
            const int q = dx >= 0.0f ? (dy >= 0.0f ? 0 : 3) : (dy >= 0.0f ? 1 : 2);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j == q && d2 < best[j]) {
                    best[j] = d2;
                    bd[j] = s_d[k];
                }
        }
        if (base + U * NT < n_pts) __syncthreads();
    }
    if (x < W && y < H) range[(long long)y * W + x] = span(best, bd, d_lo, d_hi);
}

// Side of the cells: about 3 points to a cell, so that the rings end after one
// or two steps at any density (a fixed side of 32 pixels has up to ten rings of
// empty cells where the points are few); a multiple of the tile, no more than
// the radius needs.
int cell_side(int W, int H, long long n_pts) {
    const double side = std::sqrt(3.25 * (double)W * H / (double)std::max(1LL, n_pts));
    const int most = (W / 10 + kRangeTile) / kRangeTile;
    return kRangeTile * std::max(1, std::min(most, (int)(side / kRangeTile + 0.5)));
}

// Where every tile looks at every feature.  Binning costs three launches and
// the rings a chain of dependent reads, about 20 us more than the scan at the
// smallest sizes; the scan grows with tiles x points.  Scan against cells,
// microseconds of a call: 320 x 240 18 / 39 with 1 k points and 104 / 177 with
// 20 k (one wave of tiles: the scan's latency, and cells of 16 pixels hold too
// many points there), 640 x 480 43 / 54 with 2.5 k and 81 / 72 with 6 k,
// 960 x 640 36 / 53 and 70 / 66 with 1 k and 2.5 k, 3072 x 2048 221 / 247 with
// 1 k, 526 / 273 with 2.5 k and 3807 / 392 with 20 k.
bool all_features(int W, int H, long long n_pts) {
    const long long tiles = (long long)((W + kRangeTile - 1) / kRangeTile) * ((H + kRangeTile - 1) / kRangeTile);
    return tiles <= 4 * 152 || n_pts <= 1000 || tiles * n_pts <= 5000000;
}

}  // namespace

size_t sparse_range_cells(int W, int H, long long n_pts) {
    if (all_features(W, H, n_pts)) return 0;
    const int cell = cell_side(W, H, n_pts);
    return (size_t)((W + cell - 1) / cell) * ((H + cell - 1) / cell);
}

cudaError_t launch_sparse_range(int ref, int n_views, const double Rrow2[3], double t2, const double* X,
                                const unsigned long long* vis, const double* reproj, const double* obs,
                                long long n_pts, double max_reproj, int W, int H, float d_lo, float d_hi,
                                unsigned long long* total, float4* feat, float4* binned, int* cell_of, unsigned* cells,
                                float2* range, cudaStream_t s) {
    const bool all = all_features(W, H, n_pts);
    const int cell = cell_side(W, H, n_pts), ncx = (W + cell - 1) / cell, ncy = (H + cell - 1) / cell, nc = ncx * ncy;
    unsigned *cell_n = cells, *cell_start = cells + nc;
    cudaError_t e = cudaMemsetAsync(total, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    if (!all && (e = cudaMemsetAsync(cell_n, 0, (size_t)nc * sizeof(unsigned), s)) != cudaSuccess) return e;
    const unsigned long long views_mask = n_views >= 64 ? ~0ULL : ((1ULL << n_views) - 1ULL);
    if (n_pts > 0) {
        const unsigned np = (unsigned)((n_pts + 255) / 256), nb = std::min(np, 152u * 8u);
        k_sparse_count<<<nb, 256, 0, s>>>(vis, n_pts, views_mask, total);
        k_sparse_features<<<np, 256, 0, s>>>(X, vis, reproj, obs, n_pts, views_mask, total, ref, Rrow2[0], Rrow2[1],
                                             Rrow2[2], t2, max_reproj, cell, ncx, ncy, feat, all ? nullptr : cell_of,
                                             cell_n);
        count_launch(2);
        if (!all) {
            k_sparse_scan<<<1, 1024, 0, s>>>(cell_n, cell_start, nc);
            k_sparse_fill<<<np, 256, 0, s>>>(feat, cell_of, n_pts, cell_start, cell_n, binned);
            count_launch(2);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    dim3 grid((W + kRangeTile - 1) / kRangeTile, (H + kRangeTile - 1) / kRangeTile);
    if (all)
        k_sparse_range_all<<<grid, kRangeTile * kRangeTile, 0, s>>>(feat, n_pts, W, H, d_lo, d_hi, range);
    else
        k_sparse_range<<<grid, kRangeTile * kRangeTile, 0, s>>>(binned, cell_start, cell, ncx, ncy, W, H, d_lo, d_hi,
                                                                range);
    count_launch();
    return cudaGetLastError();
}
