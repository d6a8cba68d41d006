// Geometric-consistency filter (Sec. III-D) and plane hypothesis inference
// (Sec. III-E): four-direction line-fit hypotheses, their matching cost, the
// pairwise MRF of Eq. 6-9 decoded by tree-reweighted message passing at half
// resolution, closest-hypothesis selection and Eq. 10 normals.
#include <algorithm>
#include <mutex>

#include "../../include/mvs.h"
#include "pm_device.cuh"

using namespace mvsdev;

namespace {

// ---------------------------------------------------------------------------
// Sec. III-D: geometric consistency.  Reading: the z-depth of X in view j is
// compared with the bilinear depth of view j at x'_j (a tap without depth
// makes the view inconsistent); the normal of view j at the rounded x'_j is
// rotated into the reference frame and compared sign-agnostically; the
// reprojection goes back through d_j(x'_j).  Kept with >= min_consistent.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mat3v(const float* M, float a, float b, float c, float& o0, float& o1, float& o2) {
    o0 = fmaf(M[0], a, fmaf(M[1], b, M[2] * c));
    o1 = fmaf(M[3], a, fmaf(M[4], b, M[5] * c));
    o2 = fmaf(M[6], a, fmaf(M[7], b, M[8] * c));
}

// Memory-bound (71 % of the DRAM's rate): pixels of wrong depth project
// anywhere, so the sources are read about three times.  A block is a 32 x 8
// tile, so that the source pixels its projections share are in L1 whatever the
// direction a source turns a row to.  That gives little (3072 x 2048, ten
// sources, timed in turn: 647 us in rows of 256, 633 in tiles, about what runs
// differ by; 16 x 16 the same, 8 x 32 slower than rows).
constexpr int kGeoX = 32, kGeoY = 8;
__global__ void __launch_bounds__(kGeoX * kGeoY) k_geo_filter(const __grid_constant__ FilterConst fc,
                                                              uint8_t* __restrict__ keep, int32_t* __restrict__ count) {
    const int x = blockIdx.x * kGeoX + threadIdx.x % kGeoX, y = blockIdx.y * kGeoY + threadIdx.x / kGeoX;
    if (x >= fc.W || y >= fc.H) return;
    const int i = y * fc.W + x;   // at most 2^30 pixels
    float4 pl = fc.plane[i];
    int cnt = 0;
    if (pl.w > 0.0f) {
        float r0, r1, r2;
        mat3v(fc.Kinv, (float)x, (float)y, 1.0f, r0, r1, r2);
        float X0 = pl.w * r0, X1 = pl.w * r1, X2 = pl.w * r2;
        for (int jj = 0; jj < fc.n_src; ++jj) {
            const FilterConst::Src& S = fc.src[jj];
            float Y0, Y1, Y2;
            mat3v(S.R, X0, X1, X2, Y0, Y1, Y2);
            Y0 += S.t[0]; Y1 += S.t[1]; Y2 += S.t[2];
            if (!(Y2 > 0.0f)) continue;
            float q0, q1, q2;
            mat3v(S.K, Y0, Y1, Y2, q0, q1, q2);
            float u = q0 / q2, v = q1 / q2;
            if (!(u >= 0.0f && u <= (float)(S.W - 1) && v >= 0.0f && v <= (float)(S.H - 1))) continue;
            int x0 = (int)floorf(u), y0 = (int)floorf(v);
            int x1 = min(x0 + 1, S.W - 1), y1 = min(y0 + 1, S.H - 1);
            float da = S.plane[y0 * S.W + x0].w, db = S.plane[y0 * S.W + x1].w;
            float dc = S.plane[y1 * S.W + x0].w, de = S.plane[y1 * S.W + x1].w;
            if (!(da > 0.0f && db > 0.0f && dc > 0.0f && de > 0.0f)) continue;
            float fx = u - (float)x0, fy = v - (float)y0;
            float dj = (1.0f - fy) * ((1.0f - fx) * da + fx * db) + fy * ((1.0f - fx) * dc + fx * de);
            float diff = fabsf(dj - Y2);
            if (fc.depth_relative) diff /= Y2;
            if (!(diff < fc.depth_tol)) continue;
            int xn = min((int)floorf(u + 0.5f), S.W - 1), yn = min((int)floorf(v + 0.5f), S.H - 1);
            float4 nj = S.plane[yn * S.W + xn];
            // R^T n_j
            float m0 = S.R[0] * nj.x + S.R[3] * nj.y + S.R[6] * nj.z;
            float m1 = S.R[1] * nj.x + S.R[4] * nj.y + S.R[7] * nj.z;
            float m2 = S.R[2] * nj.x + S.R[5] * nj.y + S.R[8] * nj.z;
            float cs = fabsf(pl.x * m0 + pl.y * m1 + pl.z * m2) /
                       sqrtf((pl.x * pl.x + pl.y * pl.y + pl.z * pl.z) * (m0 * m0 + m1 * m1 + m2 * m2));
            if (!(cs > fc.cos_max)) continue;
            float s0, s1, s2;
            mat3v(S.Kinv, u, v, 1.0f, s0, s1, s2);
            float Z0 = dj * s0 - S.t[0], Z1 = dj * s1 - S.t[1], Z2 = dj * s2 - S.t[2];
            float B0 = S.R[0] * Z0 + S.R[3] * Z1 + S.R[6] * Z2;
            float B1 = S.R[1] * Z0 + S.R[4] * Z1 + S.R[7] * Z2;
            float B2 = S.R[2] * Z0 + S.R[5] * Z1 + S.R[8] * Z2;
            if (!(B2 > 0.0f)) continue;
            float e0, e1, e2;
            mat3v(fc.K, B0, B1, B2, e0, e1, e2);
            float eu = e0 / e2 - (float)x, ev = e1 / e2 - (float)y;
            if (!(sqrtf(eu * eu + ev * ev) < fc.max_reproj)) continue;
            cnt++;
        }
    }
    if (count) count[i] = cnt;
    keep[i] = (uint8_t)(pl.w > 0.0f && cnt >= fc.min_consistent);
}

// ---------------------------------------------------------------------------
// Sec. III-E hypotheses.  Direction k: 0 horizontal (1,0), 1 vertical (0,1),
// 2 diagonal 45 deg below (1,1), 3 diagonal 45 deg above (1,-1).  The
// reconstructed pixels are packed into bits along each direction, so that a
// pixel finds its neighbours on a line by scanning words (32 pixels per load,
// the next ones usually in the same word) instead of following per-pixel
// distances that a thread per line wrote walking it (1.70 ms of serial walks
// and 200 MB of distances at 3072 x 2048; the four bit maps and their summaries
// take 3.5 MB and 0.19 ms).  Bit `pos` of line `li` is word [pos / 32][li] for the
// directions 1-3 (adjacent pixels read adjacent words) and [li][pos / 32]
// along the rows.  The position is x for direction 0, else y (x for the
// diagonals of images more than 32 times as high as wide, which keeps the maps
// within 8 words per pixel at any shape); lines are numbered y, x, x - y +
// H - 1, x + y.
// ---------------------------------------------------------------------------
__constant__ int c_dir[4][2] = {{1, 0}, {0, 1}, {1, 1}, {1, -1}};

struct LineMaps {
    int W, H, nwx, nwp;        // words per row; words per diagonal
    bool along_y;              // the diagonals' position is y
    uint32_t* bits[4];
    uint32_t* sum[4];          // bit w of a line's summary: word w of the line is not empty
    __host__ __device__ int lines(int k) const { return k == 0 ? H : (k == 1 ? W : W + H - 1); }
    __host__ __device__ int words(int k) const { return k == 0 ? nwx : (k == 1 ? (H + 31) / 32 : nwp); }
};
__host__ __device__ inline LineMaps line_maps(int W, int H, uint32_t* base) {
    LineMaps m;
    m.W = W;
    m.H = H;
    m.nwx = (W + 31) / 32;
    m.along_y = H / 32 <= W;
    m.nwp = ((m.along_y ? H : W) + 31) / 32;
    for (int k = 0; k < 4; ++k) {
        m.bits[k] = base;
        base += (size_t)m.lines(k) * m.words(k);
    }
    for (int k = 0; k < 4; ++k) {
        m.sum[k] = base;
        base += (size_t)m.lines(k) * ((m.words(k) + 31) / 32);
    }
    return m;
}
size_t line_map_words(int W, int H) {
    const LineMaps m = line_maps(W, H, nullptr);
    size_t n = 0;
    for (int k = 0; k < 4; ++k) n += (size_t)m.lines(k) * (m.words(k) + (m.words(k) + 31) / 32);
    return n;
}

// blockIdx.y = direction; direction 0: one warp per word, else one thread
__global__ void k_line_bits(LineMaps m, const uint8_t* __restrict__ known) {
    const int k = blockIdx.y, W = m.W, H = m.H;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k == 0) {
        const long long w = t >> 5;
        if (w >= (long long)H * m.nwx) return;
        const int y = (int)(w / m.nwx), x = (int)(w % m.nwx) * 32 + (int)(t & 31);
        const unsigned b = __ballot_sync(0xffffffffu, x < W && known[(long long)y * W + x] != 0);
        if ((t & 31) == 0) m.bits[0][w] = b;
        return;
    }
    const int lines = m.lines(k), nw = m.words(k);
    if (t >= (long long)lines * nw) return;
    const int li = (int)(t % lines), p0 = (int)(t / lines) * 32;
    uint32_t b = 0;
#pragma unroll 8
    for (int i = 0; i < 32; ++i) {
        int x, y;
        if (k == 1) {
            x = li;
            y = p0 + i;
        } else {
            const int c = k == 2 ? li - (H - 1) : li;   // x - y, x + y
            if (m.along_y) {
                y = p0 + i;
                x = k == 2 ? c + y : c - y;
            } else {
                x = p0 + i;
                y = k == 2 ? x - c : c - x;
            }
        }
        if (x >= 0 && x < W && y >= 0 && y < H && known[(long long)y * W + x]) b |= 1u << i;
    }
    m.bits[k][t] = b;
}

__global__ void k_line_sums(LineMaps m) {
    const int k = blockIdx.y, lines = m.lines(k), nw = m.words(k), ns = (nw + 31) / 32;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)lines * ns) return;
    // direction 0: [line][word], else [word][line]
    const int li = (int)(k == 0 ? t / ns : t % lines), w0 = (int)(k == 0 ? t % ns : t / lines) * 32;
    uint32_t b = 0;
#pragma unroll 8
    for (int i = 0; i < 32; ++i)
        if (w0 + i < nw && m.bits[k][k == 0 ? (long long)li * nw + w0 + i : (long long)(w0 + i) * lines + li]) b |= 1u << i;
    m.sum[k][t] = b;
}

// One side of a line: set bits strictly below (up = false) or above `pos`, in
// order of distance; empty words are skipped through the summary, 32 at a time.
struct LineScan {
    const uint32_t* base;
    const uint32_t* sums;
    long long stride, sum_stride;
    int ns, w, sw;             // summary words; current word and summary word
    uint32_t word, sum;        // bits of word w, and of the summary past w, not taken yet
    bool up;
    // distance of the next reconstructed pixel from `pos`, 0 if there is none
    __device__ __forceinline__ int next(int pos) {
        if (!word) {
            while (!sum) {
                sw += up ? 1 : -1;
                if (sw < 0 || sw >= ns) return 0;
                sum = __ldg(sums + sw * sum_stride);
            }
            const int b = up ? __ffs(sum) - 1 : 31 - __clz(sum);
            sum ^= 1u << b;
            w = 32 * sw + b;
            word = __ldg(base + w * stride);
        }
        const int b = up ? __ffs(word) - 1 : 31 - __clz(word);
        word ^= 1u << b;
        return up ? 32 * w + b - pos : pos - (32 * w + b);
    }
};

// least-squares line v = a + b t through the n_fit <= NF reconstructed pixels
// nearest along the line (negative side first at equal distance), value at
// t = 0; centred normal equations in float.  One thread per pixel and
// direction.
template <int NF>
__global__ void k_line_fit(LineMaps lm, const float* __restrict__ depth, const uint8_t* __restrict__ known, int n_fit,
                           int inverse, float d_lo, float d_hi, float* __restrict__ hyp, uint8_t* __restrict__ valid) {
    const int W = lm.W, H = lm.H;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long i = t >> 2;
    const int k = (int)t & 3;
    if (i >= (long long)W * H) return;
    float h = 0.0f;
    bool ok = false;
    if (!known[i]) {
        const int x = (int)(i % W), y = (int)(i / W);
        const int sx = c_dir[k][0], sy = c_dir[k][1];
        const int li = k == 0 ? y : (k == 1 ? x : (k == 2 ? x - y + H - 1 : x + y));
        const int pos = k == 0 || (k >= 2 && !lm.along_y) ? x : y;
        // along direction 3 with the position y, "before" is towards larger y
        const bool flip = k == 3 && lm.along_y;
        LineScan before, after;
        const int lines = lm.lines(k), nw = lm.words(k), ns = (nw + 31) / 32;
        before.base = lm.bits[k] + (k == 0 ? (long long)li * nw : li);
        before.sums = lm.sum[k] + (k == 0 ? (long long)li * ns : li);
        before.stride = before.sum_stride = k == 0 ? 1 : lines;
        before.ns = ns;
        before.w = pos >> 5;
        before.sw = pos >> 10;
        const uint32_t w0 = __ldg(before.base + before.w * before.stride);
        const uint32_t s0 = __ldg(before.sums + before.sw * before.sum_stride);
        after = before;
        before.up = flip;
        after.up = !flip;
        auto below = [](uint32_t v, int b) { return v & ((1u << b) - 1u); };
        auto above = [](uint32_t v, int b) { return v & ~((2u << b) - 1u); };
        const int pb = pos & 31, wb = before.w & 31;
        before.word = flip ? above(w0, pb) : below(w0, pb);
        before.sum = flip ? above(s0, wb) : below(s0, wb);
        after.word = flip ? below(w0, pb) : above(w0, pb);
        after.sum = flip ? below(s0, wb) : above(s0, wb);
        int dl = before.next(pos), dr = after.next(pos);   // distances of the next candidates on each side (0 = none)
        float ts[NF], vs[NF];
        int m = 0;
        float tsum = 0.0f;
#pragma unroll
        for (int a = 0; a < NF; ++a) {
            if (a >= n_fit || (dl == 0 && dr == 0)) break;
            const bool take_left = dl > 0 && (dr == 0 || dl <= dr);
            const int off = take_left ? -dl : dr;
            const float dv = depth[(long long)(y + off * sy) * W + (x + off * sx)];
            ts[a] = (float)off;
            vs[a] = inverse ? 1.0f / dv : dv;
            tsum += ts[a];
            m++;
            if (take_left) dl = before.next(pos);
            else dr = after.next(pos);
        }
        if (m >= 2) {
            float tm = tsum / (float)m, vm = 0.0f;
#pragma unroll
            for (int a = 0; a < NF; ++a)
                if (a < m) vm += vs[a];
            vm /= (float)m;
            float stt = 0.0f, stv = 0.0f;
#pragma unroll
            for (int a = 0; a < NF; ++a)
                if (a < m) {
                    float dt = ts[a] - tm;
                    stt = fmaf(dt, dt, stt);
                    stv = fmaf(dt, vs[a] - vm, stv);
                }
            float b = stv / stt;
            float av = vm - b * tm;
            h = inverse ? 1.0f / av : av;
            ok = h >= d_lo && h <= d_hi;
        }
    }
    hyp[t] = ok ? h : 0.0f;
    valid[t] = ok ? 1 : 0;
}

// ---------------------------------------------------------------------------
// hypothesis cost: fronto-parallel plane z = h, n = (0, 0, -1) (Sec. III-E)
// ---------------------------------------------------------------------------
constexpr int kBlock = 128;
constexpr int kWarps = kBlock / 32;

// One warp per pixel of the grid of every `step`-th row and column (the MRF
// reads the costs at half resolution, so the inference scores those only), the
// four hypotheses of a pixel in lanes 0..3.  5 blocks per SM (96 registers) as
// in the other kernels of one visit per pixel.
template <int G, int S>
__global__ void __launch_bounds__(kBlock, S <= 9 ? 5 : S <= 11 ? 4 : 3)
    k_phi_cost(const __grid_constant__ RefConst rc, const float* __restrict__ hyp, const uint8_t* __restrict__ valid,
               float* __restrict__ hcost, int step) {
    extern __shared__ __align__(16) unsigned char smem[];
    ViewSm* views = reinterpret_cast<ViewSm*>(smem);
    load_views(rc, views);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Ws = (rc.W + step - 1) / step, Hs = (rc.H + step - 1) / step;
    const long long npix = (long long)Ws * Hs;
    unsigned nev = 0;
    for (long long b = (long long)blockIdx.x * kWarps + warp; b < npix; b += (long long)gridDim.x * kWarps) {
        const int px = (int)(b % Ws) * step, py = (int)(b / Ws) * step;
        const long long a = (long long)py * rc.W + px;
        bool v = lane < 4 && valid[4 * a + lane] != 0;
        if (!__any_sync(0xffffffffu, v)) {
            if (lane < 4) hcost[4 * a + lane] = kCmax;
            continue;
        }
        PixWin<S> pw;
        build_window<G, S>(rc, px, py, true, pw);
        float h = lane < 4 ? hyp[4 * a + lane] : 1.0f;
        float c = kCmax;
        if (pw.ok) {
            PixView* pv = warp_pixviews(smem, rc.n_src, warp);
            pix_views(rc, views, px, py, pv);
            Cand my = make_cand(rc, pw, pw.geo, 0.0f, 0.0f, -1.0f, h, v);
            c = eval_batch<G, S, false>(rc, views, pw, pw.geo, pv, my, 4, warp_pairs(smem, rc.n_src, warp), nullptr,
                                        nev);
        }
        if (lane < 4) hcost[4 * a + lane] = v ? c : kCmax;
    }
}

// ---------------------------------------------------------------------------
// MRF (Eq. 6-9) at half resolution (node (gx, gy) <- pixel (2gx, 2gy)).
// Reading: TRW = sequential tree-reweighted min-sum message passing with
// rows and columns as monotonic chains (node weight 1 / max(#earlier,
// #later present neighbours)); one iteration = forward pass in raster order +
// backward pass; decode = per-node argmin of the belief (lowest label on a
// tie).  A node depends on its up / left neighbours only (forward; on its down
// / right ones in the backward pass, which runs the same schedule on the
// mirrored grid), so the rows run as a pipeline with the messages of the
// sequential sweep (up to rounding next to holes with one hypothesis, see
// from_known).
//
// What bounds it: a chain of gw + gh - 1 dependent nodes.  One warp walks one
// row, lane (d, lq, l) evaluating the min-sum term of own label l towards
// label lq of the d-th outgoing neighbour (down, right); the message to the
// right stays in the warp's registers and the message down goes to the next
// row's warp through a ring in shared memory (kTrwRows rows per block) or, at
// the last row of a block, through global memory.  The data is its own flag:
// an empty slot holds kTrwEmpty, a bit pattern no message has, so the reader
// polls the words it needs and nothing else is signalled; the reader of a ring
// slot empties it again and the writer finds it empty before it writes.
// Blocks are co-resident (cooperative launch) and every poll is bounded.
//
// Work that does not depend on the messages stays out of the chain: the pair
// energies of Eq. 7 come from a table (k_mrf_pairs), unaries and static
// messages are fetched a chunk of 32 columns ahead, and a message to a node
// with one label is zero (its only entry is its own minimum), so only nodes
// with several labels and their neighbours are walked.
//
// 1536 x 1024 nodes, a quarter of them holes: 0.95 ms per pass against 5.43 ms
// with 32 x 32 tiles and grid barriers (1.1 us per anti-diagonal: 32 warps of
// one multiprocessor each evaluating the logarithms between block barriers);
// all nodes holes 1.96 ms, none 0.03 ms.  A node takes about 0.3 us of a lone
// warp's issue (0.6 us with eight rows waiting on one another); 12 rows per
// block are the same within 1 %, 4 rows 4 % of the whole inference slower, and
// one lane per (direction, label) over all own labels 10 % slower.
// ---------------------------------------------------------------------------
constexpr int kTrwRows = 8, kTrwCols = 32, kTrwRing = 128;
constexpr uint32_t kTrwEmpty = 0xffffffffu;
// polls per wait before it gives up (a few tenths of a second to a second;
// a pass takes a millisecond), and in the check of that path
constexpr unsigned kTrwPolls = 1u << 23, kTrwPollsGlobal = 1u << 21, kTrwPollsTest = 1u << 10;

struct MrfBufs {
    int gw, gh;
    int8_t* nlab;     // labels per node (0 = absent)
    int8_t* lmap;     // [4] hypothesis index of each label (-1 = reconstructed pixel)
    float* lab;       // [4] label depths
    float* un;        // [4] unary energies -log phi_n
    float* msg;       // [4 dir][4 lab] incoming messages (dir 0 up, 1 down, 2 left, 3 right)
    float* pair;      // [2][4][4] Eq. 7 energies of (own label, neighbour's label): neighbour below, right
    float* bnd;       // messages into the first row of each strip of kTrwRows rows: [strip][gw][4]
    int* status;      // of this call: MVS_DEV_TIMEOUT once a wait ran out; the labels are then -2 and no map is written
};

__global__ void k_mrf_setup(int W, int H, MrfBufs mb, const uint8_t* __restrict__ known,
                            const float* __restrict__ depth, const float* __restrict__ hyp,
                            const uint8_t* __restrict__ valid, const float* __restrict__ hcost, float k1, float k2) {
    long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (long long)mb.gw * mb.gh) return;
    if (g == 0) *mb.status = 0;
    int gx = (int)(g % mb.gw), gy = (int)(g / mb.gw);
    long long i = (long long)(2 * gy) * W + 2 * gx;
    int L = 0;
    float lab[4] = {0.f, 0.f, 0.f, 0.f}, un[4] = {0.f, 0.f, 0.f, 0.f};
    int8_t lm[4] = {0, 0, 0, 0};
    if (known[i]) {
        lab[0] = depth[i];
        lm[0] = -1;
        L = 1;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (valid[4 * i + k]) {
                const float h = hyp[4 * i + k];
                const float u = -logf((kCmax - hcost[4 * i + k]) / k1 + k2);   // Eq. 6
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q == L) { lab[q] = h; un[q] = u; lm[q] = (int8_t)k; }
                L++;
            }
    }
    reinterpret_cast<float4*>(mb.lab)[g] = make_float4(lab[0], lab[1], lab[2], lab[3]);
    reinterpret_cast<float4*>(mb.un)[g] = make_float4(un[0], un[1], un[2], un[3]);
    reinterpret_cast<char4*>(mb.lmap)[g] = make_char4(lm[0], lm[1], lm[2], lm[3]);
    mb.nlab[g] = (int8_t)L;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    float4* m = reinterpret_cast<float4*>(mb.msg) + 4 * g;
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = z;
}

// ((((a + b) + c) + d) + e): the belief sum in message-slot order
__device__ __forceinline__ float un_add4(float a, float b, float c, float d, float e) {
    return (((a + b) + c) + d) + e;
}

// -log of Eq. 7: phi_e = [k3 - min(1, relative difference)]^2
__device__ __forceinline__ float pair_energy(float h1, float h2, float k3) {
    float rel = h1 > h2 ? (h1 - h2) / h2 : (h2 - h1) / h1;
    return -2.0f * logf(k3 - fminf(1.0f, rel));
}

// Pair energies of the edges whose messages are not trivially zero (one end
// with several labels, the other present): thread (node, d, a) fills the four
// entries of own label a towards the labels of the neighbour below (d 0) or
// right (d 1).
__global__ void k_mrf_pairs(MrfBufs mb, float k3) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long g = t >> 3;
    if (g >= (long long)mb.gw * mb.gh) return;
    const int d = (int)(t >> 2) & 1, a = (int)t & 3;
    const int x = (int)(g % mb.gw), y = (int)(g / mb.gw);
    if (d ? x + 1 >= mb.gw : y + 1 >= mb.gh) return;
    const long long q = d ? g + 1 : g + mb.gw;
    const int L = mb.nlab[g], Lq = mb.nlab[q];
    if (a >= L || Lq < 1 || (L < 2 && Lq < 2)) return;
    const float h = mb.lab[4 * g + a];
    const float4 hq = reinterpret_cast<const float4*>(mb.lab)[q];
    float4 o;
    o.x = pair_energy(h, hq.x, k3);
    o.y = Lq > 1 ? pair_energy(h, hq.y, k3) : 0.0f;
    o.z = Lq > 2 ? pair_energy(h, hq.z, k3) : 0.0f;
    o.w = Lq > 3 ? pair_energy(h, hq.w, k3) : 0.0f;
    reinterpret_cast<float4*>(mb.pair)[t] = o;
}

// A warp's chunk of 32 columns.
struct TrwChunk {
    float un[kTrwCols * 4];    // unaries
    float mv[kTrwCols * 4];    // static message from the pass-local lower neighbour
    float mh[kTrwCols * 4];    // static message from the pass-local right neighbour
    float mu[kTrwCols * 4];    // message from the upper neighbour if that has one label (else unused)
    float ml[kTrwCols * 4];    // message from the left neighbour likewise
    float gamma[kTrwCols];
    uint32_t info[kTrwCols];   // labels of the node | lower << 8 | right << 16 | left neighbour << 24
    float pair[kTrwCols * 32]; // the node's two pair-energy tables
};
// Shared memory of a block: per warp two chunks (the current and the next one's
// pair tables) and the ring of messages into its row.
struct TrwSm {
    TrwChunk chunk[kTrwRows][2];
    float ring[kTrwRows][kTrwRing * 4];
};

// TEST: the first strip is left out, so that the wait for it runs out (a
// variant of its own: with limits taken from the arguments an inference of
// 3072 x 2048 took 5.30 ms instead of 5.16)
template <bool TEST>
__global__ void __launch_bounds__(32 * kTrwRows, 1) k_trw_rows(MrfBufs mb, bool forward) {
    constexpr unsigned polls = TEST ? kTrwPollsTest : kTrwPolls, polls_global = TEST ? kTrwPollsTest : kTrwPollsGlobal;
    extern __shared__ __align__(16) unsigned char trw_smem[];
    TrwSm& sm = *reinterpret_cast<TrwSm*>(trw_smem);
    __shared__ volatile int dead;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) dead = 0;
    for (int i = tid; i < kTrwRows * kTrwRing * 4; i += blockDim.x)
        (&sm.ring[0][0])[i] = __uint_as_float(kTrwEmpty);
    __syncthreads();
    // after a pass that gave up no wait goes on (looked at by the block's last
    // row, which starts last)
    if (tid == 32 * (kTrwRows - 1) && __ldcg(mb.status)) dead = 1;
    const int ns = (mb.gh + kTrwRows - 1) / kTrwRows;
    // message slots (dir 0 up, 1 down, 2 left, 3 right) in pass-local terms:
    // the static ones come from the lower / right neighbours, the dynamic
    // ones from the upper / left neighbours updated earlier in this pass
    const int sv = forward ? 1 : 0, sh = forward ? 3 : 2;
    // original node index of pass-local (xf, yf), or -1 outside the grid
    auto node = [&](int xf, int yf) -> long long {
        if (xf < 0 || yf < 0 || xf >= mb.gw || yf >= mb.gh) return -1;
        const int x = forward ? xf : mb.gw - 1 - xf, y = forward ? yf : mb.gh - 1 - yf;
        return (long long)y * mb.gw + x;
    };
    auto labels = [&](long long i) { return i >= 0 ? (int)__ldg(mb.nlab + i) : 0; };
    const int dsel = lane >> 4, lq = (lane >> 2) & 3, l = lane & 3;
    const int dir = forward ? (dsel ? 3 : 1) : (dsel ? 2 : 0);
    // entry (own label l, target's label lq) of a pair table: the table
    // belongs to the upper / left end of the edge
    const int pe_at = dsel * 16 + (forward ? l * 4 + lq : lq * 4 + l);
    volatile float* ring_in = sm.ring[warp];
    const bool to_ring = warp + 1 < kTrwRows;
    volatile float* ring_out = sm.ring[to_ring ? warp + 1 : 0];

    // each warp runs its row of every strip of the block, in order; row y
    // waits for row y - 1 only, so the lowest unfinished row always advances
    for (int st = (TEST ? 1 : 0) + blockIdx.x; st < ns; st += gridDim.x) {
        const int yf = st * kTrwRows + warp;
        if (yf >= mb.gh) break;
        float* bnd_in = mb.bnd + (long long)st * mb.gw * 4;
        float* bnd_out = bnd_in + (long long)mb.gw * 4;
        const bool last_row = yf + 1 >= mb.gh;
        float4 f_un, f_mv, f_mh, f_mu, f_ml;
        float f_gm = 1.0f;
        uint32_t f_info = 0;
        int f_lu = 0;
        // message to node i (L labels) from its pass-local upper (d 0) or left
        // (d 1) neighbour q with one label: every label of i sees the same
        // belief of q, which the normalisation takes out, so the message is
        // the pair energies less their minimum, whatever the pass; also stored
        // for the other pass.  For a reconstructed neighbour, whose belief is
        // zero, that is the sweep's message bit for bit; a hole with a single
        // hypothesis has a unary and messages, which cancel up to rounding.
        auto from_known = [&](long long i, long long q, int d, int L) {
            float v[4];
            if (forward) {
                const float4 t = reinterpret_cast<const float4*>(mb.pair)[8 * q + 4 * d];
                v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = k < L ? mb.pair[32 * i + 16 * d + 4 * k] : 0.0f;
            }
            float mn = 3.0e38f;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < L) mn = fminf(mn, v[k]);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = k < L ? v[k] - mn : 0.0f;
            const float4 o = make_float4(v[0], v[1], v[2], v[3]);
            __stcg(reinterpret_cast<float4*>(mb.msg + 16 * i + 4 * ((forward ? 0 : 1) + 2 * d)), o);
            return o;
        };
        // lane c's node of the chunk at x0: into registers, and its pair
        // tables into the chunk buffer in the background
        auto fetch = [&](int x0, TrwChunk& C) {
            const int xf = x0 + lane;
            const long long i = node(xf, yf);
            f_un = f_mv = f_mh = f_mu = f_ml = make_float4(0.f, 0.f, 0.f, 0.f);
            f_info = 0;
            f_gm = 1.0f;
            f_lu = 0;
            const int L = labels(i);
            if (L >= 2) {
                const long long qd = node(xf, yf + 1), qr = node(xf + 1, yf);
                const long long qu = node(xf, yf - 1), ql = node(xf - 1, yf);
                const int Ld = labels(qd), Lr = labels(qr), Lu = labels(qu), Ll = labels(ql);
                const int mx = max((Lu > 0) + (Ll > 0), (Ld > 0) + (Lr > 0));
                f_gm = mx > 0 ? 1.0f / (float)mx : 1.0f;
                f_info = (uint32_t)L | ((uint32_t)Ld << 8) | ((uint32_t)Lr << 16) | ((uint32_t)Ll << 24);
                f_lu = Lu;
                f_un = reinterpret_cast<const float4*>(mb.un)[i];
                f_mv = __ldcg(reinterpret_cast<const float4*>(mb.msg + 16 * i + 4 * sv));
                f_mh = __ldcg(reinterpret_cast<const float4*>(mb.msg + 16 * i + 4 * sh));
                if (Lu == 1) f_mu = from_known(i, qu, 0, L);
                if (Ll == 1) f_ml = from_known(i, ql, 1, L);
                const uint32_t dst = (uint32_t)__cvta_generic_to_shared(C.pair + 32 * lane);
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    const long long o = forward ? i : (d ? qr : qd);   // the edge's upper / left end
                    if ((d ? Lr : Ld) < 2) continue;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 64u * d + 16u * k),
                                     "l"(mb.pair + 32 * o + 16 * d + 4 * k)
                                     : "memory");
                }
            }
        };
        // warp 0: the words of the 8 columns from x8 that came from the strip
        // above (lane = column, word)
        auto peek = [&](int x8) {
            const int x = x8 + (lane >> 2);
            return x < mb.gw ? __ldcv(bnd_in + 4 * x + (lane & 3)) : 0.0f;
        };
        float left_in = 0.0f;             // message from the last node to its right neighbour
        int seen8 = -1;                   // warp 0: the 8 columns that `seen` holds, all there
        float seen = 0.0f, ahead = 0.0f;
        fetch(0, sm.chunk[warp][0]);
        if (warp == 0 && st > 0) ahead = peek(0);
        int ahead8 = 0;
        for (int x0 = 0; x0 < mb.gw; x0 += kTrwCols) {
            TrwChunk& C = sm.chunk[warp][(x0 / kTrwCols) & 1];
            asm volatile("cp.async.wait_all;" ::: "memory");
            reinterpret_cast<float4*>(C.un)[lane] = f_un;
            reinterpret_cast<float4*>(C.mv)[lane] = f_mv;
            reinterpret_cast<float4*>(C.mh)[lane] = f_mh;
            reinterpret_cast<float4*>(C.mu)[lane] = f_mu;
            reinterpret_cast<float4*>(C.ml)[lane] = f_ml;
            C.gamma[lane] = f_gm;
            C.info[lane] = f_info;
            // the nodes with several labels, and those of them with a message
            // from such a node of the row above
            unsigned todo = __ballot_sync(0xffffffffu, f_info != 0);
            const unsigned in_up = __ballot_sync(0xffffffffu, f_lu >= 2);
            __syncwarp();
            if (x0 + kTrwCols < mb.gw) fetch(x0 + kTrwCols, sm.chunk[warp][((x0 / kTrwCols) & 1) ^ 1]);
            while (todo) {
                const int c = __ffs(todo) - 1, x = x0 + c;
                todo &= todo - 1u;
                const uint32_t info = C.info[c];
                const int L = info & 255, Ld = (info >> 8) & 255, Lr = (info >> 16) & 255;
                const float unl = C.un[4 * c + l], mvl = C.mv[4 * c + l], mhl = C.mh[4 * c + l], gm = C.gamma[c];
                const float pe = C.pair[32 * c + pe_at];
                // (a left neighbour with several labels was this warp's last node)
                const float dynh = (info >> 24) >= 2 ? left_in : C.ml[4 * c + l];
                // ---- message from the row above
                float dynv = C.mu[4 * c + l];
                if ((in_up >> c) & 1u) {
                    bool ok = false;
                    if (warp > 0) {
                        volatile float* slot = ring_in + 4 * (x & (kTrwRing - 1));
                        for (unsigned it = 0; it < polls; ++it) {
                            dynv = slot[l];
                            ok = __all_sync(0xffffffffu, __float_as_uint(dynv) != kTrwEmpty);
                            if (ok || __any_sync(0xffffffffu, dead)) break;
                        }
                        if (lane < 4) slot[lane] = __uint_as_float(kTrwEmpty);
                    } else {
                        const int x8 = x & ~7;
                        ok = true;
                        if (seen8 != x8) {
                            // every word of the 8 columns that will come
                            const unsigned live8 = (in_up >> (x8 - x0)) & 255u;
                            const bool want = (live8 >> (lane >> 2)) & 1u;
                            seen = ahead8 == x8 ? ahead : peek(x8);
                            for (unsigned it = 0; it < polls_global; ++it) {
                                ok = __all_sync(0xffffffffu, !want || __float_as_uint(seen) != kTrwEmpty);
                                if (ok || __any_sync(0xffffffffu, dead)) break;
                                seen = peek(x8);
                            }
                            seen8 = x8;
                            ahead8 = x8 + 8;
                            ahead = peek(ahead8);
                        }
                        dynv = __shfl_sync(0xffffffffu, seen, 4 * (x - x8) + l);
                    }
                    if (!ok) {
                        if (lane == 0) {
                            dead = 1;
                            *reinterpret_cast<volatile int*>(mb.status) = MVS_DEV_TIMEOUT;
                        }
                        return;
                    }
                }
                // ---- belief of own label l: unary + the four incoming messages in slot order
                const float bel = forward ? un_add4(unl, dynv, mvl, dynh, mhl) : un_add4(unl, mvl, dynv, mhl, dynh);
                const int Lq = dsel ? Lr : Ld;
                float e = 3.0e38f;
                if (l < L && lq < Lq && Lq >= 2) e = fmaf(gm, bel, -(dsel ? mhl : mvl)) + pe;
                // minimum over own labels, then over the target's labels (normalisation)
                e = fminf(e, __shfl_xor_sync(0xffffffffu, e, 1));
                e = fminf(e, __shfl_xor_sync(0xffffffffu, e, 2));
                float mn = fminf(e, __shfl_xor_sync(0xffffffffu, e, 4));
                mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 8));
                const float o = lq < Lq ? e - mn : 0.0f;
                // lane j < 4: the message to label j of the node below (sent by
                // lane 4 j); every lane: the message to label l of the right
                // node (sent by lane 16 + 4 l)
                left_in = __shfl_sync(0xffffffffu, o, 16 + 4 * l);
                const float out_v = __shfl_sync(0xffffffffu, o, 4 * l);
                if (Ld >= 2 && !last_row) {
                    if (to_ring) {
                        volatile float* slot = ring_out + 4 * (x & (kTrwRing - 1));
                        bool ok = false;
                        for (unsigned it = 0; it < polls; ++it) {
                            ok = __all_sync(0xffffffffu, lane >= 4 || __float_as_uint(slot[lane & 3]) == kTrwEmpty);
                            if (ok || __any_sync(0xffffffffu, dead)) break;
                        }
                        if (!ok) {
                            if (lane == 0) {
                                dead = 1;
                                *reinterpret_cast<volatile int*>(mb.status) = MVS_DEV_TIMEOUT;
                            }
                            return;
                        }
                        if (lane < 4) slot[lane] = out_v;
                    } else if (lane < 4) {
                        __stcg(bnd_out + 4 * x + lane, out_v);
                    }
                }
                if (l == 0 && lq < Lq && Lq >= 2) {
                    const long long q = dsel == 0 ? node(x, yf + 1) : node(x + 1, yf);
                    __stcg(mb.msg + 16 * q + 4 * (dir ^ 1) + lq, o);
                }
            }
        }
    }
}

// (host_status: a word that the host sees, set when a pass gave up)
__global__ void k_trw_decode(MrfBufs mb, int32_t* __restrict__ label, int* __restrict__ host_status) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)mb.gw * mb.gh) return;
    const int gave_up = __ldg(mb.status);
    int L = mb.nlab[i];
    if (gave_up && i == 0) *host_status = gave_up;
    if (!L || gave_up) { label[i] = -2; return; }
    int best = 0;
    float bv = 3.0e38f;
    for (int l = 0; l < L; ++l) {
        float b = mb.un[4 * i + l];
        for (int d = 0; d < 4; ++d) b += mb.msg[16 * i + 4 * d + l];
        if (b < bv) { bv = b; best = l; }
    }
    label[i] = mb.lmap[4 * i + best];
}

// ---------------------------------------------------------------------------
// selection: nearest up-sampled decoded depth is the reference; the closest
// valid hypothesis (lowest k on a tie) becomes the new depth of a hole
// ---------------------------------------------------------------------------
__global__ void k_select(int W, int H, const uint8_t* __restrict__ known, const float* __restrict__ hyp,
                         const uint8_t* __restrict__ valid, const int32_t* __restrict__ label,
                         const float4* __restrict__ plane, float* __restrict__ newd) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)W * H) return;
    int x = (int)(i % W), y = (int)(i / W);
    if (known[i]) { newd[i] = plane[i].w; return; }
    int gw = (W + 1) / 2;
    long long g = (long long)(y / 2) * gw + (x / 2);
    int lb = label[g];
    float nd = 0.0f;
    if (lb >= -1) {
        long long ni = (long long)(2 * (y / 2)) * W + 2 * (x / 2);
        float rd = lb == -1 ? plane[ni].w : hyp[4 * ni + lb];
        float bd = 3.0e38f;
        for (int k = 0; k < 4; ++k)
            if (valid[4 * i + k]) {
                float e = fabsf(hyp[4 * i + k] - rd);
                if (e < bd) { bd = e; nd = hyp[4 * i + k]; }
            }
    }
    newd[i] = nd;
}

// PHI-MVS/M (Sec. IV, Table I: the MRF removed): each hole takes its valid
// hypothesis of minimal matching cost, the lowest k on a tie; a hole without
// a valid hypothesis gets no depth
__global__ void k_select_min_cost(long long n, const uint8_t* __restrict__ known, const float* __restrict__ hyp,
                                  const uint8_t* __restrict__ valid, const float* __restrict__ hcost,
                                  const float4* __restrict__ plane, float* __restrict__ newd) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (known[i]) { newd[i] = plane[i].w; return; }
    const float4 h = reinterpret_cast<const float4*>(hyp)[i];
    const float4 c = reinterpret_cast<const float4*>(hcost)[i];
    const uchar4 v = reinterpret_cast<const uchar4*>(valid)[i];
    const float hv[4] = {h.x, h.y, h.z, h.w}, cv[4] = {c.x, c.y, c.z, c.w};
    const bool ok[4] = {v.x != 0, v.y != 0, v.z != 0, v.w != 0};
    int bk = -1;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (ok[k] && (bk < 0 || cv[k] < cv[bk])) bk = k;
    newd[i] = bk >= 0 ? hv[bk] : 0.0f;
}

// Eq. 10 normal from the back-projected 4-neighbours (reading: unit length,
// oriented towards the camera); a hole without all four neighbours stays
// empty.  (gave_up: MrfBufs::status of the labels' message passing, or null;
// then the map stays as it is)
__global__ void k_eq10(const __grid_constant__ RefConst rc, const uint8_t* __restrict__ known,
                       const float* __restrict__ newd, float4* __restrict__ plane, const int* __restrict__ gave_up) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int W = rc.W, H = rc.H;
    if (i >= (long long)W * H) return;
    const int keep = gave_up ? __ldg(gave_up) : 0;   // (tested at the end: nothing waits for it)
    if (known[i]) return;
    int x = (int)(i % W), y = (int)(i / W);
    float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
    float d = newd[i];
    if (d > 0.0f && x >= 1 && y >= 1 && x <= W - 2 && y <= H - 2) {
        const int nx[4] = {x, x, x - 1, x + 1}, ny[4] = {y - 1, y + 1, y, y};
        float P[4][3];
        bool ok = true;
        for (int k = 0; k < 4; ++k) {
            float dk = newd[(long long)ny[k] * W + nx[k]];
            if (!(dk > 0.0f)) { ok = false; break; }
            float r0, r1, r2;
            mat3v(rc.Kinv, (float)nx[k], (float)ny[k], 1.0f, r0, r1, r2);
            P[k][0] = dk * r0; P[k][1] = dk * r1; P[k][2] = dk * r2;
        }
        if (ok) {
            float a0 = P[0][0] - P[1][0], a1 = P[0][1] - P[1][1], a2 = P[0][2] - P[1][2];
            float b0 = P[2][0] - P[3][0], b1 = P[2][1] - P[3][1], b2 = P[2][2] - P[3][2];
            float n0 = a1 * b2 - a2 * b1, n1 = a2 * b0 - a0 * b2, n2 = a0 * b1 - a1 * b0;
            float len = sqrtf(n0 * n0 + n1 * n1 + n2 * n2);
            if (len > 0.0f) {
                n0 /= len; n1 /= len; n2 /= len;
                float r0, r1, r2;
                mat3v(rc.Kinv, (float)x, (float)y, 1.0f, r0, r1, r2);
                if (n0 * r0 + n1 * r1 + n2 * r2 > 0.0f) { n0 = -n0; n1 = -n1; n2 = -n2; }
                out = make_float4(n0, n1, n2, d);
            }
        }
    }
    if (!keep) plane[i] = out;
}

__global__ void k_known_from_cost(long long n, const float4* __restrict__ plane, const float* __restrict__ cost,
                                  float hole_cost, uint8_t* __restrict__ known, float* __restrict__ depth) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float d = plane[i].w;
    bool k = d > 0.0f && cost[i] < hole_cost;
    known[i] = k ? 1 : 0;
    depth[i] = k ? d : 0.0f;
}

__global__ void k_depth_of(long long n, const float4* __restrict__ plane, const uint8_t* __restrict__ known,
                           float* __restrict__ depth) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    depth[i] = known[i] ? plane[i].w : 0.0f;
}

unsigned blocks_for(long long n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

cudaError_t launch_geo_filter(const FilterConst& fc, uint8_t* keep, int32_t* count, cudaStream_t s) {
    k_geo_filter<<<dim3(blocks_for(fc.W, kGeoX), blocks_for(fc.H, kGeoY)), kGeoX * kGeoY, 0, s>>>(fc, keep, count);
    count_launch();
    return cudaGetLastError();
}

// Fixed line-map scratch of mvs_phi_hypotheses_static: 8 words per pixel (no
// shape of an image needs more, see LineMaps) for up to
// MVS_PHI_STATIC_MAX_PIXELS pixels, in the library's own device memory.
static __device__ __align__(256) int32_t g_phi_gaps_static[8 * (size_t)MVS_PHI_STATIC_MAX_PIXELS];

// Device address of g_phi_gaps_static on the current device, looked up once
// per device with that device current (host code only sees a stand-in for the
// symbol, never its device address).
cudaError_t phi_static_scratch(int32_t** out) {
    static std::mutex mu;
    static int32_t* ptr[128] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_phi_gaps_static);
        if (e != cudaSuccess) return e;
        ptr[dev] = (int32_t*)p;
    }
    *out = ptr[dev];
    return cudaSuccess;
}

cudaError_t launch_phi_hypotheses(int W, int H, const float* depth, const uint8_t* known, int n_fit, int inverse,
                                  float d_lo, float d_hi, float* hyp, uint8_t* valid, int32_t* scratch,
                                  cudaStream_t s) {
    const LineMaps lm = line_maps(W, H, (uint32_t*)scratch);
    const long long n = (long long)W * H;
    const long long threads = std::max({32LL * H * lm.nwx, (long long)W * ((H + 31) / 32),
                                        (long long)lm.nwp * (W + H - 1)});
    k_line_bits<<<dim3(blocks_for(threads, 256), 4), 256, 0, s>>>(lm, known);
    count_launch();
    const long long sums = ((long long)W + H - 1) * ((std::max(lm.nwx, (H + 31) / 32) + 31) / 32);
    k_line_sums<<<dim3(blocks_for(sums, 256), 4), 256, 0, s>>>(lm);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (n_fit <= 8)
        k_line_fit<8><<<blocks_for(4 * n, 256), 256, 0, s>>>(lm, depth, known, n_fit, inverse, d_lo, d_hi, hyp, valid);
    else
        k_line_fit<32><<<blocks_for(4 * n, 256), 256, 0, s>>>(lm, depth, known, n_fit, inverse, d_lo, d_hi, hyp, valid);
    count_launch();
    return cudaGetLastError();
}

// scratch of launch_phi_hypotheses, in 32-bit words (at most 8 per pixel)
size_t phi_line_words(int W, int H) { return line_map_words(W, H); }

#define MVS_DISPATCH(n, CALL)                       \
    do {                                            \
        int _s = (n) * (n);                         \
        if (_s <= 16) { CALL(4, 4); }               \
        else if (_s <= 36) { CALL(4, 9); }          \
        else if (_s <= 64) { CALL(8, 8); }          \
        else if (_s <= 128) { CALL(16, 8); }        \
        else if (_s <= 176) { CALL(16, 11); }       \
        else if (_s <= 256) { CALL(16, 16); }       \
        else if (_s <= 320) { CALL(32, 10); }       \
        else if (_s <= 384) { CALL(32, 12); }       \
        else if (_s <= 448) { CALL(32, 14); }       \
        else { CALL(32, 16); }                      \
    } while (0)

cudaError_t launch_phi_cost(const RefConst& rc, const float* hyp, const uint8_t* valid, float* hcost, int step,
                            cudaStream_t s) {
    long long npix = (long long)((rc.W + step - 1) / step) * ((rc.H + step - 1) / step);
    const size_t smem = smem_block_bytes(rc.n_src, kWarps);
    const long long units = (npix + kWarps - 1) / kWarps;
#define CALL(G, S)                                                                                        \
    k_phi_cost<G, S><<<pm_grid_for((const void*)k_phi_cost<G, S>, units, smem, kBlock), kBlock, smem, s>>>( \
        rc, hyp, valid, hcost, step)
    MVS_DISPATCH(rc.n, CALL);
#undef CALL
    count_launch();
    const cudaError_t g = pm_grid_error();
    return g != cudaSuccess ? g : cudaGetLastError();
}

size_t phi_mrf_work_floats(int W, int H) {
    size_t g = (size_t)((W + 1) / 2) * ((H + 1) / 2);
    const size_t strips = ((size_t)(H + 1) / 2 + kTrwRows - 1) / kTrwRows;
    // msg 16, lab 4, un 4, pair 32 floats; nlab 1 + lmap 4 bytes (rounded up to 2 floats); strip boundaries; the status
    return g * (16 + 4 + 4 + 32 + 2) + strips * ((size_t)(W + 1) / 2) * 4 + 64;
}

cudaError_t launch_phi_mrf(int W, int H, const uint8_t* known, const float* depth, const float* hyp,
                           const uint8_t* valid, const float* hcost, float k1, float k2, float k3, int iters,
                           int32_t* label, float* work, int* status, bool test_timeout, const int** gave_up,
                           cudaStream_t s) {
    MrfBufs mb;
    mb.gw = (W + 1) / 2;
    mb.gh = (H + 1) / 2;
    long long g = (long long)mb.gw * mb.gh;
    mb.msg = work;
    mb.lab = mb.msg + 16 * g;
    mb.un = mb.lab + 4 * g;
    mb.pair = mb.un + 4 * g;
    const long long ns = (mb.gh + kTrwRows - 1) / kTrwRows;
    mb.bnd = mb.pair + 32 * g;
    mb.status = (int*)(mb.bnd + 4 * ns * mb.gw);
    mb.lmap = (int8_t*)(mb.status + 4);
    mb.nlab = mb.lmap + 4 * g;
    *gave_up = mb.status;
    k_mrf_setup<<<blocks_for(g, 256), 256, 0, s>>>(W, H, mb, known, depth, hyp, valid, hcost, k1, k2);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (iters > 0) {
        k_mrf_pairs<<<blocks_for(8 * g, 256), 256, 0, s>>>(mb, k3);
        count_launch();
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // one block per strip, at most as many as are co-resident; the shared-
    // memory opt-in and the occupancy belong to the current device
    const void* const kernel = test_timeout ? (const void*)k_trw_rows<true> : (const void*)k_trw_rows<false>;
    int max_blocks = 0;
    {
        static std::mutex mu;
        static int per_dev[2][128] = {};
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lk(mu);
        if (!per_dev[test_timeout][dev]) {
            int sms = 0, per_sm = 0;
            if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
            if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)sizeof(TrwSm))) != cudaSuccess)
                return e;
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * kTrwRows,
                                                                   sizeof(TrwSm))) != cudaSuccess)
                return e;
            if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
            per_dev[test_timeout][dev] = sms * per_sm;
        }
        max_blocks = per_dev[test_timeout][dev];
    }
    dim3 grid((unsigned)std::max<long long>(1, std::min<long long>(ns, max_blocks))), block(32 * kTrwRows);
    for (int it = 0; it < iters; ++it)
        for (int pass = 0; pass < 2; ++pass) {
            bool forward = pass == 0;
            void* args[] = {(void*)&mb, (void*)&forward};
            if ((e = cudaMemsetAsync(mb.bnd, 0xff, sizeof(float) * 4 * ns * mb.gw, s)) != cudaSuccess) return e;
            e = cudaLaunchCooperativeKernel(kernel, grid, block, args, sizeof(TrwSm), s);
            count_launch();
            if (e != cudaSuccess) return e;
        }
    k_trw_decode<<<blocks_for(g, 256), 256, 0, s>>>(mb, label, status);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_phi_select(const RefConst& rc, const uint8_t* known, const float* hyp, const uint8_t* valid,
                              const int32_t* label, float4* plane, float* newdepth, const int* gave_up,
                              cudaStream_t s) {
    long long n = (long long)rc.W * rc.H;
    k_select<<<blocks_for(n, 256), 256, 0, s>>>(rc.W, rc.H, known, hyp, valid, label, plane, newdepth);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_eq10<<<blocks_for(n, 256), 256, 0, s>>>(rc, known, newdepth, plane, gave_up);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_phi_select_min_cost(const RefConst& rc, const uint8_t* known, const float* hyp,
                                       const uint8_t* valid, const float* hcost, float4* plane, float* newdepth,
                                       cudaStream_t s) {
    long long n = (long long)rc.W * rc.H;
    k_select_min_cost<<<blocks_for(n, 256), 256, 0, s>>>(n, known, hyp, valid, hcost, plane, newdepth);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_eq10<<<blocks_for(n, 256), 256, 0, s>>>(rc, known, newdepth, plane, nullptr);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_known_from_cost(int W, int H, const float4* plane, const float* cost, float hole_cost,
                                   uint8_t* known, float* depth, cudaStream_t s) {
    long long n = (long long)W * H;
    k_known_from_cost<<<blocks_for(n, 256), 256, 0, s>>>(n, plane, cost, hole_cost, known, depth);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_depth_of(int W, int H, const float4* plane, const uint8_t* known, float* depth, cudaStream_t s) {
    long long n = (long long)W * H;
    k_depth_of<<<blocks_for(n, 256), 256, 0, s>>>(n, plane, known, depth);
    count_launch();
    return cudaGetLastError();
}
