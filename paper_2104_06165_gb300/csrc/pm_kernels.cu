// PatchMatch kernels: texture build, random initialisation, plane-map cost
// and one checkerboard phase (propagation + random refinement).
//   Sec. III-B  random initialisation
//   Sec. III-C  Eq. 4 weighted ZNCC, Eq. 5 aggregation, refinement
//   Sec. III    red-black checkerboard updating
#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <unordered_map>

#include "pm_device.cuh"

using namespace mvsdev;

namespace {

constexpr int kBlock = 128;

// ---------------------------------------------------------------------------
// bilinear-coefficient texture (layout documented in mvs_internal.h)
// ---------------------------------------------------------------------------
__global__ void k_build_texture(const uint8_t* __restrict__ img, int W, int H, int pitch, uint2* __restrict__ tex) {
    long long n = (long long)(W + 1) * (H + 1);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        int i = (int)(t % (W + 1)) - 1, j = (int)(t / (W + 1)) - 1;
        int x0 = min(max(i, 0), W - 1), x1 = min(max(i + 1, 0), W - 1);
        int y0 = min(max(j, 0), H - 1), y1 = min(max(j + 1, 0), H - 1);
        float p00 = img[(long long)y0 * W + x0], p01 = img[(long long)y0 * W + x1];
        float p10 = img[(long long)y1 * W + x0], p11 = img[(long long)y1 * W + x1];
        __half2 ab = __floats2half2_rn(p00 + p01 + p10 + p11, (p01 - p00) + (p11 - p10));
        __half2 cd = __floats2half2_rn((p10 - p00) + (p11 - p01), p00 - p01 - p10 + p11);
        uint2 q;
        q.x = *reinterpret_cast<const uint32_t*>(&ab);
        q.y = *reinterpret_cast<const uint32_t*>(&cd);
        tex[(long long)(j + 1) * pitch + (i + 1)] = q;
    }
}

// Per-block shared memory: the source-view table and one pair list per warp.
constexpr int kWarps = kBlock / 32;
// Checkerboard phases: one block per SM whose warps take single pixels of the
// active colour from the block's tiles, 1 x kTileY such pixels each.  A short
// tile leaves the blocks even (320 x 240, 3 iterations: 1108 us with 8 pixels,
// 1139 with 16, 1239 with 32; 1511 x 1007 the same within 1 %), a vertical
// one shares more L1 lines than a square (2 x 10: 4 % slower).
constexpr int kTileY = 8;
// Warps of the block: 24 at 80 registers (11 x 11 samples: 80 to 120 bytes
// spilled outside the sample loop) were chosen with the windows read back and
// an earlier sample loop (1511 x 1007, 8 iterations: 75.0 ms against 78.2 with
// 20 at 96, 78.6 with 16, 75.5 with 28).  With this loop 20 are a little better
// where the windows are read back (24 / 20 warps, timed in turn: 320 x 240 1058
// / 1042 us, 1511 x 1007 76.3 / 75.6 ms, 3072 x 2048 383 / 367 ms, six views in
// a batch 127.2 / 124.6 ms); where they are rebuilt (two phases from a given
// state, 1536 x 1024, 24 / 20 / 16 warps) mixed precision takes 18.5 / 18.5 /
// 19.0 ms and FP32 18.4 / 18.6 / 17.6.  Layouts with more slots per lane need
// the registers.
template <int S>
constexpr int phase_max_warps() { return S <= 9 ? 24 : S <= 11 ? 20 : S <= 14 ? 16 : 12; }

// Blocks of the one-hypothesis kernels per SM: 5 (96 registers, no spills)
// for windows of up to 9 slots per lane; 16 slots need more registers.
template <int S>
constexpr int one_hyp_blocks() { return S <= 9 ? 5 : S <= 11 ? 4 : S <= 14 ? 3 : 1; }

// ---------------------------------------------------------------------------
// Sec. III-B: random initialisation, then the cost of the initial plane.
// One warp per pixel, grid-stride over the pixels.
// ---------------------------------------------------------------------------
template <int G, int S, bool MIXED>
__global__ void __launch_bounds__(kBlock, one_hyp_blocks<S>()) k_init(const __grid_constant__ RefConst rc) {
    extern __shared__ __align__(16) unsigned char smem[];
    ViewSm* views = reinterpret_cast<ViewSm*>(smem);
    load_views(rc, views);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long npix = (long long)rc.W * rc.H;
    unsigned nev = 0, it = 0;
    // the draws of this warp's next 32 pixels, one per lane: the depth's
    // uniform and the normal before it is turned to the camera
    float u0 = 0.0f, dn0 = 0.0f, dn1 = 0.0f, dn2 = 0.0f;
    for (long long a = (long long)blockIdx.x * kWarps + warp; a < npix; a += (long long)gridDim.x * kWarps, ++it) {
        const int px = (int)(a % rc.W), py = (int)(a / rc.W);
        PixWin<S> pw;
        build_window<G, S>(rc, px, py, true, pw);
        if (rc.win) store_window<G, S>(rc.win + a * win_record_floats(G, S), pw);
        if ((it & 31u) == 0) {
            float u[3];
            draws3(rc, a + (long long)lane * gridDim.x * kWarps, -1, u);
            float st, ct, sp, cp;
            sincosf(2.0f * kPi * u[1], &st, &ct);
            sincosf(kPi * (u[2] - 0.5f), &sp, &cp);
            u0 = u[0];
            dn0 = ct * sp;
            dn1 = st * sp;
            dn2 = cp;
        }
        const float u = __shfl_sync(0xffffffffu, u0, it & 31u);
        float n0 = __shfl_sync(0xffffffffu, dn0, it & 31u), n1 = __shfl_sync(0xffffffffu, dn1, it & 31u);
        float n2 = __shfl_sync(0xffffffffu, dn2, it & 31u);
        float d = rc.d_lo + (rc.d_hi - rc.d_lo) * u;
        if (rc.init_range) {   // Sec. III-B: a depth between the nearest sparse features
            const float2 r = rc.init_range[a];
            if (r.x == r.x) d = r.x + (r.y - r.x) * u;
        }
        if (n0 * pw.geo.rx0 + n1 * pw.geo.rx1 + n2 * pw.geo.rx2 > 0.0f) {   // face the camera
            n0 = -n0;
            n1 = -n1;
            n2 = -n2;
        }
        float c = kCmax;
        if (pw.ok) {
            PixView* pv = warp_pixviews(smem, rc.n_src, warp);
            pix_views(rc, views, px, py, pv);
            Cand my = make_cand(rc, pw, pw.geo, n0, n1, n2, d, lane == 0);
            c = eval_batch<G, S, false, MIXED>(rc, views, pw, pw.geo, pv, my, 1, warp_pairs(smem, rc.n_src, warp),
                                               nullptr, nev);
        }
        if (lane == 0) {
            rc.plane[a] = make_float4(n0, n1, n2, d);
            rc.cost[a] = c;
        }
    }
    flush_evals(rc.eval_counter, nev);
}

// the stored windows of a call that starts from given planes
template <int G, int S>
__global__ void __launch_bounds__(kBlock, one_hyp_blocks<S>()) k_window(const __grid_constant__ RefConst rc) {
    const int warp = threadIdx.x >> 5;
    const long long npix = (long long)rc.W * rc.H;
    for (long long a = (long long)blockIdx.x * kWarps + warp; a < npix; a += (long long)gridDim.x * kWarps) {
        PixWin<S> pw;
        build_window<G, S>(rc, (int)(a % rc.W), (int)(a / rc.W), true, pw);
        store_window<G, S>(rc.win + a * win_record_floats(G, S), pw);
    }
}

// cost of a given plane map
template <int G, int S, bool MIXED>
__global__ void __launch_bounds__(kBlock, one_hyp_blocks<S>())
    k_cost(const __grid_constant__ RefConst rc, const float4* __restrict__ plane, float* __restrict__ cost,
           float* view_cost) {
    extern __shared__ __align__(16) unsigned char smem[];
    ViewSm* views = reinterpret_cast<ViewSm*>(smem);
    load_views(rc, views);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long npix = (long long)rc.W * rc.H;
    unsigned nev = 0;
    for (long long a = (long long)blockIdx.x * kWarps + warp; a < npix; a += (long long)gridDim.x * kWarps) {
        const int px = (int)(a % rc.W), py = (int)(a / rc.W);
        PixWin<S> pw;
        build_window<G, S>(rc, px, py, true, pw);
        float4 pl = plane[a];
        float* vc = view_cost ? view_cost + a * rc.n_src : nullptr;
        float c = kCmax;
        if (pw.ok) {
            PixView* pv = warp_pixviews(smem, rc.n_src, warp);
            pix_views(rc, views, px, py, pv);
            Cand my = make_cand(rc, pw, pw.geo, pl.x, pl.y, pl.z, pl.w, lane == 0);
            c = eval_batch<G, S, true, MIXED>(rc, views, pw, pw.geo, pv, my, 1, warp_pairs(smem, rc.n_src, warp), vc,
                                              nev);
        } else if (vc && lane < rc.n_src) {
            vc[lane] = kCmax;
        }
        if (lane == 0) cost[a] = c;
    }
    flush_evals(rc.eval_counter, nev);
}

// ---------------------------------------------------------------------------
// Checkerboard phase.  Reading of the cited (undescribed) sampling pattern:
// eight groups of other-colour neighbours, the member with the lowest stored
// cost of each group is a candidate (first listed wins a tie).
//   groups 0..3: near V-shapes up / down / left / right, six members
//   groups 4..7: far lines up / down / left / right at distances 5, 7, .., 25
// ---------------------------------------------------------------------------
// offset of member k of group g (members past the group's size: any in-range
// shift value, masked by the caller)
__device__ __forceinline__ void group_member(int g, int k, int& dx, int& dy) {
    if (g < 4) {
        k = min(k, 5);
        // up-pointing V {(0,-1), (-1,-2), (1,-2), (-2,-3), (0,-3), (2,-3)},
        // packed 3 bits per member (x + 2, y + 3), rotated per group
        const int a = (int)((0x220CAu >> (3 * k)) & 7u) - 2;   // x + 2: 2, 1, 3, 0, 2, 4
        const int b = (int)((0x4Au >> (3 * k)) & 7u) - 3;      // y + 3: 2, 1, 1, 0, 0, 0
        switch (g) {
            case 0: dx = a; dy = b; break;
            case 1: dx = a; dy = -b; break;
            case 2: dx = b; dy = a; break;
            default: dx = -b; dy = a; break;
        }
    } else {
        const int dist = 5 + 2 * k;
        dx = g == 6 ? -dist : (g == 7 ? dist : 0);
        dy = g == 4 ? -dist : (g == 5 ? dist : 0);
    }
}

// The 8 groups x 16 member slots as the phase kernel scans them: entry
// 16 g + k of the block's table is the pixel-index offset of member k of group
// g and its (dx + 32) << 8 | (dy + 32), or -1 past the group's size.
constexpr int kMemberSlots = 128, kReach = 25;   // members lie at most kReach pixels away
__device__ __forceinline__ void fill_members(const RefConst& rc, int2* tab) {
    for (int i = threadIdx.x; i < kMemberSlots; i += blockDim.x) {
        const int g = i >> 4, k = i & 15;
        int dx, dy;
        group_member(g, k, dx, dy);
        const bool in = k < (g < 4 ? 6 : 11);
        tab[i] = in ? make_int2(dy * rc.W + dx, ((dx + 32) << 8) | (dy + 32)) : make_int2(0, -1);
    }
}

// Member of group g with the lowest stored cost (in-image members only, the
// first listed wins a tie), as a pixel index on lane g < 8, or -1, with its
// position.  The 128 slots are spread over 4 registers of the warp (register
// r, lane l: slot 32 r + l), each half warp takes the minimum of its register,
// and the lowest member holding it wins; stored costs are >= 0, so their bit
// patterns order like the values.  The members have the other colour, which
// this phase does not write.  The table replaces the offset arithmetic and,
// away from the image border, the bounds tests.
__device__ __forceinline__ int best_members(const RefConst& rc, const int2* tab, int px, int py, int& member, int& x2,
                                            int& y2) {
    const int lane = threadIdx.x & 31, half = lane >> 4;
    const int pix = py * rc.W + px;
    const bool inner = px >= kReach && py >= kReach && px < rc.W - kReach && py < rc.H - kReach;   // warp-uniform
    unsigned first[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int2 e = tab[32 * r + lane];
        bool in = e.y >= 0;
        if (!inner) {
            const int x = px + (e.y >> 8) - 32, y = py + (e.y & 0xff) - 32;
            in = in && x >= 0 && x < rc.W && y >= 0 && y < rc.H;
        }
        const unsigned bits = in ? __float_as_uint(__ldg(rc.cost + (pix + e.x)) + 0.0f) : 0xffffffffu;
        const unsigned mn0 = __reduce_min_sync(0xffffffffu, half ? 0xffffffffu : bits);
        const unsigned mn1 = __reduce_min_sync(0xffffffffu, half ? bits : 0xffffffffu);
        first[r] = __ballot_sync(0xffffffffu, in && bits == (half ? mn1 : mn0));
    }
    int q = -1;
    member = -1;
    x2 = y2 = 0;
    if (lane < 8) {
        const unsigned fm = lane & 4 ? (lane & 2 ? first[3] : first[2]) : (lane & 2 ? first[1] : first[0]);
        const unsigned m = (fm >> (16 * (lane & 1))) & 0xffffu;
        if (m) {
            member = __ffs(m) - 1;
            const int2 e = tab[16 * lane + member];
            x2 = px + (e.y >> 8) - 32;
            y2 = py + (e.y & 0xff) - 32;
            q = pix + e.x;
        }
    }
    return q;
}

// Refinement perturbations (Sec. III-C) of one iteration, both colours, one
// pixel per thread: delta_d in [-d_hi/4, d_hi/4], and cos / sin of
// delta_theta in [-pi/2, pi/2] and of delta_phi in [-pi/12, pi/12].  Drawn
// ahead of the phases: one pixel per lane, not one per warp.
__global__ void __launch_bounds__(256) k_draws(const __grid_constant__ RefConst rc, int iter) {
    const long long n = (long long)rc.W * rc.H;
    for (long long a = blockIdx.x * 256LL + threadIdx.x; a < n; a += gridDim.x * 256LL) {
        const int x = (int)(a % rc.W), y = (int)(a / rc.W);
        float u[3];
        draws3(rc, a, 2 * iter + ((x + y) & 1), u);
        float sdt, cdt, sdp, cdp;
        sincosf((2.0f * u[1] - 1.0f) * (kPi * 0.5f), &sdt, &cdt);
        sincosf((2.0f * u[2] - 1.0f) * (kPi / 12.0f), &sdp, &cdp);
        rc.draw4[a] = make_float4((2.0f * u[0] - 1.0f) * (rc.d_hi * 0.25f), cdt, sdt, cdp);
        rc.draw1[a] = sdp;
    }
}

// Per-warp state of the current pixel kept in shared memory rather than in
// registers through the evaluation rounds: its window geometry, its plane and
// cost so far, its perturbations, and the hypothesis each lane proposes in the
// current stage.
struct __align__(16) PhaseWarp {
    WinGeo geo;
    float draw[5];     // delta_d, cos / sin delta_theta, cos / sin delta_phi
    float cur_c, pad_[2];
    float4 cur;
    float4 hyp[8];     // the stage's hypotheses (at most 8: propagation groups, proposals, refinement)
};
// Landing buffer of a warp (floats): the next pixel's perturbations (5, padded)
// after its stored window (rec floats, 0 when windows are rebuilt).
constexpr int kDrawFloats = 8;
// Shared memory of a phase block (the same for both precisions).
__host__ __device__ constexpr size_t phase_smem_bytes(int n_src, int warps, int rec) {
    return smem_block_bytes(n_src, warps) +
           (size_t)warps * (sizeof(PhaseWarp) + (size_t)(rec + kDrawFloats) * sizeof(float));
}

// Warps of a phase block: phase_max_warps<S>(), or fewer when the warps' pair
// lists (which grow with the number of sources) would exceed the per-block
// shared memory.
// The limit is a property of the current device (queried once per device;
// a failed query leaves 48 KB, the limit without the opt-in).
int max_block_smem() {
    static std::atomic<int> bytes[128];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return 48 * 1024;
    int v = bytes[dev].load();
    if (v == 0) {
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || v <= 0)
            return 48 * 1024;
        bytes[dev].store(v);
    }
    return v;
}
template <int S>
int phase_warps(int n_src, int rec) {
    int w = phase_max_warps<S>();
    // the kernel's static shared memory (member table, queue) counts as well
    while (w > 1 && phase_smem_bytes(n_src, w, rec) + kMemberSlots * sizeof(int2) + 64 > (size_t)max_block_smem()) --w;
    return w;
}

// Tiles are visited in super-tiles of kSuperX x kSuperY tiles (fewer at the
// right and lower edge) so that the pixels in flight at once form a compact
// region (a smaller source footprint in L2; within a phase the order of the
// pixels does not change the result).  Pixel of the active colour that slot
// `slot` of tile t < ntx * nty covers, as y << 16 | x (sides are at most
// 32768), or -1.
constexpr int kSuperX = 8, kSuperY = 32;
__device__ __forceinline__ int phase_pixel(const RefConst& rc, int t, int slot, int color, int ntx, int nty) {
    const int sr = t / (kSuperY * ntx), r = t - sr * kSuperY * ntx;    // row of super-tiles
    const int h = min(kSuperY, nty - kSuperY * sr);
    const int sc = r / (kSuperX * h), r2 = r - sc * kSuperX * h;       // super-tile of the row
    const int w = min(kSuperX, ntx - kSuperX * sc);
    const int ry = r2 / w, rx = r2 - ry * w;
    const int py = (sr * kSuperY + ry) * kTileY + slot, px = 2 * (sc * kSuperX + rx) + ((py + color) & 1);
    return px < rc.W && py < rc.H ? (py << 16) | px : -1;
}

template <int G, int S, bool MIXED, bool STORED>
__global__ void __launch_bounds__(32 * phase_max_warps<S>(), 1)
    k_phase(const __grid_constant__ RefConst rc, int phase) {
    const int kWarpsB = (int)(blockDim.x >> 5);   // phase_warps<S>, chosen by the host
    extern __shared__ __align__(16) unsigned char smem[];   // phase_smem_bytes(n_src, kWarpsB, record floats)
    __shared__ int2 members[kMemberSlots];
    __shared__ int queue;    // pixels of this block's tiles handed to its warps so far
    ViewSm* views = reinterpret_cast<ViewSm*>(smem);
    fill_members(rc, members);
    if (threadIdx.x == 0) queue = 0;
    load_views(rc, views);   // (ends with a block barrier)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int color = phase & 1;
    constexpr int kRec = STORED ? win_record_floats(G, S) : 0;
    PhaseWarp* ws = reinterpret_cast<PhaseWarp*>(smem + smem_block_bytes(rc.n_src, kWarpsB)) + warp;
    // the next pixel's stored window and perturbations land here while the
    // current one is scored
    float* land = reinterpret_cast<float*>(smem + smem_block_bytes(rc.n_src, kWarpsB) +
                                           (size_t)kWarpsB * sizeof(PhaseWarp)) + (size_t)warp * (kRec + kDrawFloats);
    const int ntx = (rc.W + 1) >> 1, nty = (rc.H + kTileY - 1) / kTileY;
    // The block takes every gridDim.x-th tile and its warps draw the tiles'
    // pixels from one queue, in order: the warps of an SM stay on neighbouring
    // pixels (which share L1 lines) and end together, although the work of a
    // pixel varies several-fold.  Returns a phase_pixel, or -1 at the end.
    auto take = [&]() {
        for (;;) {
            int i = 0;
            if (lane == 0) i = atomicAdd(&queue, 1);
            i = __shfl_sync(0xffffffffu, i, 0);
            const int t = (int)blockIdx.x + i / kTileY * (int)gridDim.x;
            if (t >= ntx * nty) return -1;
            const int p = phase_pixel(rc, t, i % kTileY, color, ntx, nty);
            if (p >= 0) return p;
        }
    };
    auto fetch = [&](int p) {
        if (p < 0) return;
        const long long a = (long long)(p >> 16) * rc.W + (p & 0xffff);
        if constexpr (STORED) fetch_window<G, S>(land, rc.win + a * kRec);
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(land + kRec);
        if (lane == 30)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(rc.draw4 + a) : "memory");
        if (lane == 31)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 16u), "l"(rc.draw1 + a) : "memory");
    };
    PixWin<S> pw;
    bool o2_full = false;   // pw.o2 holds the offsets of a window wholly inside the image
    unsigned nev = 0;
    int next = take();
    fetch(next);
    while (next >= 0) {
        const int px = next & 0xffff, py = next >> 16;
        const long long pix = (long long)py * rc.W + px;
        fetch_wait();
        __syncwarp();
        if constexpr (STORED) {
            const float2* wp = reinterpret_cast<const float2*>(land) + (lane & (G - 1));
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const float2 v = wp[s * G];
                pw.w[s] = v.x;
                pw.wr[s] = v.y;
            }
            pw.ok = land[2 * G * S + 12] != 0.0f;
            if (lane < 12) reinterpret_cast<float*>(&ws->geo)[lane] = land[2 * G * S + lane];
        }
        if (lane < 5) ws->draw[lane] = land[kRec + lane];
        __syncwarp();
        next = take();
        fetch(next);
        if constexpr (STORED) {
            if (!pw.ok) continue;   // flat patch: every hypothesis costs C_max
            int ku_lo, ku_hi, kv_lo, kv_hi;
            window_range(rc, px, py, ku_lo, ku_hi, kv_lo, kv_hi);
            const bool full = ku_lo == 0 && kv_lo == 0 && ku_hi == rc.n - 1 && kv_hi == rc.n - 1;
            if (!full || !o2_full) window_offsets<G, S>(rc, ku_lo, ku_hi, kv_lo, kv_hi, pw.o2);
            o2_full = full;
        } else {
            build_window<G, S>(rc, px, py, true, pw);
            if (!pw.ok) continue;
            if (lane == 0) ws->geo = pw.geo;
        }
        // the pixel's state waits in shared memory (fewer live registers
        // through the evaluation rounds)
        if (lane == 0) {
            ws->cur = rc.plane[pix];
            ws->cur_c = rc.cost[pix];
        }
        PixView* pv = warp_pixviews(smem, rc.n_src, warp);
        pix_views(rc, views, px, py, pv);   // (ends with a warp barrier)
        const WinGeo& geo = ws->geo;

        // ---- propagation: lane g < 8 takes group g's cheapest member and
        // carries its plane over
        int member, x2, y2;
        const int q = best_members(rc, members, px, py, member, x2, y2);
        // candidate memo: group g's (member, plane generation) now and at this
        // pixel's last visit in this call; an unchanged one was scored then
        uint32_t key = 0xfffffffeu;
        bool repeat = false;
        if (lane < 8) {
            if (q >= 0) key = ((uint32_t)member << 28) | (__ldg(rc.gen + q) & 0x0fffffffu);
            repeat = q >= 0 && key == rc.memo[pix * MVS_MEMO_WORDS + lane];
        }
        float4 np = make_float4(0.f, 0.f, -1.f, 1.f);
        float d = 0.0f;
        bool ok = q >= 0;
        if (ok) {
            // the neighbour's plane carried over as a plane (reading)
            np = rc.plane[q];
            const float* Ki = rc.Kinv;
            float r0 = fmaf(Ki[0], (float)x2, fmaf(Ki[1], (float)y2, Ki[2]));
            float r1 = fmaf(Ki[3], (float)x2, fmaf(Ki[4], (float)y2, Ki[5]));
            float r2 = fmaf(Ki[6], (float)x2, fmaf(Ki[7], (float)y2, Ki[8]));
            float rho = np.w * (np.x * r0 + np.y * r1 + np.z * r2);
            float den = np.x * geo.rx0 + np.y * geo.rx1 + np.z * geo.rx2;
            ok = den < 0.0f;
            d = ok ? rho * rcp_approx(den) : 0.0f;
            ok = ok && d >= rc.d_lo && d <= rc.d_hi;
        }
        // A carried-over plane equal (to float rounding) to the pixel's own
        // plane or to an earlier group's plane scores the same cost, so it
        // cannot be strictly cheaper than that plane: it is not evaluated.
        {
            // lane b (b - 1) / 2 + a tests the pair of groups a < b (28 pairs)
            if (lane < 8) ws->hyp[lane] = make_float4(np.x, np.y, np.z, ok ? d : __int_as_float(0x7fc00000));
            __syncwarp();
            const int b = 1 + (lane >= 1) + (lane >= 3) + (lane >= 6) + (lane >= 10) + (lane >= 15) + (lane >= 21);
            const int a = min(lane - b * (b - 1) / 2, 7);
            const unsigned eq = __ballot_sync(0xffffffffu, lane < 28 && same_plane(ws->hyp[b], ws->hyp[a]));
            const int lb = lane & 7;
            const bool dup = ok && (((eq >> (lb * (lb - 1) / 2)) & ((1u << lb) - 1u)) != 0u ||
                                    same_plane(make_float4(np.x, np.y, np.z, d), ws->cur));
            __syncwarp();
            ok = ok && !dup;
        }
        ok = ok && !repeat;
        // stage 0: the eight propagated planes; stage 1: the learned
        // proposals of this pixel (when given); stage 2: the three refinement
        // candidates built from the state after stages 0 and 1.  One call
        // site keeps a single copy of the evaluation in the instruction cache.
        float4 hyp4 = make_float4(np.x, np.y, np.z, d);
        bool want = ok;
        bool changed = false;
#pragma unroll 1
        for (int stage = 0; stage < 3; ++stage) {
            if (stage == 1) {
                if (rc.n_prop == 0) continue;
                // proposals already scored at this pixel in this call (the
                // memo word holds the complement of their mask)
                const uint32_t scored = ~rc.memo[pix * MVS_MEMO_WORDS + 8];
                const bool has = lane < rc.n_prop;
                hyp4 = has ? rc.props[pix * rc.n_prop + lane] : make_float4(0.f, 0.f, -1.f, 0.f);
                want = has && !((scored >> lane) & 1u) && hyp4.w >= rc.d_lo && hyp4.w <= rc.d_hi &&
                       !same_plane(hyp4, ws->cur);
            } else if (stage == 2) {
                const float4 cur = ws->cur;
                // refinement (Sec. III-C): d + delta_d clamped to the range;
                // the normal's angles theta = atan2(m1, m0), phi = acos(m2)
                // (after flipping to m2 >= 0) move by delta_theta, delta_phi,
                // taken through the angle-addition formulas
                const float4 r4 = make_float4(ws->draw[0], ws->draw[1], ws->draw[2], ws->draw[3]);
                const float sdp = ws->draw[4];
                float d_new = fminf(fmaxf(cur.w + r4.x, rc.d_lo), rc.d_hi);
                float m0 = cur.x, m1 = cur.y, m2 = cur.z;
                if (m2 < 0.0f) { m0 = -m0; m1 = -m1; m2 = -m2; }
                const float rr = sqrtf(m0 * m0 + m1 * m1);
                // cos / sin of atan2(m1, m0); atan2(+-0, x) is 0 for x = +0 and pi for x = -0
                const float irr = rr > 0.0f ? 1.0f / rr : 0.0f;
                const float ct = rr > 0.0f ? m0 * irr : (signbit(m0) ? -1.0f : 1.0f), st = m1 * irr;
                const float cp = fminf(1.0f, fmaxf(-1.0f, m2)), sp = sqrtf(fmaxf(0.0f, 1.0f - cp * cp));
                const float ct2 = ct * r4.y - st * r4.z, st2 = st * r4.y + ct * r4.z;
                const float cp2 = cp * r4.w - sp * sdp, sp2 = sp * r4.w + cp * sdp;
                float nn0 = ct2 * sp2, nn1 = st2 * sp2, nn2 = cp2;
                if (nn0 * geo.rx0 + nn1 * geo.rx1 + nn2 * geo.rx2 > 0.0f) {   // face the camera
                    nn0 = -nn0;
                    nn1 = -nn1;
                    nn2 = -nn2;
                }
                // candidates (d_new, n_old), (d_old, n_new), (d_new, n_new) in lanes 0..2
                hyp4 = lane == 0 ? make_float4(cur.x, cur.y, cur.z, d_new)
                     : (lane == 1 ? make_float4(nn0, nn1, nn2, cur.w) : make_float4(nn0, nn1, nn2, d_new));
                want = lane < 3;
            }
            const int nc = stage == 0 ? 8 : (stage == 1 ? rc.n_prop : 3);
            if (lane < 8) ws->hyp[lane] = hyp4;
            Cand my = make_cand(rc, pw, geo, hyp4.x, hyp4.y, hyp4.z, hyp4.w, want);
            float c = eval_batch<G, S, false, MIXED>(rc, views, pw, geo, pv, my, nc,
                                                     warp_pairs(smem, rc.n_src, warp), nullptr,
                                                     nev);   // (ends with a warp barrier)
            float bc;
            int bi = warp_argmin(my.ok ? c : 3.0e38f, nc, bc);
            if (bc < ws->cur_c && lane == 0) {
                ws->cur = ws->hyp[bi];
                ws->cur_c = bc;
                changed = true;
            }
            __syncwarp();
        }
        if (lane == 0) {
            rc.plane[pix] = ws->cur;
            rc.cost[pix] = ws->cur_c;
            if (changed) rc.gen[pix] = rc.gen[pix] + 1u;
        }
        if (lane < 8) rc.memo[pix * MVS_MEMO_WORDS + lane] = key;
        if (lane == 8 && rc.n_prop > 0)
            rc.memo[pix * MVS_MEMO_WORDS + 8] = rc.n_prop >= 32 ? 0u : ~((1u << rc.n_prop) - 1u);
    }
    flush_evals(rc.eval_counter, nev);
}

// grid of the grid-stride kernels: as many blocks as fit on the device at
// once (occupancy query, cached per kernel), at most one warp per unit
}  // namespace

namespace {
thread_local cudaError_t t_grid_err = cudaSuccess;
}

// Launch-shape cache per (device, kernel): the SM count, the dynamic shared
// memory opt-in and the occupancy query are all properties of the current
// device.  A failed query leaves grid 0 (the launch then fails) and the
// query's own error for pm_grid_error().
unsigned pm_grid_for(const void* kernel, long long units, size_t smem, int block) {
    static std::mutex mu;
    struct Cfg { size_t smem; int block, per_sm; };
    static std::map<std::pair<int, const void*>, Cfg> cache;
    static std::map<int, int> sms_of;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        t_grid_err = e;
        return 0;
    }
    {
        std::lock_guard<std::mutex> lk(mu);
        auto si = sms_of.find(dev);
        if (si == sms_of.end()) {
            if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
                t_grid_err = e;
                return 0;
            }
            sms_of[dev] = sms;
        } else {
            sms = si->second;
        }
        const auto key = std::make_pair(dev, kernel);
        auto it = cache.find(key);
        if (it != cache.end() && it->second.smem == smem && it->second.block == block) {
            per_sm = it->second.per_sm;
        } else {
            // 48 KB without the opt-in, static shared memory included
            if (smem > 44 * 1024 &&
                (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
                    cudaSuccess) {
                t_grid_err = e;
                return 0;
            }
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem)) != cudaSuccess) {
                t_grid_err = e;
                return 0;
            }
            per_sm = std::max(per_sm, 1);
            cache[key] = {smem, block, per_sm};
        }
    }
    long long need = units;   // blocks of work
    long long full = (long long)sms * per_sm;
    return (unsigned)std::max<long long>(1, std::min(need, full));
}

cudaError_t pm_grid_error() {
    const cudaError_t e = t_grid_err;
    t_grid_err = cudaSuccess;
    return e;
}

// the error of the launch-shape queries of this thread, else of the launches
static cudaError_t launch_status() {
    const cudaError_t g = pm_grid_error();
    const cudaError_t l = cudaGetLastError();
    return g != cudaSuccess ? g : l;
}

// Lanes per pixel group (G) and slots per lane (S) for an n x n window: the
// smallest built G * S >= n * n, since an empty slot costs as much as a sample.
// The dense windows get layouts of their own (768 x 513, 8 sources, 3
// iterations): 13 x 13 on 16 x 11 instead of 16 x 16 slots 25.3 -> 13.8 ms,
// 17 x 17 on 32 x 10 instead of 32 x 16 38.2 -> 21.6 ms, 19 x 19 on 32 x 12
// 38.8 -> 25.3 ms, 21 x 21 on 32 x 14 39.5 -> 29.7 ms (15 x 15 keeps 16 x 16).
// Slots past the window add exact zeros, so the results are the same bit for
// bit.  lanes_hint 0 picks the default; 4, 8, 16 or 32 picks G.
// The mixed-precision kernels exist for the default layout of each window
// size only.
#define MVS_DISPATCH_DEFAULT(n, CALL)                                                     \
    do {                                                                                  \
        int _s = (n) * (n);                                                               \
        if (_s <= 16) { CALL(4, 4); }                                                     \
        else if (_s <= 36) { CALL(4, 9); }                                                \
        else if (_s <= 64) { CALL(8, 8); }                                                \
        else if (_s <= 128) { CALL(16, 8); }                                              \
        else if (_s <= 176) { CALL(16, 11); }                                             \
        else if (_s <= 256) { CALL(16, 16); }                                             \
        else if (_s <= 320) { CALL(32, 10); }                                             \
        else if (_s <= 384) { CALL(32, 12); }                                             \
        else if (_s <= 448) { CALL(32, 14); }                                             \
        else { CALL(32, 16); }                                                            \
    } while (0)

#define MVS_DISPATCH(n, hint, CALL)                                                       \
    do {                                                                                  \
        int _s = (n) * (n), _h = (hint);                                                  \
        if (_s <= 16) { CALL(4, 4); }                                                     \
        else if (_s <= 36) { if (_h == 8) { CALL(8, 5); } else { CALL(4, 9); } }          \
        else if (_s <= 64) { if (_h == 16) { CALL(16, 4); } else { CALL(8, 8); } }        \
        else if (_s <= 128) {                                                             \
            if (_h == 8) { CALL(8, 16); } else if (_h == 32) { CALL(32, 4); }             \
            else { CALL(16, 8); }                                                         \
        }                                                                                 \
        else if (_s <= 256 && _h == 32) { CALL(32, 8); }                                  \
        else { MVS_DISPATCH_DEFAULT(n, CALL); }                                           \
    } while (0)

template <int G, int S, bool MX>
const void* phase_kernel(const RefConst& rc) {
    return rc.win ? (const void*)k_phase<G, S, MX, true> : (const void*)k_phase<G, S, MX, false>;
}

// floats of shared memory per phase warp for the stored windows
static int phase_rec(const RefConst& rc, int G, int S) { return rc.win ? win_record_floats(G, S) : 0; }

// Resolves (and caches) the grid sizes of the init / cost / phase kernels of
// this configuration without launching anything, so that a later stream
// capture contains kernel launches only.
cudaError_t prime_launch_configs(const RefConst& rc) {
    const size_t smem = smem_block_bytes(rc.n_src, kWarps);
#define CALL(G, S)                                                                                    \
    do {                                                                                              \
        pm_grid_for((const void*)k_init<G, S, MX>, 1, smem, kBlock);                                  \
        pm_grid_for((const void*)k_cost<G, S, MX>, 1, smem, kBlock);                                  \
        const int rec = phase_rec(rc, G, S), w = phase_warps<S>(rc.n_src, rec);                       \
        pm_grid_for(phase_kernel<G, S, MX>(rc), 1, phase_smem_bytes(rc.n_src, w, rec), 32 * w);       \
        if (rc.win) pm_grid_for((const void*)k_window<G, S>, 1, 0, kBlock);                            \
    } while (0)
    if (rc.precision) {
        constexpr bool MX = true;
        MVS_DISPATCH_DEFAULT(rc.n, CALL);
    } else {
        constexpr bool MX = false;
        MVS_DISPATCH(rc.n, rc.lanes_hint, CALL);
    }
#undef CALL
    return launch_status();
}

cudaError_t launch_build_texture(const uint8_t* img, int W, int H, uint2* tex, cudaStream_t s) {
    long long n = (long long)(W + 1) * (H + 1);
    unsigned blocks = (unsigned)std::min<long long>((n + 255) / 256, 152LL * 16);
    k_build_texture<<<blocks, 256, 0, s>>>(img, W, H, tex_pitch(W), tex);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_init(const RefConst& rc, cudaStream_t s) {
    long long npix = (long long)rc.W * rc.H;
    const size_t smem = smem_block_bytes(rc.n_src, kWarps);
    const unsigned units = (unsigned)((npix + kWarps - 1) / kWarps);
#define CALL(G, S) \
    k_init<G, S, MX><<<pm_grid_for((const void*)k_init<G, S, MX>, units, smem, kBlock), kBlock, smem, s>>>(rc)
    if (rc.precision) {
        constexpr bool MX = true;
        MVS_DISPATCH_DEFAULT(rc.n, CALL);
    } else {
        constexpr bool MX = false;
        MVS_DISPATCH(rc.n, rc.lanes_hint, CALL);
    }
#undef CALL
    count_launch();
    return launch_status();
}

cudaError_t launch_cost(const RefConst& rc, const float4* plane, float* cost, float* view_cost, cudaStream_t s) {
    long long npix = (long long)rc.W * rc.H;
    const size_t smem = smem_block_bytes(rc.n_src, kWarps);
    const unsigned units = (unsigned)((npix + kWarps - 1) / kWarps);
#define CALL(G, S)                                                                                         \
    k_cost<G, S, MX><<<pm_grid_for((const void*)k_cost<G, S, MX>, units, smem, kBlock), kBlock, smem, s>>>( \
        rc, plane, cost, view_cost)
    if (rc.precision) {
        constexpr bool MX = true;
        MVS_DISPATCH_DEFAULT(rc.n, CALL);
    } else {
        constexpr bool MX = false;
        MVS_DISPATCH(rc.n, rc.lanes_hint, CALL);
    }
#undef CALL
    count_launch();
    return launch_status();
}

// perturbations of an iteration (both colours)
static void launch_draws(const RefConst& rc, int iter, cudaStream_t s) {
    const long long n = (long long)rc.W * rc.H;
    k_draws<<<(unsigned)std::min<long long>((n + 255) / 256, 152LL * 8), 256, 0, s>>>(rc, iter);
    count_launch();
}

template <int G, int S, bool MX>
void phase_launch(const RefConst& rc, int phase, cudaStream_t s) {
    const int rec = phase_rec(rc, G, S), w = phase_warps<S>(rc.n_src, rec), block = 32 * w;
    const long long ntiles = (long long)((rc.W + 1) / 2) * ((rc.H + kTileY - 1) / kTileY);
    const size_t smem = phase_smem_bytes(rc.n_src, w, rec);
    const unsigned grid = pm_grid_for(phase_kernel<G, S, MX>(rc), ntiles, smem, block);
    if (rc.win) k_phase<G, S, MX, true><<<grid, block, smem, s>>>(rc, phase);
    else k_phase<G, S, MX, false><<<grid, block, smem, s>>>(rc, phase);
}

size_t pm_window_bytes(const RefConst& rc) {
    size_t b = 0;
#define CALL(G, S) b = (size_t)win_record_floats(G, S) * sizeof(float)
    if (rc.precision) {
        MVS_DISPATCH_DEFAULT(rc.n, CALL);
    } else {
        MVS_DISPATCH(rc.n, rc.lanes_hint, CALL);
    }
#undef CALL
    return b;
}

cudaError_t launch_windows(const RefConst& rc, cudaStream_t s) {
    const unsigned units = (unsigned)(((long long)rc.W * rc.H + kWarps - 1) / kWarps);
#define CALL(G, S) k_window<G, S><<<pm_grid_for((const void*)k_window<G, S>, units, 0, kBlock), kBlock, 0, s>>>(rc)
    if (rc.precision) {
        MVS_DISPATCH_DEFAULT(rc.n, CALL);
    } else {
        MVS_DISPATCH(rc.n, rc.lanes_hint, CALL);
    }
#undef CALL
    count_launch();
    return launch_status();
}

cudaError_t launch_memo_reset(const RefConst& rc, cudaStream_t s) {
    return cudaMemsetAsync(rc.memo, 0xff, (size_t)rc.W * rc.H * MVS_MEMO_WORDS * sizeof(uint32_t), s);
}

cudaError_t launch_phase(const RefConst& rc, int phase, bool first, cudaStream_t s) {
    if (first || (phase & 1) == 0) launch_draws(rc, phase >> 1, s);
    if (rc.precision) {
#define CALL(G, S) phase_launch<G, S, true>(rc, phase, s)
        MVS_DISPATCH_DEFAULT(rc.n, CALL);
#undef CALL
    } else {
#define CALL(G, S) phase_launch<G, S, false>(rc, phase, s)
        MVS_DISPATCH(rc.n, rc.lanes_hint, CALL);
#undef CALL
    }
    count_launch();
    return launch_status();
}
