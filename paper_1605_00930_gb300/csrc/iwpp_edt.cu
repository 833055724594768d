// iwpp_edt.cu — Euclidean distance transform by Voronoi-site propagation (Sec. 3.2,
// Algorithm 8) on the persistent tile engine (include/iwpp.h, iwpp_edt).
//
// Every pixel carries a site: the background pixel it is nearest to among those its
// neighbours have offered, packed as (y << 16) | x, or kNoSite. Background pixels are
// their own sites. A warp holds a 16 x 64 tile with its halo in shared memory and repeats down /
// up Gauss-Seidel passes in which every pixel takes a neighbour's site if that site is
// strictly closer to it (the propagation step of Algorithm 8), until nothing changes: then
// no neighbour offers any pixel of the tile a closer site. A halo pixel that one of the tile's
// sites would bring strictly closer marks its tile for a visit, as in the reconstruction.
// Distances are squared Euclidean, exact in 32-bit integers for sides below 32768.
//
// Large images are bound by how many row steps are run and by how well their instructions are
// fetched and overlapped, small ones (fewer tiles than the 4864 warps of a full grid) and long chains of tiles by the
// latency of a row step and of a visit's loads and stores. The tile lies in shared memory, not in
// registers, so that the passes are loops over a row index: one row step per direction in the code
// instead of 2 x 16 (whose fetches were the largest stall), 32 warps fit an SM
// instead of 8, and rows without foreground, or whose neighbours have not changed, are skipped by
// bit masks. For the latency, rows that follow one another are a run (edt_pass), a row step takes minima
// of three (edt_step), and a visit's loads and stores go out together. The distances are written
// with the sites. Whole calls with distances, microseconds: register tiles of 220 registers and a
// distance pass / shared tiles with each row through shared memory and ten offers in turn / now:
//   tissue (10 % foreground), 8-connectivity: 4096^2 965 / 266 / 256, 512^2 155 / 80 / 68, 200^2 71 / 45 / 37;
//   4-connectivity: 4096^2 624 / 414 / 362, 2048^2 264 / 259 / 230, 750^2 187 / 213 / 143, 512^2 133 / 145 / 102;
//   one background pixel, 4-connectivity (a chain of tiles): 1001 x 1003 1184 / 1537 / 1061, 512^2
//   630 / 824 / 553, 4096 x 202 1938 / 2559 / 1822.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/iwpp.h"
#include "iwpp_engine.cuh"
#include "iwpp_host.h"

namespace iwpp {
namespace {

constexpr uint32_t kNoSite = 0xFFFFFFFFu;
constexpr int ETH = 16, ETW = 64;   // tile rows, columns

__device__ __forceinline__ uint32_t site_d2(int y, int x, uint32_t s) {
    // unsigned arithmetic: exact for real sites (< 2^31), wraps harmlessly for kNoSite
    const uint32_t dy = (uint32_t)(y - (int)(s >> 16)), dx = (uint32_t)(x - (int)(s & 0xFFFFu));
    return s == kNoSite ? 0xFFFFFFFFu : dy * dy + dx * dx;
}
// A warp's tile with its one-pixel halo: row y0 + r at index r + 1, column x0 + c at c + 1. The pair
// of columns 2c - 1, 2c of a row is 8-byte aligned: lane c reads its two pixels and
// both their horizontal neighbours in two 64-bit accesses.
constexpr int EPW = ETW + 4;
struct EdtSmem {
    uint32_t s[ETH + 2][EPW];
};
constexpr size_t kEdtSmemPerWarp = (sizeof(EdtSmem) + 15) & ~(size_t)15;

__device__ __forceinline__ uint32_t ld_site(const ImageView &im, int y, int x) {
    const bool in = y >= 0 && y < im.H && x >= 0 && x < im.W;
    const uint32_t *S = reinterpret_cast<const uint32_t *>(im.J);
    const uint32_t v = __ldcg(S + (size_t)min(max(y, 0), im.H - 1) * im.W + min(max(x, 0), im.W - 1));
    return in ? v : kNoSite;
}

// The rows of work left (bit r: row r): n from the row above, s from the row below, h from
// the row itself and the side halo. A down pass settles n, an up pass s, either h when it
// changes nothing.
struct EdtWork {
    uint32_t n, s, h;
};
constexpr uint32_t kRowBits = (1u << ETH) - 1u;

// Loads the tile and its halo; returns the rows that hold a foreground pixel (only those can
// change: a background pixel is its own site). In two halves: all 36 loads of a lane at once do not
// fit 64 registers (80 bytes of spills against 40; one background pixel in 512^2 266 us against 248).
__device__ uint32_t edt_load(const ImageView &im, EdtSmem &t, int y0, int x0, int lane) {
    uint32_t fg = 0;
    const uint32_t hl = ld_site(im, y0 + lane - 1, x0 - 1), hr = ld_site(im, y0 + lane - 1, x0 + ETW);
#pragma unroll
    for (int h = 0; h < 2; h++) {
        constexpr int N = (ETH + 2) / 2;
        uint32_t v0[N], v1[N];
#pragma unroll
        for (int k = 0; k < N; k++) {
            v0[k] = ld_site(im, y0 + h * N + k - 1, x0 + lane);
            v1[k] = ld_site(im, y0 + h * N + k - 1, x0 + 32 + lane);
        }
#pragma unroll
        for (int k = 0; k < N; k++) {
            const int r = h * N + k;
            t.s[r][lane + 1] = v0[k];
            t.s[r][lane + 33] = v1[k];
            if (r >= 1 && r <= ETH) {
                const int y = y0 + r - 1;
                const uint32_t self = ((uint32_t)y << 16) | (uint32_t)(x0 + lane);
                const bool f = y < im.H && ((x0 + lane < im.W && v0[k] != self) || (x0 + 32 + lane < im.W && v1[k] != self + 32u));
                fg |= (uint32_t)f << (r - 1);
            }
        }
    }
    if (lane < ETH + 2) {
        t.s[lane][0] = hl;
        t.s[lane][ETW + 1] = hr;
    }
    __syncwarp();
    return __reduce_or_sync(0xffffffffu, fg);
}

// The halo again; adds the rows that its changes may change to the work.
__device__ void edt_reload_halo(const ImageView &im, EdtSmem &t, int y0, int x0, EdtWork &w, int lane) {
    const uint32_t t0 = ld_site(im, y0 - 1, x0 + lane), t1 = ld_site(im, y0 - 1, x0 + 32 + lane);
    const uint32_t b0 = ld_site(im, y0 + ETH, x0 + lane), b1 = ld_site(im, y0 + ETH, x0 + 32 + lane);
    const uint32_t hl = ld_site(im, y0 + lane - 1, x0 - 1), hr = ld_site(im, y0 + lane - 1, x0 + ETW);
    if (__any_sync(0xffffffffu, t.s[0][lane + 1] != t0 || t.s[0][lane + 33] != t1)) w.n |= 1u;
    if (__any_sync(0xffffffffu, t.s[ETH + 1][lane + 1] != b0 || t.s[ETH + 1][lane + 33] != b1)) w.s |= 1u << (ETH - 1);
    t.s[0][lane + 1] = t0;
    t.s[0][lane + 33] = t1;
    t.s[ETH + 1][lane + 1] = b0;
    t.s[ETH + 1][lane + 33] = b1;
    bool d = false;
    if (lane < ETH + 2) {
        d = t.s[lane][0] != hl || t.s[lane][ETW + 1] != hr;
        t.s[lane][0] = hl;
        t.s[lane][ETW + 1] = hr;
    }
    const uint32_t rows = __ballot_sync(0xffffffffu, d);   // bit r + 1: the halo beside row r changed
    const uint32_t near = (rows | (rows >> 1) | (rows >> 2)) & kRowBits;   // rows beside and next to it
    w.h |= near;
    w.n |= near;
    w.s |= near;
    __syncwarp();
}

__device__ __forceinline__ void ld4(const uint32_t *p, uint32_t (&q)[4]) {
    const uint2 a = *reinterpret_cast<const uint2 *>(p), b = *reinterpret_cast<const uint2 *>(p + 2);
    q[0] = a.x; q[1] = a.y; q[2] = b.x; q[3] = b.y;
}
// Squared distances of site s to (y, x) and (y, x + 1): (dx + 1)^2 = dx^2 + 2 dx + 1.
__device__ __forceinline__ void site_d2_pair(int y, int x, uint32_t s, uint32_t &d0, uint32_t &d1) {
    const uint32_t dy = (uint32_t)(y - (int)(s >> 16)), dx = (uint32_t)(x - (int)(s & 0xFFFFu)), d = dy * dy + dx * dx;
    d0 = s == kNoSite ? 0xFFFFFFFFu : d;
    d1 = s == kNoSite ? 0xFFFFFFFFu : d + 2u * dx + 1u;
}
// The first of three sites at the smallest of their distances, and that distance.
__device__ __forceinline__ void nearest3(uint32_t s0, uint32_t s1, uint32_t s2, uint32_t d0, uint32_t d1, uint32_t d2,
                                         uint32_t &s, uint32_t &d) {
    d = __vimin3_u32(d0, d1, d2);
    s = d0 == d ? s0 : (d1 == d ? s1 : s2);
}

// A row step: the pixels at columns xe and xe + 1 (sites q[1], q[2]) from their row's sites q and the
// previous row's p, both of columns xe - 1 .. xe + 2. Own sites stay unless another is strictly
// closer. What waits longest, the previous row's sites and then the even pixel's new one, is weighed
// last: 3-way minima of distances and their sites, instead of ten offers one after the other.
template <int CONN>
__device__ __forceinline__ bool edt_step(const uint32_t (&q)[4], const uint32_t (&p)[4], int y, int xe, bool ve, bool vo,
                                         uint32_t &e, uint32_t &o) {
    uint32_t dq2, eq2, dp1, ep1, dp2, ep2;   // d..: to the even pixel, e..: to the odd one
    site_d2_pair(y, xe, q[2], dq2, eq2);
    site_d2_pair(y, xe, p[1], dp1, ep1);
    site_d2_pair(y, xe, p[2], dp2, ep2);
    uint32_t sv, dv, su, du, t, dt;
    nearest3(q[1], q[0], q[2], site_d2(y, xe, q[1]), site_d2(y, xe, q[0]), dq2, sv, dv);
    const uint32_t eq3 = site_d2(y, xe + 1, q[3]);
    if (CONN == 8) {
        nearest3(p[1], p[0], p[2], dp1, site_d2(y, xe, p[0]), dp2, t, dt);
        sv = dt < dv ? t : sv;
        const uint32_t ep3 = site_d2(y, xe + 1, p[3]);
        nearest3(p[2], p[1], p[3], ep2, ep1, ep3, su, du);
        su = eq3 <= du ? q[3] : su;
        du = min(eq3, du);
    } else {
        sv = dp1 < dv ? p[1] : sv;
        su = eq3 <= ep2 ? q[3] : p[2];
        du = min(eq3, ep2);
    }
    e = ve ? sv : kNoSite;
    // (of equally near sites the own one, then the even pixel's, then the others)
    const uint32_t de = site_d2(y, xe + 1, e);
    o = eq2 <= de && eq2 <= du ? q[2] : (de <= du ? e : su);
    if (!vo) o = kNoSite;
    return e != q[1] || o != q[2];
}

// One pass over the rows with work, in the order DIR (+1 down, -1 up). Rows that follow one another are
// a run: the next row's sites are loaded ahead and the previous one's stay in registers (its
// neighbour columns by shuffles beside the vote), so that a row does not wait for the one before to
// pass through shared memory. Adds the rows that changed to `rows`.
template <int CONN, int DIR>
__device__ __forceinline__ void edt_pass(EdtSmem &t, EdtWork &w, uint32_t fg, int y0, int xe, bool ve, bool vo,
                                         uint32_t &rows, int lane) {
    uint32_t &v = DIR > 0 ? w.n : w.s, &u = DIR > 0 ? w.s : w.n;
    for (uint32_t left = kRowBits;;) {
        const uint32_t m = (v | w.h) & fg & left;
        if (m == 0) break;
        int r = DIR > 0 ? __ffs(m) - 1 : 31 - __clz(m);
        uint32_t bit = 1u << r, q[4], p[4];
        __syncwarp();   // rows written before are read by other lanes
        ld4(&t.s[r + 1][2 * lane], q);
        ld4(&t.s[r + 1 - DIR][2 * lane], p);
        for (;;) {
            uint32_t *row = &t.s[r + 1][2 * lane], nx[4], e, o;
            ld4(&t.s[r + 1 + DIR][2 * lane], nx);
            const bool ch = edt_step<CONN>(q, p, y0 + r, xe, ve, vo, e, o);
            if (CONN == 8) {
                p[0] = __shfl_up_sync(0xffffffffu, o, 1);
                p[3] = __shfl_down_sync(0xffffffffu, e, 1);
                if (lane == 0) p[0] = q[0];
                if (lane == 31) p[3] = q[3];
            }
            p[1] = e;
            p[2] = o;
            const bool any = __any_sync(0xffffffffu, ch);
            __syncwarp();   // every lane has read the row
            if (ch) {
                row[1] = e;
                row[2] = o;
            }
            const uint32_t next = DIR > 0 ? bit << 1 : bit >> 1, prev = DIR > 0 ? bit >> 1 : bit << 1;
            v &= ~bit;
            w.h &= ~bit;
            if (any) {
                rows |= bit;
                w.h |= bit;
                v |= next;
                u |= prev;
            }
            left = DIR > 0 ? ~(next - 1u) : bit - 1u;
            if (((v | w.h) & fg & next) == 0) break;   // (fg holds rows of the tile only)
            r += DIR;
            bit = next;
#pragma unroll
            for (int i = 0; i < 4; i++) q[i] = nx[i];
        }
    }
}

// Passes until the tile is settled; returns the rows that changed. Rows are taken in the order
// of full down / up passes, less those with nothing to do.
template <int CONN>
__device__ uint32_t edt_settle(EdtSmem &t, EdtWork &w, uint32_t fg, int y0, int x0, int W, uint32_t &passes, int lane) {
    const int xe = x0 + 2 * lane;
    const bool ve = xe < W, vo = xe + 1 < W;
    uint32_t rows = 0;
    while ((w.n | w.s | w.h) & fg) {
        edt_pass<CONN, 1>(t, w, fg, y0, xe, ve, vo, rows, lane);
        edt_pass<CONN, -1>(t, w, fg, y0, xe, ve, vo, rows, lane);
        passes += 2;
    }
    __syncwarp();
    return rows;
}

// The neighbours one of whose halo pixels a site of the tile would bring strictly closer:
// bit (dy + 1) * 3 + dx + 1.
template <int CONN>
__device__ uint32_t edt_notify_mask(const EdtSmem &t, int y0, int x0, int lane) {
    // halo rows: candidates from the tile's first / last row (the tile's own columns only)
    uint32_t mask = 0;
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const int rt = e ? ETH : 1, rh = e ? ETH + 1 : 0, y = y0 + rh - 1;
        bool hit = false;
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int c = 1 + lane + 32 * q, x = x0 + lane + 32 * q;
            const uint32_t h = t.s[rh][c], d0 = site_d2(y, x, h);
            uint32_t d = site_d2(y, x, t.s[rt][c]);
            if (CONN == 8) {
                if (c > 1) d = min(d, site_d2(y, x, t.s[rt][c - 1]));
                if (c < ETW) d = min(d, site_d2(y, x, t.s[rt][c + 1]));
            }
            hit |= d < d0;
        }
        if (__any_sync(0xffffffffu, hit)) mask |= e ? 128u : 2u;
    }
    // halo columns: lane -> side (lane / 16) and row (lane % 16)
    {
        const int side = lane >> 4, r = lane & 15, y = y0 + r, x = side ? x0 + ETW : x0 - 1;
        const int ct = side ? ETW : 1, ch = side ? ETW + 1 : 0;
        uint32_t d = site_d2(y, x, t.s[r + 1][ct]);
        if (CONN == 8) {
            if (r > 0) d = min(d, site_d2(y, x, t.s[r][ct]));
            if (r < ETH - 1) d = min(d, site_d2(y, x, t.s[r + 2][ct]));
        }
        const uint32_t b = __ballot_sync(0xffffffffu, d < site_d2(y, x, t.s[r + 1][ch]));
        if (b & 0xFFFFu) mask |= 8u;
        if (b >> 16) mask |= 32u;
    }
    if (CONN == 8) {   // corners: lanes 0..3
        const int dn = (lane >> 1) & 1, rg = lane & 1;
        const int y = dn ? y0 + ETH : y0 - 1, x = rg ? x0 + ETW : x0 - 1;
        const bool hit = lane < 4 && site_d2(y, x, t.s[dn ? ETH : 1][rg ? ETW : 1]) <
                                         site_d2(y, x, t.s[dn ? ETH + 1 : 0][rg ? ETW + 1 : 0]);
        const uint32_t b = __ballot_sync(0xffffffffu, hit);
        mask |= (b & 1u) | ((b & 2u) << 1) | ((b & 4u) << 4) | ((b & 8u) << 5);
    }
    return mask;
}

// Stores the changed rows' sites and, when asked for (D), their squared distances.
__device__ void edt_store(const ImageView &im, uint32_t *D, const EdtSmem &t, int y0, int x0, uint32_t rows, int lane) {
    uint32_t *S = reinterpret_cast<uint32_t *>(im.J);
    const bool in0 = x0 + lane < im.W, in1 = x0 + 32 + lane < im.W;
#pragma unroll 4
    for (int r = 0; r < ETH; r++) {
        if (!((rows >> r) & 1u)) continue;   // (changed rows lie inside the image)
        const size_t e = (size_t)(y0 + r) * im.W + x0 + lane;
        const uint32_t v0 = t.s[r + 1][lane + 1], v1 = t.s[r + 1][lane + 33];
        if (in0) __stcg(S + e, v0);
        if (in1) __stcg(S + e + 32, v1);
        if (D) {
            if (in0) __stcg(D + e, site_d2(y0 + r, x0 + lane, v0));
            if (in1) __stcg(D + e + 32, site_d2(y0 + r, x0 + 32 + lane, v1));
        }
    }
}

template <int CONN>
__device__ void edt_visit(const EngineArgs &a, uint32_t *D, uint32_t t, EdtSmem &sm, VisitStats &st, int lane) {
    const ImageView &im = a.img0;
    const int ty = (int)(t / im.tiles_x), tx = (int)(t % im.tiles_x);
    const int y0 = ty * ETH, x0 = tx * ETW;
    const uint32_t fg = edt_load(im, sm, y0, x0, lane);
    uint32_t passes = 0;
    EdtWork w = {kRowBits, kRowBits, kRowBits};
    for (;;) {
        const uint32_t rows = edt_settle<CONN>(sm, w, fg, y0, x0, im.W, passes, lane);
        st.visits++;
        if (rows) {
            edt_store(im, D, sm, y0, x0, rows, lane);
            const uint32_t note = edt_notify_mask<CONN>(sm, y0, x0, lane);
            __threadfence();
            __syncwarp();
            if (lane < 9 && lane != 4 && ((note >> lane) & 1u)) {
                const int ny = ty + lane / 3 - 1, nx = tx + lane % 3 - 1;
                if (ny >= 0 && nx >= 0 && ny < im.tiles_y && nx < im.tiles_x)
                    notify_tile(a, (uint32_t)(ny * im.tiles_x + nx));
            }
        }
        if (!finish_tile(a, t, lane)) break;
        __syncwarp();
        edt_reload_halo(im, sm, y0, x0, w, lane);
    }
    st.waves += passes;
}

// Initialisation (Algorithm 8's first phase): background pixels are their own sites (distance
// 0), foreground pixels have none; every tile with a foreground pixel is queued (its first
// visit takes what its halo offers). VEC: four pixels per lane and step (the width a multiple
// of 4, the arrays aligned for it), 8 x 4 + 4 or 8 bytes of a row in flight per lane; else one.
template <bool VEC>
__global__ void __launch_bounds__(256) edt_init_kernel(EngineArgs a, uint32_t *D) {
    const ImageView &im = a.img0;
    const int lane = threadIdx.x & 31;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    uint32_t *S = reinterpret_cast<uint32_t *>(im.J);
    for (uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < a.ntiles; t += nw) {
        const int ty = (int)(t / im.tiles_x), tx = (int)(t % im.tiles_x);
        const int y0 = ty * ETH, x0 = tx * ETW;
        bool fg = false;
        if (VEC) {
            const int x = x0 + 4 * (lane & 15);
            uint32_t m[ETH / 2];
#pragma unroll
            for (int k = 0; k < ETH / 2; k++) {
                const int y = y0 + 2 * k + (lane >> 4);
                m[k] = y < im.H && x < im.W ? __ldg(reinterpret_cast<const uint32_t *>(im.I + (size_t)y * im.W + x)) : 0u;
            }
#pragma unroll
            for (int k = 0; k < ETH / 2; k++) {
                const int y = y0 + 2 * k + (lane >> 4);
                if (y >= im.H || x >= im.W) continue;
                fg |= m[k] != 0;
                const size_t e = (size_t)y * im.W + x;
                const uint32_t p = ((uint32_t)y << 16) | (uint32_t)x;
                const bool f0 = m[k] & 0xFFu, f1 = m[k] & 0xFF00u, f2 = m[k] & 0xFF0000u, f3 = m[k] >> 24;
                *reinterpret_cast<uint4 *>(S + e) =
                    make_uint4(f0 ? kNoSite : p, f1 ? kNoSite : p + 1, f2 ? kNoSite : p + 2, f3 ? kNoSite : p + 3);
                if (D)
                    *reinterpret_cast<uint4 *>(D + e) = make_uint4(f0 ? kNoSite : 0u, f1 ? kNoSite : 0u, f2 ? kNoSite : 0u,
                                                                   f3 ? kNoSite : 0u);
            }
        } else {
            for (int r = 0; r < ETH; r++) {
                const int y = y0 + r;
                if (y >= im.H) break;
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const int x = x0 + lane + 32 * q;
                    if (x >= im.W) continue;
                    const size_t e = (size_t)y * im.W + x;
                    const bool f = im.I[e] != 0;
                    fg |= f;
                    S[e] = f ? kNoSite : ((uint32_t)y << 16) | (uint32_t)x;
                    if (D) D[e] = f ? kNoSite : 0u;
                }
            }
        }
        fg = __any_sync(0xffffffffu, fg);
        if (lane == 0 && fg) notify_tile(a, t);   // (the drain is a later kernel: its tiles' sites are visible)
    }
}

// 8 CTAs (of 4 warps) per SM: 64 registers, 157 KB of shared memory.
template <int CONN>
__global__ void __launch_bounds__(kThreads, 8) edt_drain_kernel(EngineArgs a, uint32_t *D) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    EdtSmem &sm = *reinterpret_cast<EdtSmem *>(smem_raw + warp * kEdtSmemPerWarp);
    VisitStats st = {0, 0, 0, 0};
    unsigned long long idle = 0, busy = 0;
    for (;;) {
        bool first;
        const uint32_t t = acquire_tile(a, first, idle, lane);
        if (t == kDone) break;
        const unsigned long long b0 = globaltimer_ns();
        edt_visit<CONN>(a, D, t, sm, st, lane);
        busy += globaltimer_ns() - b0;
    }
    flush_stats(a, st, idle, busy, lane);
}

// The distances by themselves, from the final sites (which they may overwrite).
__global__ void edt_dist2_kernel(const uint32_t *S, uint32_t *D, int W, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        D[i] = site_d2((int)(i / W), (int)(i % W), S[i]);
}

// Workspace: header (256 B) | tile states | tile-queue ring.
struct EdtLayout {
    size_t state, queue, total;
    uint32_t ntiles;
    int tiles_x, tiles_y;
};

bool edt_layout(int64_t H, int64_t W, EdtLayout &L) {
    if (H < 1 || W < 1 || H > 32767 || W > 32767) return false;
    L.tiles_x = (int)((W + ETW - 1) / ETW);
    L.tiles_y = (int)((H + ETH - 1) / ETH);
    L.ntiles = (uint32_t)L.tiles_x * (uint32_t)L.tiles_y;
    L.state = 256;
    L.queue = L.state + align256((size_t)L.ntiles * 4);
    L.total = L.queue + align256((size_t)L.ntiles * 4);
    return true;
}

}  // namespace
}  // namespace iwpp

extern "C" size_t iwpp_edt_workspace_bytes(int64_t H, int64_t W) {
    iwpp::EdtLayout L;
    return iwpp::edt_layout(H, W, L) ? L.total : 0;
}

extern "C" int iwpp_edt(const void *mask, uint32_t *site_out, uint32_t *dist2_out, int64_t H, int64_t W,
                        int connectivity, void *workspace, size_t ws_bytes, void *stream) {
    using namespace iwpp;
    if (!mask || !site_out) return IWPP_ERR_ARG;
    if (connectivity != 4 && connectivity != 8) return IWPP_ERR_ARG;
    if (((uintptr_t)site_out & 3) || (dist2_out && ((uintptr_t)dist2_out & 3))) return IWPP_ERR_ARG;
    EdtLayout L;
    if (!edt_layout(H, W, L)) return IWPP_ERR_ARG;
    if (!workspace || ((uintptr_t)workspace & 255)) return IWPP_ERR_WORKSPACE;
    if (ws_bytes < L.total) return IWPP_ERR_WORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t *base = static_cast<uint8_t *>(workspace);
    EngineArgs a = {};
    a.img0.J = reinterpret_cast<uint8_t *>(site_out);
    a.img0.I = static_cast<const uint8_t *>(mask);
    a.img0.H = (int)H;
    a.img0.W = (int)W;
    a.img0.tiles_x = L.tiles_x;
    a.img0.tiles_y = L.tiles_y;
    a.hdr = reinterpret_cast<WsHeader *>(base);
    a.state = reinterpret_cast<uint32_t *>(base + L.state);
    a.queue = reinterpret_cast<uint32_t *>(base + L.queue);
    a.ntiles = L.ntiles;
    a.watchdog_ns = 10ll * 1000 * 1000 * 1000;
    a.nlevels = 1;
    if (cudaMemsetAsync(base, 0, L.queue + (size_t)L.ntiles * 4, s) != cudaSuccess) return IWPP_ERR_CUDA;
    const int sms = device_sm_count();
    if (sms <= 0) return IWPP_ERR_CUDA;
    // Distances that go where the sites or the mask are cannot be written with the sites: they follow
    // the drain (41 us at 4096^2).
    const size_t n = (size_t)H * (size_t)W;
    const auto shares = [&](const void *p, size_t bytes) {
        const uintptr_t d = (uintptr_t)dist2_out, q = (uintptr_t)p;
        return d < q + bytes && q < d + 4 * n;
    };
    uint32_t *const D = dist2_out && (shares(site_out, 4 * n) || shares(mask, n)) ? nullptr : dist2_out;
    const uint32_t warps_needed = L.ntiles;
    uint32_t ig = (warps_needed + 7) / 8;
    if (ig > (uint32_t)sms * 8) ig = (uint32_t)sms * 8;
    const bool vec = (W & 3) == 0 && ((uintptr_t)mask & 3) == 0 && ((uintptr_t)site_out & 15) == 0 &&
                     ((uintptr_t)D & 15) == 0;
    if (vec) edt_init_kernel<true><<<ig, 256, 0, s>>>(a, D);
    else edt_init_kernel<false><<<ig, 256, 0, s>>>(a, D);
    const size_t smem = kEdtSmemPerWarp * kWarpsPerCta;
    void (*drain)(EngineArgs, uint32_t *) = connectivity == 8 ? edt_drain_kernel<8> : edt_drain_kernel<4>;
    int bps = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, drain, kThreads, smem) != cudaSuccess || bps < 1)
        return IWPP_ERR_CUDA;
    long long g = (long long)bps * sms;
    const long long need = ((long long)L.ntiles + kWarpsPerCta - 1) / kWarpsPerCta;
    if (g > need) g = need;
    drain<<<(int)g, kThreads, smem, s>>>(a, D);
    if (D != dist2_out) edt_dist2_kernel<<<sms * 8, 256, 0, s>>>(site_out, dist2_out, (int)W, n);
    return cudaGetLastError() == cudaSuccess ? IWPP_OK : IWPP_ERR_CUDA;
}
