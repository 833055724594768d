// iwpp_skiz.cu — geodesic skeleton by influence zones (SKIZ) as an IWPP propagation on the
// persistent tile engine (include/iwpp.h, iwpp_skiz). SKIZ is one of the operators the
// paper names as future work for the pattern (Sec. 6).
//
// Every pixel carries a state (d, l): d the number of steps from the nearest marker found so
// far, l the packed pair (min label << 16) | (0xFFFF - max label) of the markers at that
// distance. A neighbour q offers p (d(q) + 1, l(q)); p takes an offer with a smaller d, and
// on an equal d merges the label sets — the per-half minimum of the packed pair (min of the
// smallest labels, max of the largest). That update is a join on a distributive lattice, so
// every order of work reaches the same fixed point: d = the geodesic distance to the
// nearest marker and the labels of all markers at that distance. Pixels outside the domain
// carry d = kBlocked and never change. One CTA settles a 64 x 64 tile held in shared memory as
// eight 8-row strips (iwpp_smemtile.cuh); a halo pixel that the tile's border would change marks
// its tile for a visit.
//
// A row step weighs ~70 instructions (10 candidates of two words each per lane); what bounds the
// drain is the number of row steps, the latency of one and the warps there are to overlap them.
// 4096^2 porous domain, 2000 markers, 8-connectivity, zones, distances and label pairs, whole call:
// 3.31 ms with the tile in registers (152 of them, 12 warps per SM, every row in every pass), 1.19 ms now.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/iwpp.h"
#include "iwpp_engine.cuh"
#include "iwpp_host.h"
#include "iwpp_smemtile.cuh"

namespace iwpp {
namespace {

constexpr uint32_t kUnr = 0xC0000000u;      // domain pixel not reached yet (real d < 2^31)
constexpr uint32_t kBlocked = 0xE0000000u;  // outside the domain (also outside the image)
constexpr uint32_t kNoLab = 0xFFFFFFFFu;
constexpr int STH = kSmStrip, STW = kSmSide, SKW = kSmWarps, SCH = kSmSide;   // strip rows, tile columns, strips, rows

struct St {
    uint32_t d, l;
};

__device__ __forceinline__ St unpack(unsigned long long v) { return St{(uint32_t)(v >> 32), (uint32_t)v}; }
__device__ __forceinline__ unsigned long long pack(St s) { return ((unsigned long long)s.d << 32) | s.l; }

// Accept the offer (m + 1, lc) at pixel s (unless s is outside the domain).
__device__ __forceinline__ St accept(St s, uint32_t m, uint32_t lc) {
    if (s.d == kBlocked) return s;
    const uint32_t o = m + 1;
    St r;
    r.l = o < s.d ? lc : (o == s.d ? __vminu2(s.l, lc) : s.l);
    r.d = min(s.d, o);
    return r;
}
__device__ __forceinline__ bool would_change(St h, uint32_t m, uint32_t lc) {
    const St r = accept(h, m, lc);
    return r.d != h.d || r.l != h.l;
}

// The join of n candidates (no step added): the smallest distance and, per half, the smallest
// label word among the candidates at that distance.
template <int N>
__device__ __forceinline__ void join(const unsigned long long (&q)[N], uint32_t &m, uint32_t &lc) {
    m = (uint32_t)(q[0] >> 32);
#pragma unroll
    for (int k = 1; k < N; k++) m = min(m, (uint32_t)(q[k] >> 32));
    lc = kNoLab;
#pragma unroll
    for (int k = 0; k < N; k++) lc = __vminu2(lc, (uint32_t)(q[k] >> 32) == m ? (uint32_t)q[k] : kNoLab);
}

struct SkOp {
    using Px = unsigned long long;   // (d << 32) | l
    struct Aux {};
    struct RowAux {};
    struct Ctx {};
    static __device__ __forceinline__ RowAux row_aux(const Aux &, int, int) { return RowAux{}; }
    static __device__ __forceinline__ Px none() { return pack(St{kBlocked, kNoLab}); }
    static __device__ __forceinline__ Px load(const ImageView &im, size_t e) {
        return __ldcg(reinterpret_cast<const Px *>(im.J) + e);
    }
    static __device__ __forceinline__ void store(const ImageView &im, size_t e, Px v) {
        __stcg(reinterpret_cast<Px *>(im.J) + e, v);
    }
    static __device__ __forceinline__ void load_aux(Aux &, const ImageView &, const Ctx &, int, int, int, int) {}
    static __device__ __forceinline__ uint32_t halo_aux(const Aux &, int, int) { return 0; }

    template <int CONN>
    static __device__ __forceinline__ bool row(const Px (&q)[4], const Px (&p)[4], const RowAux &, int, Px &e, Px &o) {
        uint32_t m, lc;
        if (CONN == 8) {
            const Px c[5] = {q[0], q[2], p[0], p[1], p[2]};
            join(c, m, lc);
        } else {
            const Px c[3] = {q[0], q[2], p[1]};
            join(c, m, lc);
        }
        e = pack(accept(unpack(q[1]), m, lc));
        if (CONN == 8) {
            const Px c[5] = {e, q[3], p[1], p[2], p[3]};
            join(c, m, lc);
        } else {
            const Px c[3] = {e, q[3], p[2]};
            join(c, m, lc);
        }
        o = pack(accept(unpack(q[2]), m, lc));
        return e != q[1] || o != q[2];
    }
    static __device__ __forceinline__ bool changes(Px h, uint32_t, const Px (&q)[3], int n) {
        const Px c[3] = {q[0], n > 1 ? q[1] : none(), n > 2 ? q[2] : none()};
        uint32_t m, lc;
        join(c, m, lc);
        return would_change(unpack(h), m, lc);
    }
    static __device__ __forceinline__ bool changes_own(Px v, const Aux &, const Ctx &, int, int, const Px (&q)[3], int n) {
        return changes(v, 0, q, n);
    }
};

// Initialisation, one warp per 8 x 64 strip: markers take (0, their label), other domain
// pixels are unreached, the rest blocked; the CTA tile of every strip holding a marker is
// queued. Labels above 65534 stop the call with IWPP_ERR_ARG.
__global__ void __launch_bounds__(256) sk_init_kernel(EngineArgs a, const uint32_t *markers, const uint8_t *mask,
                                                      uint32_t nstrips) {
    const ImageView &im = a.img0;
    const int lane = threadIdx.x & 31;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    unsigned long long *V = reinterpret_cast<unsigned long long *>(im.J);
    for (uint32_t u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < nstrips; u += nw) {
        const int uy = (int)(u / im.tiles_x), ux = (int)(u % im.tiles_x);
        const int y0 = uy * STH, x0 = ux * STW;
        bool any = false, bad = false;
        for (int r = 0; r < STH; r++) {
            const int y = y0 + r;
            if (y >= im.H) break;
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int x = x0 + 2 * lane + q;
                if (x >= im.W) continue;
                const size_t e = (size_t)y * im.W + x;
                const uint32_t m = markers[e];
                bad |= m > 65534u;
                any |= m != 0;
                St s;
                if (m) s = St{0u, (m << 16) | (0xFFFFu - m)};
                else s = St{mask[e] ? kUnr : kBlocked, kNoLab};
                V[e] = pack(s);
            }
        }
        any = __any_sync(0xffffffffu, any);
        bad = __any_sync(0xffffffffu, bad);
        __threadfence();
        if (lane == 0 && bad) set_status(a.hdr, kErrArg);
        if (lane == 0 && any) notify_tile(a, (uint32_t)((uy / SKW) * im.tiles_x + ux));
    }
}

#ifndef IWPP_SKIZ_MINB
#define IWPP_SKIZ_MINB 4   // CTAs (of 8 warps) per SM: 64 registers; 3 were 9 % slower on 4096^2 before rows became runs
#endif
template <int CONN>
__global__ void __launch_bounds__(kSmThreads, IWPP_SKIZ_MINB) sk_drain_kernel(EngineArgs a) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    sm_drain<SkOp, CONN>(a, SkOp::Ctx{}, *reinterpret_cast<SmemTile<SkOp> *>(smem_raw));
}

// zone (label where one label is nearest, else 0), optional distance (-1 where unreached)
// and optional label pair (min label << 16) | max label (0 where unreached)
__global__ void sk_finish_kernel(const unsigned long long *V, uint32_t *zone, int32_t *dist, uint32_t *lpair,
                                 size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const St s = unpack(V[i]);
        const bool reached = s.d < kUnr;
        const uint32_t lmin = s.l >> 16, lmax = 0xFFFFu - (s.l & 0xFFFFu);
        zone[i] = reached && lmin == lmax ? lmin : 0u;
        if (dist) dist[i] = reached ? (int32_t)s.d : -1;
        if (lpair) lpair[i] = reached ? (lmin << 16) | lmax : 0u;
    }
}

struct SkLayout {
    size_t state, queue, px, total;
    uint32_t ntiles, nstrips;   // 64 x 64 CTA tiles; 8 x 64 strips
    int tiles_x, tiles_y;
};

bool sk_layout(int64_t H, int64_t W, SkLayout &L) {
    if (H < 1 || W < 1 || H >= (1ll << 31) || W >= (1ll << 31) || (uint64_t)H * (uint64_t)W >= (1ull << 31))
        return false;
    const uint64_t tx = (uint64_t)((W + STW - 1) / STW), ty = (uint64_t)((H + SCH - 1) / SCH);
    L.tiles_x = (int)tx;
    L.tiles_y = (int)ty;
    L.ntiles = (uint32_t)(tx * ty);
    L.nstrips = (uint32_t)(tx * (uint64_t)((H + STH - 1) / STH));
    L.state = 256;
    L.queue = L.state + align256((size_t)L.ntiles * 4);
    L.px = L.queue + align256((size_t)L.ntiles * 4);
    L.total = L.px + align256((size_t)H * (size_t)W * 8);
    return true;
}

}  // namespace
}  // namespace iwpp

extern "C" size_t iwpp_skiz_workspace_bytes(int64_t H, int64_t W) {
    iwpp::SkLayout L;
    return iwpp::sk_layout(H, W, L) ? L.total : 0;
}

extern "C" int iwpp_skiz(const uint32_t *markers, const uint8_t *mask, uint32_t *zone_out, int32_t *dist_out,
                         uint32_t *lpair_out, int64_t H, int64_t W, int connectivity, void *workspace,
                         size_t ws_bytes, void *stream) {
    using namespace iwpp;
    if (!markers || !mask || !zone_out) return IWPP_ERR_ARG;
    if (connectivity != 4 && connectivity != 8) return IWPP_ERR_ARG;
    if (((uintptr_t)markers & 3) || ((uintptr_t)zone_out & 3) || (dist_out && ((uintptr_t)dist_out & 3)) ||
        (lpair_out && ((uintptr_t)lpair_out & 3)))
        return IWPP_ERR_ARG;
    SkLayout L;
    if (!sk_layout(H, W, L)) return IWPP_ERR_ARG;
    if (!workspace || ((uintptr_t)workspace & 255)) return IWPP_ERR_WORKSPACE;
    if (ws_bytes < L.total) return IWPP_ERR_WORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t *base = static_cast<uint8_t *>(workspace);
    EngineArgs a = {};
    a.img0.J = base + L.px;
    a.img0.I = mask;
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
    uint32_t ig = (L.nstrips + 7) / 8;
    if (ig > (uint32_t)sms * 8) ig = (uint32_t)sms * 8;
    sk_init_kernel<<<ig, 256, 0, s>>>(a, markers, mask, L.nstrips);
    const size_t smem = sizeof(SmemTile<SkOp>);
    void (*drain)(EngineArgs) = connectivity == 8 ? sk_drain_kernel<8> : sk_drain_kernel<4>;
    int bps = 0;
    if (cudaFuncSetAttribute((const void *)drain, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared) != cudaSuccess)
        return IWPP_ERR_CUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, drain, kSmThreads, smem) != cudaSuccess || bps < 1)
        return IWPP_ERR_CUDA;
    long long g = (long long)bps * sms;
    if (g > (long long)L.ntiles) g = L.ntiles;   // one CTA per tile
    drain<<<(int)g, kSmThreads, smem, s>>>(a);
    const size_t n = (size_t)H * (size_t)W;
    sk_finish_kernel<<<sms * 8, 256, 0, s>>>(reinterpret_cast<const unsigned long long *>(base + L.px), zone_out,
                                              dist_out, lpair_out, n);
    return cudaGetLastError() == cudaSuccess ? IWPP_OK : IWPP_ERR_CUDA;
}
