// iwpp_wshed.cu — marker-controlled watershed by flooding as an IWPP propagation on the
// persistent tile engine (include/iwpp.h, iwpp_watershed).
//
// Every pixel carries a pair packed as (level << 16) | label, 0xFFFFFFFF while unreached.
// Markers are fixed at (gradient, label). A neighbour q offers pixel p the pair
// (max(level(q), gradient(p)), label(q)) — in the packing, max(v_q, gradient(p) << 16 |
// label(q)) — and p keeps the smaller of its own pair and every offer. One CTA settles a
// 64 x 64 tile held in shared memory with its gradient as eight 8-row strips
// (iwpp_smemtile.cuh); a halo pixel that the tile's border would improve marks its tile for a
// visit. The levels reached are unique (the minimax flooding level); which label wins where several
// reach a pixel at its level depends on the order of work, as in any flooding watershed.
//
// A row step weighs ~60 instructions (10 offers of three per lane); what bounds the drain is the
// number of row steps, the latency of one and the warps there are to overlap them. Whole calls with levels,
// 8-connectivity, tiles of one warp's registers (254 of them, 8 warps per SM, every row in every pass)
// and now: 2048^2 u16 gradient, 500 markers 1.65 and 1.12 ms, 4096^2 u16, a marker per 4000 pixels
// 4.50 and 2.96, 200^2 u8, two markers 0.230 and 0.197.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/iwpp.h"
#include "iwpp_engine.cuh"
#include "iwpp_host.h"
#include "iwpp_smemtile.cuh"

namespace iwpp {
namespace {

constexpr uint32_t kUnreached = 0xFFFFFFFFu;
constexpr int WTH = kSmStrip, WTW = kSmSide, WSW = kSmWarps, WCH = kSmSide;   // strip rows, tile columns, strips, rows

// The offer of pair v (at a neighbour) to a pixel whose gradient is g (already << 16).
__device__ __forceinline__ uint32_t offer_ws(uint32_t v, uint32_t g16) { return max(v, g16 | (v & 0xFFFFu)); }

struct WsArgs {
    const uint32_t *markers;
    const void *grad;
    int u16;
};

__device__ __forceinline__ bool inside(const ImageView &im, int y, int x) {
    return y >= 0 && y < im.H && x >= 0 && x < im.W;
}
__device__ __forceinline__ size_t clamp_e(const ImageView &im, int y, int x) {
    return (size_t)min(max(y, 0), im.H - 1) * im.W + min(max(x, 0), im.W - 1);
}
__device__ __forceinline__ uint32_t ld_grad(const ImageView &im, const WsArgs &w, int y, int x) {
    const size_t e = clamp_e(im, y, x);
    return w.u16 ? (uint32_t)reinterpret_cast<const uint16_t *>(w.grad)[e]
                 : (uint32_t)reinterpret_cast<const uint8_t *>(w.grad)[e];
}

struct WsOp {
    using Px = uint32_t;   // (level << 16) | label
    struct Aux {
        uint32_t g[kSmSide][kSmSide / 2];    // gradient pairs of the tile (even low, odd high)
        uint32_t fixed[kSmSide][2];          // per row: lanes whose even / odd pixel is fixed (a marker, or outside)
        uint32_t hg[4][kSmSide + 2];         // the halo's gradient << 16 per side (all ones outside the image)
    };
    struct RowAux {
        uint32_t g, fe, fo;   // the lane's gradient pair; which lanes' pixels are fixed
    };
    using Ctx = WsArgs;
    static __device__ __forceinline__ RowAux row_aux(const Aux &x, int r, int lane) {
        return RowAux{x.g[r][lane], x.fixed[r][0], x.fixed[r][1]};
    }
    static __device__ __forceinline__ Px none() { return kUnreached; }
    static __device__ __forceinline__ Px load(const ImageView &im, size_t e) {
        return __ldcg(reinterpret_cast<const uint32_t *>(im.J) + e);
    }
    static __device__ __forceinline__ void store(const ImageView &im, size_t e, Px v) {
        __stcg(reinterpret_cast<uint32_t *>(im.J) + e, v);
    }
    static __device__ __forceinline__ uint32_t halo_aux(const Aux &x, int side, int i) { return x.hg[side][i + 1]; }
    static __device__ __forceinline__ uint32_t halo_g(const ImageView &im, const Ctx &c, int y, int x) {
        const uint32_t g = ld_grad(im, c, y, x);
        return inside(im, y, x) ? g << 16 : 0xFFFFFFFFu;   // an offer there is never an improvement
    }

    static __device__ void load_aux(Aux &x, const ImageView &im, const Ctx &c, int y0, int x0, int w, int lane) {
        const int xe = x0 + 2 * lane;
#pragma unroll 8
        for (int k = 0; k < kSmStrip; k++) {
            const int r = kSmStrip * w + k, y = y0 + r;
            const uint32_t ge = ld_grad(im, c, y, xe), go = ld_grad(im, c, y, xe + 1);
            const bool me = c.markers[clamp_e(im, y, xe)] != 0, mo = c.markers[clamp_e(im, y, xe + 1)] != 0;
            x.g[r][lane] = ge | (go << 16);
            const uint32_t fe = __ballot_sync(0xffffffffu, me || !inside(im, y, xe));
            const uint32_t fo = __ballot_sync(0xffffffffu, mo || !inside(im, y, xe + 1));
            if (lane == 0) {
                x.fixed[r][0] = fe;
                x.fixed[r][1] = fo;
            }
        }
        if (lane < 2 * kSmStrip) {   // side halo: this strip's rows on both sides
            const int r = kSmStrip * w + lane % kSmStrip, right = lane / kSmStrip % 2;
            x.hg[right ? kRight : kLeft][r + 1] = halo_g(im, c, y0 + r, right ? x0 + kSmSide : x0 - 1);
        }
        if (w == 0 || w == kSmWarps - 1) {
            const int side = w == 0 ? kTop : kBottom, y = w == 0 ? y0 - 1 : y0 + kSmSide;
            for (int i = lane; i < kSmSide + 2; i += 32) x.hg[side][i] = halo_g(im, c, y, x0 + i - 1);
        }
    }

    template <int CONN>
    static __device__ __forceinline__ bool row(const Px (&q)[4], const Px (&p)[4], const RowAux &x, int lane, Px &e,
                                               Px &o) {
        const uint32_t ge = x.g << 16, go = x.g & 0xFFFF0000u;
        // (the offers of this row first, those of the row just written last: the shorter chain)
        uint32_t v = __vimin3_u32(q[1], offer_ws(q[0], ge), offer_ws(q[2], ge));
        uint32_t u = __vimin3_u32(q[2], offer_ws(q[3], go), offer_ws(p[2], go));
        if (CONN == 8) {
            v = min(v, __vimin3_u32(offer_ws(p[0], ge), offer_ws(p[1], ge), offer_ws(p[2], ge)));
            u = __vimin3_u32(u, offer_ws(p[1], go), offer_ws(p[3], go));
        } else {
            v = min(v, offer_ws(p[1], ge));
        }
        e = (x.fe >> lane) & 1u ? q[1] : v;
        o = (x.fo >> lane) & 1u ? q[2] : min(u, offer_ws(e, go));
        return e != q[1] || o != q[2];
    }
    static __device__ __forceinline__ bool changes(Px h, uint32_t g16, const Px (&q)[3], int n) {
        uint32_t v = offer_ws(q[0], g16);
        if (n > 1) v = __vimin3_u32(v, offer_ws(q[1], g16), offer_ws(q[2], g16));
        return v < h;
    }
    static __device__ __forceinline__ bool changes_own(Px v, const Aux &x, const Ctx &, int r, int c, const Px (&q)[3],
                                                       int n) {
        if ((x.fixed[r][c & 1] >> (c >> 1)) & 1u) return false;
        const uint32_t gp = x.g[r][c >> 1];
        return changes(v, (c & 1) ? gp & 0xFFFF0000u : gp << 16, q, n);
    }
};

// Initialisation, one warp per 8 x 64 strip: markers take (gradient, label), everything else
// is unreached; the CTA tile of every strip holding a marker is queued. Labels above 65534
// stop the call with IWPP_ERR_ARG.
__global__ void __launch_bounds__(256) ws_init_kernel(EngineArgs a, WsArgs w, uint32_t nstrips) {
    const ImageView &im = a.img0;
    const int lane = threadIdx.x & 31;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    uint32_t *V = reinterpret_cast<uint32_t *>(im.J);
    for (uint32_t u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < nstrips; u += nw) {
        const int uy = (int)(u / im.tiles_x), ux = (int)(u % im.tiles_x);
        const int y0 = uy * WTH, x0 = ux * WTW;
        bool any = false, bad = false;
        for (int r = 0; r < WTH; r++) {
            const int y = y0 + r;
            if (y >= im.H) break;
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int x = x0 + 2 * lane + q;
                if (x >= im.W) continue;
                const size_t e = (size_t)y * im.W + x;
                const uint32_t m = w.markers[e];
                const uint32_t g = w.u16 ? reinterpret_cast<const uint16_t *>(w.grad)[e]
                                         : reinterpret_cast<const uint8_t *>(w.grad)[e];
                bad |= m > 65534u;
                any |= m != 0;
                V[e] = m ? (g << 16) | m : kUnreached;
            }
        }
        any = __any_sync(0xffffffffu, any);
        bad = __any_sync(0xffffffffu, bad);
        __threadfence();
        if (lane == 0 && bad) set_status(a.hdr, kErrArg);
        if (lane == 0 && any) notify_tile(a, (uint32_t)((uy / WSW) * im.tiles_x + ux));
    }
}

#ifndef IWPP_WS_MINB
#define IWPP_WS_MINB 3   // CTAs (of 8 warps) per SM: 80 registers; 4 (64) were 8 % faster on 4096^2 and 10 % slower on 2048^2 before rows became runs
#endif
template <int CONN>
__global__ void __launch_bounds__(kSmThreads, IWPP_WS_MINB) ws_drain_kernel(EngineArgs a, WsArgs wa) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    sm_drain<WsOp, CONN>(a, wa, *reinterpret_cast<SmemTile<WsOp> *>(smem_raw));
}

// labels in place (0 where unreached), levels optionally (-1 where unreached)
__global__ void ws_finish_kernel(uint32_t *V, int32_t *levels, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const uint32_t v = V[i];
        if (levels) levels[i] = v == kUnreached ? -1 : (int32_t)(v >> 16);
        V[i] = v == kUnreached ? 0u : (v & 0xFFFFu);
    }
}

struct WsLayout {
    size_t state, queue, total;
    uint32_t ntiles, nstrips;   // 64 x 64 CTA tiles; 8 x 64 strips
    int tiles_x, tiles_y;
};

bool ws_layout(int64_t H, int64_t W, WsLayout &L) {
    if (H < 1 || W < 1 || H >= (1ll << 31) || W >= (1ll << 31) || (uint64_t)H * (uint64_t)W >= (1ull << 40))
        return false;
    const uint64_t tx = (uint64_t)((W + WTW - 1) / WTW), ty = (uint64_t)((H + WCH - 1) / WCH);
    const uint64_t sy = (uint64_t)((H + WTH - 1) / WTH);
    if (tx * sy >= (1ull << 31)) return false;
    L.tiles_x = (int)tx;
    L.tiles_y = (int)ty;
    L.ntiles = (uint32_t)(tx * ty);
    L.nstrips = (uint32_t)(tx * sy);
    L.state = 256;
    L.queue = L.state + align256((size_t)L.ntiles * 4);
    L.total = L.queue + align256((size_t)L.ntiles * 4);
    return true;
}

}  // namespace
}  // namespace iwpp

extern "C" size_t iwpp_watershed_workspace_bytes(int64_t H, int64_t W) {
    iwpp::WsLayout L;
    return iwpp::ws_layout(H, W, L) ? L.total : 0;
}

extern "C" int iwpp_watershed(const uint32_t *markers, const void *gradient, int dtype, uint32_t *labels_out,
                              int32_t *levels_out, int64_t H, int64_t W, int connectivity, void *workspace,
                              size_t ws_bytes, void *stream) {
    using namespace iwpp;
    if (!markers || !gradient || !labels_out) return IWPP_ERR_ARG;
    if (connectivity != 4 && connectivity != 8) return IWPP_ERR_ARG;
    if (dtype != IWPP_U8 && dtype != IWPP_U16) return IWPP_ERR_ARG;
    if (((uintptr_t)labels_out & 3) || ((uintptr_t)markers & 3) || (levels_out && ((uintptr_t)levels_out & 3)))
        return IWPP_ERR_ARG;
    WsLayout L;
    if (!ws_layout(H, W, L)) return IWPP_ERR_ARG;
    if (!workspace || ((uintptr_t)workspace & 255)) return IWPP_ERR_WORKSPACE;
    if (ws_bytes < L.total) return IWPP_ERR_WORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t *base = static_cast<uint8_t *>(workspace);
    EngineArgs a = {};
    a.img0.J = reinterpret_cast<uint8_t *>(labels_out);
    a.img0.I = static_cast<const uint8_t *>(gradient);
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
    WsArgs w;
    w.markers = markers;
    w.grad = gradient;
    w.u16 = dtype == IWPP_U16;
    if (cudaMemsetAsync(base, 0, L.queue + (size_t)L.ntiles * 4, s) != cudaSuccess) return IWPP_ERR_CUDA;
    const int sms = device_sm_count();
    if (sms <= 0) return IWPP_ERR_CUDA;
    uint32_t ig = (L.nstrips + 7) / 8;
    if (ig > (uint32_t)sms * 8) ig = (uint32_t)sms * 8;
    ws_init_kernel<<<ig, 256, 0, s>>>(a, w, L.nstrips);
    const size_t smem = sizeof(SmemTile<WsOp>);
    void (*drain)(EngineArgs, WsArgs) = connectivity == 8 ? ws_drain_kernel<8> : ws_drain_kernel<4>;
    int bps = 0;
    if (cudaFuncSetAttribute((const void *)drain, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared) != cudaSuccess)
        return IWPP_ERR_CUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, drain, kSmThreads, smem) != cudaSuccess || bps < 1)
        return IWPP_ERR_CUDA;
    long long g = (long long)bps * sms;
    if (g > (long long)L.ntiles) g = L.ntiles;   // one CTA per tile
    drain<<<(int)g, kSmThreads, smem, s>>>(a, w);
    const size_t n = (size_t)H * (size_t)W;
    ws_finish_kernel<<<sms * 8, 256, 0, s>>>(labels_out, levels_out, n);
    return cudaGetLastError() == cudaSuccess ? IWPP_OK : IWPP_ERR_CUDA;
}
