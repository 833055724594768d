// iwpp_scan.cuh — the scan of the cooperative solver's 64 x 64 tiles (sm_103a).
//
// The scan is the initialisation pass of Algorithm 7 reduced to what the persistent drain
// needs: per tile, whether the precondition J <= I holds and whether one step of the update
// (Eq. "recon") would raise one of its pixels, in which case the tile enters the queue. It
// reads every pixel once, so it is bound by HBM and by how many loads are in flight.
//
// One warp tests a strip of 16 rows x 64 columns at a time (a tile is four strips) as a 4 x 8
// grid of lane blocks: lane (lr, lc) = (lane / 8, lane % 8) holds rows 4 lr .. + 3 and columns
// 8 lc .. + 7, with the row above and below them. Rows are read in 8-pixel spans, one 64-bit
// (u8) or 128-bit (u16) load where the image's width keeps spans aligned, else 32-bit words
// joined by funnel shifts, and every load of the strip is issued before the first is used:
// one memory round trip per strip, 2-4 KB in flight per warp. (A scan that streamed a tile row
// by row through one warp, 2 pixels per lane and two rows ahead, took 33 round trips per tile:
// 512^2 u8 34 us against 8 now, 4096^2 u8 40 against 18, 16384^2 u8 482 against 195 (2.8 TB/s),
// 48 u8 + u16 images of 166 MB 245 against 153, 256 images with features 1.43 ms against 1.08.)
// Word k (k = 0..3) of a row packs the block's columns k and k + 4 as u16x2 in the dilation domain, so that horizontal
// neighbours are other words of the lane but for the block's edges (two shuffles per row). Learned batches
// also add up the tile's feature sums over its sampled rows (iwpp_feat.cuh): there a warp
// takes the tile's four strips in turn and writes its 16 features.
#pragma once
#include <type_traits>

#include "iwpp_feat.cuh"
#include "iwpp_regtile.cuh"

namespace iwpp {

// CTAs (of 4 warps) per SM: one pixel type 8 (64 registers, the u16 builds with
// 220-300 B of spills; 12 and 6 are slower, 4096^2 u8 18.1 us against 24.3 and 19.7), u8 + u16 6 (their variants spill at 64: 48 images 153 us against 161),
// with the feature sums 4 (256 images: 1.08 ms against 1.20 with 6 and 1.27 with 5).
#ifndef IWPP_SCAN_MINB
#define IWPP_SCAN_MINB 8
#endif
#ifndef IWPP_SCAN_ANY_MINB
#define IWPP_SCAN_ANY_MINB 6
#endif
#ifndef IWPP_SCAN_FEATS_MINB
#define IWPP_SCAN_FEATS_MINB 4
#endif

constexpr int kScanRows = 4;   // rows per lane block

// How an image's rows can be read at a strip: aligned 8-pixel spans (width a multiple of 8),
// or aligned 32-bit words (every other width of 8 or more). Images narrower than 8 pixels, and
// strips that reach (with their halo row) the image's last pixels when those do not fill a
// word, go pixel by pixel, so that nothing outside the buffers is touched.
enum ScanMode { kScanSpan, kScanWord, kScanPixel };
__device__ __forceinline__ ScanMode scan_mode(const ImageView &im, bool w16, int y0, int x0) {
    if ((im.W & 7) == 0) return kScanSpan;
    const bool last = y0 + kCoopStrip + 1 >= im.H && x0 + 64 + 3 >= im.W;
    const bool tail = (((((uint32_t)im.H & 3u) * ((uint32_t)im.W & 3u)) << (w16 ? 1 : 0)) & 3u) != 0;
    return im.W < 8 || (last && tail) ? kScanPixel : kScanWord;
}

// The raw words of pixels (y, x .. x + 7) at clamped addresses (what lies outside the image is
// masked by the caller): span u8 2 / u16 4 words; word u8 3 / u16 5, joined by scan_join.
template <bool W16, int M>
__device__ __forceinline__ void scan_issue(const ImageView &im, const uint8_t *p, int y, int x, uint32_t (&v)[5]) {
    const size_t row = (size_t)min(max(y, 0), im.H - 1) * (size_t)im.W;
    if (M == kScanSpan) {
        const size_t e = row + (size_t)min(x, im.W - 8);
        if (W16) {
            const uint4 u = __ldg(reinterpret_cast<const uint4 *>(p + 2 * e));
            v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
        } else {
            const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p + e));
            v[0] = u.x; v[1] = u.y;
        }
    } else if (M == kScanWord) {
        const size_t a = (row + (size_t)min(x, im.W - 1)) << (W16 ? 1 : 0), a4 = a & ~(size_t)3;
        const size_t last = ((((size_t)im.H * (size_t)im.W) << (W16 ? 1 : 0)) - 4) & ~(size_t)3;   // last whole word
#pragma unroll
        for (int i = 0; i < (W16 ? 5 : 3); i++) {
            const size_t o = a4 + 4 * i;
            v[i] = __ldg(reinterpret_cast<const uint32_t *>(p + (o < last ? o : last)));
        }
    } else {
        v[0] = v[1] = v[2] = v[3] = 0;
        for (int k = 0; k < 8; k++) {
            const size_t e = row + (size_t)min(x + k, im.W - 1);
            const uint32_t q = W16 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(p) + e) : (uint32_t)__ldg(p + e);
            const uint32_t s = q << (W16 ? 16 * (k & 1) : 8 * (k & 3));
            const int d = W16 ? k >> 1 : k >> 2;
            v[0] |= d == 0 ? s : 0u;
            v[1] |= d == 1 ? s : 0u;
            v[2] |= d == 2 ? s : 0u;
            v[3] |= d == 3 ? s : 0u;
        }
    }
}
// The issued words as words (k, k + 4) in the dilation domain, 0 outside the image.
template <bool W16, int M>
__device__ __forceinline__ void scan_unpack(const ImageView &im, int y, int x, const uint32_t (&cm)[4],
                                            const uint32_t (&t)[5], uint32_t (&o)[4]) {
    uint32_t v[4] = {t[0], t[1], t[2], t[3]};
    if (M == kScanWord) {
        const size_t a = ((size_t)min(max(y, 0), im.H - 1) * (size_t)im.W + (size_t)min(x, im.W - 1)) << (W16 ? 1 : 0);
        const uint32_t sh = 8u * (uint32_t)(a & 3);
#pragma unroll
        for (int i = 0; i < (W16 ? 4 : 2); i++) v[i] = __funnelshift_r(t[i], t[i + 1], sh);
    }
    if (W16) {
        o[0] = __byte_perm(v[0], v[2], 0x5410);
        o[1] = __byte_perm(v[0], v[2], 0x7632);
        o[2] = __byte_perm(v[1], v[3], 0x5410);
        o[3] = __byte_perm(v[1], v[3], 0x7632);
    } else {
        const uint32_t a = __byte_perm(v[0], v[1], 0x5410), b = __byte_perm(v[0], v[1], 0x7632);
        o[0] = __byte_perm(a, 0u, 0x4240);
        o[1] = __byte_perm(a, 0u, 0x4341);
        o[2] = __byte_perm(b, 0u, 0x4240);
        o[3] = __byte_perm(b, 0u, 0x4341);
    }
    const uint32_t f2 = im.flip | (im.flip << 16);
    const bool in = y >= 0 && y < im.H;
#pragma unroll
    for (int k = 0; k < 4; k++) o[k] = in ? (o[k] ^ f2) & cm[k] : 0u;
}

// One strip: rows y0 .. y0 + 15 (y0 < H), columns x0 .. x0 + 63. Sets `can` (a pixel can rise:
// min(I, max over its neighbourhood of J) != J) and `bad` (J > I somewhere) for this lane; FEATS:
// adds the lane's pixels to `fa`.
template <bool W16, int M, int CONN, bool FEATS>
__device__ __forceinline__ void scan_strip(const ImageView &im, int y0, int x0, int lane, bool &can, bool &bad,
                                           FeatAcc &fa) {
    constexpr int RB = kScanRows;
    const int lr = lane >> 3, lc = lane & 7;
    const int y = y0 + RB * lr, x = x0 + 8 * lc;
    uint32_t rj[RB + 2][5], ri[RB][5];
#pragma unroll
    for (int r = 0; r < RB + 2; r++) scan_issue<W16, M>(im, im.J, y + r - 1, x, rj[r]);
#pragma unroll
    for (int r = 0; r < RB; r++) scan_issue<W16, M>(im, im.I, y + r, x, ri[r]);
    // side halo: lanes lc == 0 read column x0 - 1, lanes lc == 7 column x0 + 64
    const int xs = lc == 0 ? x0 - 1 : x0 + 64;
    const bool xin = (lc == 0 && xs >= 0) || (lc == 7 && xs < im.W);
    uint32_t hs[RB + 2];
#pragma unroll
    for (int r = 0; r < RB + 2; r++) {
        const int yr = y + r - 1;
        hs[r] = 0;
        if (xin && yr >= 0 && yr < im.H) {
            const size_t e = (size_t)yr * (size_t)im.W + (size_t)xs;
            hs[r] = W16 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(im.J) + e) : (uint32_t)__ldg(im.J + e);
            hs[r] ^= im.flip;
        }
    }
    const int nv = im.W - x;   // pixels of the block's rows inside the image
    uint32_t cm[4];
#pragma unroll
    for (int k = 0; k < 4; k++) cm[k] = (k < nv ? 0xFFFFu : 0u) | (k + 4 < nv ? 0xFFFF0000u : 0u);
    uint32_t p[4], c[4], n[4];   // rows r - 1, r, r + 1 of J
    scan_unpack<W16, M>(im, y - 1, x, cm, rj[0], p);
    scan_unpack<W16, M>(im, y, x, cm, rj[1], c);
    uint32_t any = 0, nok = 0;
#pragma unroll
    for (int r = 0; r < RB; r++) {
        uint32_t i[4], v[4];
        scan_unpack<W16, M>(im, y + r + 1, x, cm, rj[r + 2], n);
        scan_unpack<W16, M>(im, y + r, x, cm, ri[r], i);
#pragma unroll
        for (int k = 0; k < 4; k++) v[k] = max3(p[k], c[k], n[k]);
        // left of word 0 and right of word 3: the adjacent lanes' edge columns or the side halo
        uint32_t l = __shfl_up_sync(0xffffffffu, CONN == 8 ? v[3] : c[3], 1);
        uint32_t q = __shfl_down_sync(0xffffffffu, CONN == 8 ? v[0] : c[0], 1);
        const uint32_t h = CONN == 8 ? max(hs[r], max(hs[r + 1], hs[r + 2])) : hs[r + 1];
        if (lc == 0) l = h << 16;
        if (lc == 7) q = h;
        uint32_t m[4];
        if (CONN == 8) {
            m[0] = max3(__byte_perm(l, v[3], 0x5432), v[0], v[1]);
            m[1] = max3(v[0], v[1], v[2]);
            m[2] = max3(v[1], v[2], v[3]);
            m[3] = max3(v[2], v[3], __byte_perm(v[0], q, 0x5432));
        } else {
            m[0] = max3(__byte_perm(l, c[3], 0x5432), v[0], c[1]);
            m[1] = max3(c[0], v[1], c[2]);
            m[2] = max3(c[1], v[2], c[3]);
            m[3] = max3(c[2], v[3], __byte_perm(c[0], q, 0x5432));
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            any |= min2(i[k], m[k]) ^ c[k];
            nok |= max2(c[k], i[k]) ^ i[k];
        }
        if (FEATS && r == 0) {   // the block's first row is a sampled row of the tile
            static_assert(RB == kFeatRowStep, "a lane block starts on a sampled row");
            uint32_t nx[4];
            scan_unpack<W16, M>(im, y + 1, x, cm, ri[1], nx);
            const bool down = y + 1 < im.H;
            const uint32_t w0 = __shfl_down_sync(0xffffffffu, i[0], 1);
            const int nc = min(max(nv, 0), 8);
            if (y < im.H) {
                fa.n += (uint32_t)nc;
                fa.h03 -= (uint32_t)(8 - nc);   // columns outside the image are counted in bin 0 below
                const uint32_t thr = 16u * ((W16 ? 0xFFFFu : 0xFFu) / 255u);
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const uint32_t iv = i[k], jv = c[k];
                    const uint32_t dv = max2(iv, jv) - jv;   // per half max(I - J, 0): no borrow
                    const uint32_t d8 = W16 ? (dv >> 8) & 0x00FF00FFu : dv;
                    const uint32_t bl = min(7u, 32u - (uint32_t)__clz(d8 & 0xFFFFu));   // bit length, 0 for 0
                    const uint32_t bh = min(7u, 32u - (uint32_t)__clz(d8 >> 16));
                    fa.h03 += (bl < 4 ? 1u << (8 * bl) : 0u) + (bh < 4 ? 1u << (8 * bh) : 0u);
                    fa.h47 += (bl >= 4 ? 1u << (8 * bl - 32) : 0u) + (bh >= 4 ? 1u << (8 * bh - 32) : 0u);
                    const uint32_t e = iv ^ jv;
                    fa.seeds += (uint32_t)((e & 0xFFFFu) == 0 && (jv & 0xFFFFu) != 0) +
                                (uint32_t)((e >> 16) == 0 && (jv >> 16) != 0);
                    fa.sI = __dp2a_lo(iv, 0x0101u, fa.sI);
                    fa.sJ = __dp2a_lo(jv, 0x0101u, fa.sJ);
                    fa.sD = __dp2a_lo(dv, 0x0101u, fa.sD);
                    fa.sI2 += (unsigned long long)(iv & 0xFFFFu) * (iv & 0xFFFFu);
                    fa.sI2 += (unsigned long long)(iv >> 16) * (iv >> 16);
                    fa.sJ2 += (unsigned long long)(jv & 0xFFFFu) * (jv & 0xFFFFu);
                    fa.sJ2 += (unsigned long long)(jv >> 16) * (jv >> 16);
                    // edges: the right neighbours in the tile, the pixel below in the tile
                    const uint32_t rp = k < 3 ? i[k < 3 ? k + 1 : k] : __byte_perm(i[0], w0, 0x5432);
                    const uint32_t rm = (k + 1 < nv ? 0xFFFFu : 0u) |
                                        (k + 5 < nv && (k < 3 || lc < 7) ? 0xFFFF0000u : 0u);
                    const uint32_t gxv = (max2(iv, rp) - min2(iv, rp)) & rm;
                    const uint32_t gyv = down ? max2(iv, nx[k]) - min2(iv, nx[k]) : 0u;
                    fa.edges += (uint32_t)((gxv & 0xFFFFu) + (gyv & 0xFFFFu) > thr) +
                                (uint32_t)((gxv >> 16) + (gyv >> 16) > thr);
                }
            }
            fa.npix += (uint32_t)(min(max(im.H - y, 0), RB) * nc);
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            p[k] = c[k];
            c[k] = n[k];
        }
    }
    can |= any != 0;
    bad |= nok != 0;
}

template <bool W16, int CONN, bool FEATS>
__device__ __forceinline__ void scan_strip_of(const ImageView &im, int y0, int x0, int lane, bool &can, bool &bad,
                                              FeatAcc &fa) {
    switch (scan_mode(im, W16, y0, x0)) {   // warp-uniform
        case kScanSpan: scan_strip<W16, kScanSpan, CONN, FEATS>(im, y0, x0, lane, can, bad, fa); break;
        case kScanWord: scan_strip<W16, kScanWord, CONN, FEATS>(im, y0, x0, lane, can, bad, fa); break;
        default: scan_strip<W16, kScanPixel, CONN, FEATS>(im, y0, x0, lane, can, bad, fa); break;
    }
}

// The scan: one strip per warp and step of the grid-stride loop (a strip that can rise marks
// its tile PENDING); FEATS (learned batches): one tile, whose features (tile t = feature
// block t) go to a.feats.
template <typename T, int CONN, bool FEATS>
__global__ void __launch_bounds__(kThreads, FEATS ? IWPP_SCAN_FEATS_MINB
                                                 : (std::is_same<T, AnyPix>::value ? IWPP_SCAN_ANY_MINB : IWPP_SCAN_MINB))
    scan_block_kernel(EngineArgs a) {
    using RT = RegTile<T, CONN, kCoopStrip>;
    constexpr int SPT = kCoopRows / kCoopStrip;   // strips per tile
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t nw = (uint64_t)gridDim.x * kWarpsPerCta, nu = (uint64_t)a.ntiles * (FEATS ? 1 : SPT);
    for (uint64_t u = (uint64_t)blockIdx.x * kWarpsPerCta + w; u < nu; u += nw) {
        const uint32_t t = (uint32_t)(FEATS ? u : u / SPT);
        const long long c0 = clock64();
        const ImageView im = image_of(a, t);
        const uint32_t lt = t - im.tile_base;
        const int ty = (int)(lt / im.tiles_x), tx = (int)(lt % im.tiles_x);
        const int x0 = tx * RT::TW;
        int y0 = ty * kCoopRows + (FEATS ? 0 : (int)(u % SPT) * kCoopStrip);
        if (!FEATS && y0 >= im.H) continue;   // a strip below the image (warp-uniform)
        bool can = false, bad = false;
        FeatAcc fa;
        const bool wide = RT::wide(im);
        for (int s = 0; s < (FEATS ? SPT : 1) && y0 < im.H; s++, y0 += kCoopStrip) {
            if constexpr (std::is_same<T, AnyPix>::value) {
                if (wide) scan_strip_of<true, CONN, FEATS>(im, y0, x0, lane, can, bad, fa);
                else scan_strip_of<false, CONN, FEATS>(im, y0, x0, lane, can, bad, fa);
            } else {
                scan_strip_of<sizeof(T) == 2, CONN, FEATS>(im, y0, x0, lane, can, bad, fa);
            }
        }
        can = __any_sync(0xffffffffu, can);
        bad = __any_sync(0xffffffffu, bad);
        if (FEATS) {
            uint32_t v[16];
            unsigned long long sI2, sJ2;
            feat_reduce(fa, v, sI2, sJ2);
            if (lane < IWPP_NFEAT) a.feats[(size_t)t * IWPP_NFEAT + lane] = block_feature(lane, v, sI2, sJ2, wide ? 0xFFFFu : 0xFFu);
        }
        if (lane == 0) {
            if (can) {
                if (a.defer_push) mark_pending(a, t); else notify_tile(a, t);
            }
            if (bad) set_status(a.hdr, kErrPrecondition);
            if (a.tile_work) atomicAdd(a.tile_work + a.ntiles + t, (uint32_t)min(clock64() - c0, 0x7fffffffll));
        }
    }
}

}  // namespace iwpp
