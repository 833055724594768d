// iwpp_smemtile.cuh — a 64 x 64 tile in shared memory, settled by the eight warps of a CTA
// (sm_103a): the local solver of the operators whose row steps are heavy (watershed, influence
// zones). Each warp owns a strip of 8 rows; lane c updates columns 2c and 2c + 1 of a row.
//
// A row step of these operators weighs 60-100 instructions, so the drain is bound by how many
// row steps it runs and by the warps there are to overlap them; small images by the chain of row
// steps between two barriers. With the tile in shared memory the passes are loops over a row index:
// the code holds one row step per direction, a thread needs 64-80 registers instead of 150-250, so
// three times as many warps fit, and only the rows whose neighbours changed are run, by three bit
// masks per strip: n, a pixel may change through the row above; s, through the row below; h, through
// its own row. A down pass (rows top to bottom) settles n, an up pass s, either h when it changes
// nothing. A tile that was visited before starts with the rows next to its halo that the halo can
// change, and nothing else.
//
// Strips exchange after one pass pair, eight strips of 8 rows. Both were chosen with rows that each
// went through shared memory (and plain accesses between strips), on inputs of their own, with
// (warps, exchange):
// watershed of 2048^2 u16 and 4096^2 u16, influence zones of 4096^2 and 1000^2:
// (4, when clean) 1565 / 2742 / 1173 / 642 us, (4, pair) 1282 / 2489 / 1133 / 527, (8, when clean)
// 1500 / 3119 / 1316 / 591, (8, pair) 1122 / 2946 / 1171 / 423, (8, single pass) 1432 / 2974 / 1217 / 458,
// (16, pair) 1324 / 4011 / 1767 / 440. They have not been timed again since.
//
// Runs of rows (sm_pass_pair), whole calls, against strips of 16 rows in one warp's registers (the form
// before these tiles), 57 watersheds and 57 influence zones from 200^2 to 4096^2, u8 and u16, both
// connectivities: geometric mean 1.63 and 2.58 times as fast, the slowest 1.16 and 2.17 (each
// row through shared memory: 1.04 and 2.05, with 200^2 watersheds down to 0.88).
//
// Strips read the adjacent strips' boundary rows where they lie. A pixel is written by its own strip
// only; between two barriers those writes, and the reads of another strip's row, are single relaxed
// accesses of a whole pixel (sm_st_relaxed, sm_ld_relaxed): a pixel read while it changes is its
// older or its newer state, never half of each, and pixels only ever improve, so either is
// valid; the strip whose row changed hands its neighbour the row again at the next barrier.
//
// Op: the operator. Px (a pixel's state, one aligned 4- or 8-byte word), Aux (what it needs
// beside it), RowAux (a lane's part of that for a row, row_aux) and Ctx (kernel arguments), none() (outside the image), load / store, load_aux,
// row<CONN> (one lane's two pixels of a row step, from columns 2c - 1 .. 2c + 2 of the row and of the
// one before it), halo_aux and changes (whether pixels offered to a halo pixel change it).
#pragma once
#include "iwpp_engine.cuh"

namespace iwpp {

constexpr int kSmWarps = 8, kSmThreads = 32 * kSmWarps;
constexpr int kSmSide = 64, kSmStrip = kSmSide / kSmWarps, kSmPitch = kSmSide + 4;
constexpr uint32_t kSmRows = (1u << kSmStrip) - 1u;
// Sides of the halo: index i runs along the side (columns or rows of the tile); corners by side
// kTop / kBottom with i = -1 or 64.
enum : int { kTop = 0, kBottom = 1, kLeft = 2, kRight = 3 };

// The tile with its one-pixel halo: row r at index r + 1, column c at c + 1, so that the pair of
// columns 2c - 1, 2c is aligned: a lane reads its two pixels and both their horizontal
// neighbours in two accesses.
template <class Op>
struct SmemTile {
    typename Op::Px v[kSmSide + 2][kSmPitch];
    typename Op::Aux aux;
    uint32_t in[2][kSmWarps];   // work handed to a strip by its neighbours: bit 0 n of its first row, 1 s of its last
    uint32_t note;                  // neighbours to notify (3 x 3 grid bits)
    uint32_t tile, first, redo;
};

struct RowWork {
    uint32_t n, s, h;
};

// One whole pixel of shared memory, relaxed at block scope.
__device__ __forceinline__ uint32_t sm_ld_relaxed(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.relaxed.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long sm_ld_relaxed(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.cta.shared.u64 %0, [%1];" : "=l"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
    return v;
}
__device__ __forceinline__ void sm_st_relaxed(uint32_t *p, uint32_t v) {
    asm volatile("st.relaxed.cta.shared.u32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void sm_st_relaxed(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.cta.shared.u64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "l"(v) : "memory");
}
// Four pixels of a row of the warp's own strip or of the halo, from an even index on.
__device__ __forceinline__ void sm_ld4(const uint32_t *p, uint32_t (&q)[4]) {
    const uint2 a = *reinterpret_cast<const uint2 *>(p), b = *reinterpret_cast<const uint2 *>(p + 2);
    q[0] = a.x; q[1] = a.y; q[2] = b.x; q[3] = b.y;
}
__device__ __forceinline__ void sm_ld4(const unsigned long long *p, unsigned long long (&q)[4]) {
    const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(p), b = *reinterpret_cast<const ulonglong2 *>(p + 2);
    q[0] = a.x; q[1] = a.y; q[2] = b.x; q[3] = b.y;
}

template <class Op>
__device__ __forceinline__ typename Op::Px sm_ld(const ImageView &im, int y, int x) {
    const bool in = y >= 0 && y < im.H && x >= 0 && x < im.W;
    const typename Op::Px v = Op::load(im, (size_t)min(max(y, 0), im.H - 1) * im.W + min(max(x, 0), im.W - 1));
    return in ? v : Op::none();
}

template <class Op>
__device__ void sm_load(const ImageView &im, SmemTile<Op> &S, int y0, int x0, int w, int lane) {
    const int ys = y0 + kSmStrip * w;
#pragma unroll 8
    for (int r = 0; r < kSmStrip; r++) {
        const typename Op::Px a = sm_ld<Op>(im, ys + r, x0 + lane), b = sm_ld<Op>(im, ys + r, x0 + 32 + lane);
        S.v[kSmStrip * w + r + 1][lane + 1] = a;
        S.v[kSmStrip * w + r + 1][lane + 33] = b;
    }
}

// The halo beside and, for the outer strips, above / below the strip. RELOAD: the rows that its
// changes may change are added to the work.
template <class Op, bool RELOAD>
__device__ void sm_load_halo(const ImageView &im, SmemTile<Op> &S, int y0, int x0, RowWork &k, int w, int lane) {
    // this lane's pixel of the side halo (those of lanes from 2 kSmStrip on repeat and are not used)
    const int r = lane % kSmStrip, right = lane / kSmStrip % 2;
    const bool side = lane < 2 * kSmStrip;
    const int ri = kSmStrip * w + r + 1, ci = right ? kSmSide + 1 : 0;
    const typename Op::Px sv = sm_ld<Op>(im, y0 + kSmStrip * w + r, right ? x0 + kSmSide : x0 - 1);
    const bool outer = w == 0 || w == kSmWarps - 1;
    const int yh = w == 0 ? y0 - 1 : y0 + kSmSide, rh = w == 0 ? 0 : kSmSide + 1;
    typename Op::Px a = Op::none(), b = Op::none(), c = Op::none();
    if (outer) {   // warp-uniform
        a = sm_ld<Op>(im, yh, x0 + lane);
        b = sm_ld<Op>(im, yh, x0 + 32 + lane);
        c = sm_ld<Op>(im, yh, (lane & 1) ? x0 + kSmSide : x0 - 1);
    }
    if (RELOAD) {
        const uint32_t d = __ballot_sync(0xffffffffu, side && S.v[ri][ci] != sv);
        const uint32_t rows = (d | (d >> kSmStrip)) & kSmRows;
        const uint32_t near = (rows | (rows << 1) | (rows >> 1)) & kSmRows;   // beside or next to a changed pixel
        k.n |= near;
        k.s |= near;
        k.h |= near;
        // rows of the adjacent strips next to this strip's end rows' halo pixels
        if (lane == 0) {
            if (w > 0 && (rows & 1u)) atomicOr(&S.in[0][w - 1], 4u);
            if (w < kSmWarps - 1 && (rows >> (kSmStrip - 1))) atomicOr(&S.in[0][w + 1], 8u);
        }
        if (outer) {
            const bool ch = S.v[rh][lane + 1] != a || S.v[rh][lane + 33] != b ||
                            (lane < 2 && S.v[rh][lane ? kSmSide + 1 : 0] != c);
            if (__any_sync(0xffffffffu, ch)) {
                const uint32_t bit = w == 0 ? 1u : 1u << (kSmStrip - 1);
                if (w == 0) k.n |= bit; else k.s |= bit;
            }
        }
    }
    if (side) S.v[ri][ci] = sv;
    if (outer) {
        S.v[rh][lane + 1] = a;
        S.v[rh][lane + 33] = b;
        if (lane < 2) S.v[rh][lane ? kSmSide + 1 : 0] = c;
    }
}

// The work of a tile visited before, whose pixels were settled under the halo of that visit: the
// strip's rows that the side halo can change now, and the rows next to the tile's halo rows.
template <class Op, int CONN>
__device__ RowWork sm_revisit_work(const SmemTile<Op> &S, const typename Op::Ctx &ctx, int w, int lane) {
    const int r = kSmStrip * w + lane % kSmStrip, right = lane / kSmStrip % 2;
    const int ci = right ? kSmSide + 1 : 0, ct = right ? kSmSide : 1;
    typename Op::Px q[3] = {S.v[r + 1][ci], S.v[r][ci], S.v[r + 2][ci]};
    const bool ch = Op::changes_own(S.v[r + 1][ct], S.aux, ctx, r, right ? kSmSide - 1 : 0, q, CONN == 8 ? 3 : 1);
    const uint32_t d = __ballot_sync(0xffffffffu, ch);
    const uint32_t rows = (d | (d >> kSmStrip)) & kSmRows;
    RowWork k = {rows, rows, rows};
    if (w == 0) k.n |= 1u;
    if (w == kSmWarps - 1) k.s |= 1u << (kSmStrip - 1);
    return k;
}

// One down and one up pass over the strip's rows with work; returns the rows changed. Rows that
// follow one another are a run: the next row is loaded ahead and the previous one stays in registers (its
// neighbour columns by shuffles beside the vote), so that a row does not wait for the one before
// to pass through shared memory.
template <class Op, int CONN>
__device__ uint32_t sm_pass_pair(SmemTile<Op> &S, const typename Op::Ctx &ctx, RowWork &k, uint32_t &passes, int w, int lane) {
    using Px = typename Op::Px;
    uint32_t rows = 0;
#pragma unroll   // (a direction known at compile time: 5-12 % faster)
    for (int dir = 1; dir >= -1; dir -= 2) {
        uint32_t v = dir > 0 ? k.n : k.s, u = dir > 0 ? k.s : k.n;
        for (uint32_t left = kSmRows;;) {
            const uint32_t m = (v | k.h) & left;
            if (m == 0) break;
            int r = dir > 0 ? __ffs(m) - 1 : 31 - __clz(m);
            uint32_t bit = 1u << r;
            Px q[4], p[4];
            __syncwarp();   // rows written before are read by other lanes
            Px *row = &S.v[kSmStrip * w + r + 1][2 * lane];
            const Px *prv = row - dir * kSmPitch;
            sm_ld4(row, q);
            if (dir > 0 ? r == 0 && w > 0 : r == kSmStrip - 1 && w < kSmWarps - 1) {   // another strip's row
#pragma unroll
                for (int i = 0; i < 4; i++) p[i] = sm_ld_relaxed(prv + i);
            } else {
                sm_ld4(prv, p);
            }
            typename Op::RowAux x = Op::row_aux(S.aux, kSmStrip * w + r, lane);
            for (;;) {
                const uint32_t next = dir > 0 ? (bit << 1) & kSmRows : bit >> 1;
                const int step = next ? dir : 0;   // (at the strip's end the row itself again)
                Px nx[4], e, o;
                sm_ld4(row + step * kSmPitch, nx);
                const typename Op::RowAux xn = Op::row_aux(S.aux, kSmStrip * w + r + step, lane);
                const bool ch = Op::template row<CONN>(q, p, x, lane, e, o);
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
                    sm_st_relaxed(row + 1, e);
                    sm_st_relaxed(row + 2, o);
                }
                v &= ~bit;
                k.h &= ~bit;
                if (any) {
                    rows |= bit;
                    k.h |= bit;
                    v |= next;
                    u |= dir > 0 ? bit >> 1 : (bit << 1) & kSmRows;
                }
                left = dir > 0 ? ~((bit << 1) - 1u) & kSmRows : bit - 1u;
                if (((v | k.h) & next) == 0) break;
                r += dir;
                bit = next;
                row += dir * kSmPitch;
                x = xn;
#pragma unroll
                for (int i = 0; i < 4; i++) q[i] = nx[i];
            }
        }
        k.n = dir > 0 ? v : u;
        k.s = dir > 0 ? u : v;
    }
    __syncwarp();
    passes += 2;
    return rows;
}

// The tile's neighbours that the strip's pixels (with those of the strips beside it) can change.
template <class Op, int CONN>
__device__ uint32_t sm_notify_mask(const SmemTile<Op> &S, const typename Op::Ctx &ctx, int w, int lane) {
    uint32_t mask = 0;
    {
        const int r = kSmStrip * w + lane % kSmStrip, right = lane / kSmStrip % 2;   // row of the tile, side
        const int ci = right ? kSmSide + 1 : 0, ct = right ? kSmSide : 1;
        typename Op::Px q[3] = {S.v[r + 1][ct], r > 0 ? S.v[r][ct] : Op::none(),
                                r < kSmSide - 1 ? S.v[r + 2][ct] : Op::none()};
        const bool ch = Op::changes(S.v[r + 1][ci], Op::halo_aux(S.aux, right ? kRight : kLeft, r), q, CONN == 8 ? 3 : 1);
        const uint32_t b = __ballot_sync(0xffffffffu, ch);
        if (b & kSmRows) mask |= 8u;
        if ((b >> kSmStrip) & kSmRows) mask |= 32u;
    }
    if (w == 0 || w == kSmWarps - 1) {   // warp-uniform
        const int rh = w == 0 ? 0 : kSmSide + 1, rt = w == 0 ? 1 : kSmSide, side = w == 0 ? kTop : kBottom;
        bool ch = false;
#pragma unroll
        for (int p = 0; p < 2; p++) {
            const int c = lane + 32 * p;
            typename Op::Px q[3] = {S.v[rt][c + 1], c > 0 ? S.v[rt][c] : Op::none(),
                                    c < kSmSide - 1 ? S.v[rt][c + 2] : Op::none()};
            ch |= Op::changes(S.v[rh][c + 1], Op::halo_aux(S.aux, side, c), q, CONN == 8 ? 3 : 1);
        }
        if (__any_sync(0xffffffffu, ch)) mask |= w == 0 ? 2u : 128u;
        if (CONN == 8) {   // corners: lanes 0 and 1
            const int right = lane & 1;
            typename Op::Px q[3] = {S.v[rt][right ? kSmSide : 1], Op::none(), Op::none()};
            const bool cc = lane < 2 && Op::changes(S.v[rh][right ? kSmSide + 1 : 0],
                                                    Op::halo_aux(S.aux, side, right ? kSmSide : -1), q, 1);
            const uint32_t b = __ballot_sync(0xffffffffu, cc);
            mask |= ((b & 1u) | ((b & 2u) << 1)) << (w == 0 ? 0 : 6);
        }
    }
    return mask;
}

// One visit of tile t by the whole CTA, with the rounds it is notified to repeat.
template <class Op, int CONN>
__device__ void sm_visit(const EngineArgs &a, const typename Op::Ctx &ctx, uint32_t t, bool first, SmemTile<Op> &S,
                         VisitStats &st, int w, int lane) {
    const ImageView &im = a.img0;
    const int ty = (int)(t / im.tiles_x), tx = (int)(t % im.tiles_x);
    const int y0 = ty * kSmSide, x0 = tx * kSmSide;
    RowWork k = {kSmRows, kSmRows, kSmRows};
    sm_load<Op>(im, S, y0, x0, w, lane);
    sm_load_halo<Op, false>(im, S, y0, x0, k, w, lane);
    Op::load_aux(S.aux, im, ctx, y0, x0, w, lane);
    __syncthreads();
    if (!first) k = sm_revisit_work<Op, CONN>(S, ctx, w, lane);
    uint32_t passes = 0, par = 0;
    for (;;) {
        uint32_t rows = 0;
        for (;;) {   // joint iterations of the strips
            const uint32_t ch = sm_pass_pair<Op, CONN>(S, ctx, k, passes, w, lane);
            rows |= ch;
            const bool up = w > 0 && (ch & 1u), dn = w < kSmWarps - 1 && (ch >> (kSmStrip - 1));
            if (lane == 0) {   // hand the changed end rows to the strips beside them
                if (up) atomicOr(&S.in[par][w - 1], 2u);
                if (dn) atomicOr(&S.in[par][w + 1], 1u);
            }
            const bool more = __syncthreads_or(up || dn || (k.n | k.s | k.h) != 0);
            const uint32_t in = S.in[par][w];
            __syncwarp();
            if (lane == 0) S.in[par][w] = 0;   // (written again two barriers from here)
            if (in & 1u) k.n |= 1u;
            if (in & 2u) k.s |= 1u << (kSmStrip - 1);
            par ^= 1;
            if (!more) break;
        }
        if (w == 0 && lane == 0) st.visits++;
        if (__syncthreads_or(rows != 0)) {
            for (uint32_t m = rows; m; m &= m - 1) {   // changed rows (they lie inside the image)
                const int r = kSmStrip * w + __ffs(m) - 1;
                const size_t row = (size_t)(y0 + r) * im.W;
                if (x0 + lane < im.W) Op::store(im, row + x0 + lane, S.v[r + 1][lane + 1]);
                if (x0 + 32 + lane < im.W) Op::store(im, row + x0 + 32 + lane, S.v[r + 1][lane + 33]);
            }
            const uint32_t note = sm_notify_mask<Op, CONN>(S, ctx, w, lane);
            if (lane == 0 && note) atomicOr(&S.note, note);
            __threadfence();
            __syncthreads();
            if (w == 0) {
                const uint32_t n = S.note;
                __syncwarp();
                if (lane == 0) S.note = 0;
                if (lane < 9 && lane != 4 && ((n >> lane) & 1u)) {
                    const int ny = ty + lane / 3 - 1, nx = tx + lane % 3 - 1;
                    if (ny >= 0 && nx >= 0 && ny < im.tiles_y && nx < im.tiles_x)
                        notify_tile(a, (uint32_t)(ny * im.tiles_x + nx));
                }
            }
        }
        if (w == 0) {
            const bool r = finish_tile(a, t, lane);
            if (lane == 0) S.redo = r;
        }
        __syncthreads();
        if (S.redo == 0) break;
        // re-process: only the halo can have changed (in[0] and in[1] are zero here)
        sm_load_halo<Op, true>(im, S, y0, x0, k, w, lane);
        __syncthreads();
        const uint32_t in = S.in[0][w];
        __syncwarp();
        if (lane == 0) S.in[0][w] = 0;
        if (in & 4u) {   // the halo pixel beside the next strip's first row changed
            k.s |= 1u << (kSmStrip - 1);
            k.h |= 1u << (kSmStrip - 1);
        }
        if (in & 8u) {
            k.n |= 1u;
            k.h |= 1u;
        }
        par = 1;
    }
    st.waves += passes;
}

// The persistent kernel's body: warp 0 pops a tile for the CTA, the CTA visits it.
template <class Op, int CONN>
__device__ __forceinline__ void sm_drain(const EngineArgs &a, const typename Op::Ctx &ctx, SmemTile<Op> &S) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    VisitStats st = {0, 0, 0, 0};
    unsigned long long idle = 0, busy = 0;
    if (threadIdx.x < 2 * kSmWarps) S.in[threadIdx.x / kSmWarps][threadIdx.x % kSmWarps] = 0;
    if (threadIdx.x == 0) S.note = 0;
    for (;;) {
        if (warp == 0) {
            bool first;
            const uint32_t t = acquire_tile(a, first, idle, lane);
            if (lane == 0) {
                S.tile = t;
                S.first = first;
            }
        }
        __syncthreads();
        const uint32_t t = S.tile;
        if (t == kDone) break;
        const unsigned long long b0 = globaltimer_ns();
        sm_visit<Op, CONN>(a, ctx, t, S.first != 0, S, st, warp, lane);
        if (warp == 0) busy += globaltimer_ns() - b0;
        __syncthreads();   // every warp has read S.tile before the next pop overwrites it
    }
    flush_stats(a, st, idle, busy, lane);
}

}  // namespace iwpp
