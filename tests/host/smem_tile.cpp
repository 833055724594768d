// The shared-memory tile (iwpp_smemtile.cuh) on the host, with an operator whose pixels record every
// access to the tile: two accesses to one pixel, at least one a write, by threads that no barrier
// orders are a race unless both are whole relaxed accesses of different warps' threads. The
// operator (fewest steps to a source, then smallest label) has one fixed point; results are compared with it.
#include "iwpp_smemtile.cuh"   // beside host_cta.h and the engine below

#include <map>

using namespace iwpp;

struct Px;
static const char *tile_begin, *tile_end;
static long races[3];   // between warps; within a warp two writes, a read and a write
struct Access { int tid; unsigned warp_epoch; bool write, strong; };
struct Log { unsigned epoch = 0; std::vector<Access> a; };
static std::map<const void *, Log> logs;
static void note(const void *p, bool write, bool strong) {
    if ((const char *)p < tile_begin || (const char *)p >= tile_end) return;
    const auto &t = H.th[H.cur];
    Log &l = logs[p];
    if (l.epoch != t.cta_epoch) { l.epoch = t.cta_epoch; l.a.clear(); }
    for (const Access &o : l.a) {
        if (o.tid == H.cur || !(o.write || write)) continue;
        const bool same_warp = o.tid / 32 == H.cur / 32;
        if (same_warp ? o.warp_epoch == t.warp_epoch : !(o.strong && strong)) {
            if (races[!same_warp ? 0 : (o.write && write ? 1 : 2)]++ == 0)
                printf("race: threads %d and %d at +%ld\n", o.tid, H.cur, (long)((const char *)p - tile_begin));
            break;
        }
    }
    for (const Access &o : l.a)
        if (o.tid == H.cur && o.warp_epoch == t.warp_epoch && o.write == write && o.strong == strong) return;
    l.a.push_back({H.cur, t.warp_epoch, write, strong});
}
struct Px {
    unsigned long long v;
    Px() = default;
    explicit Px(unsigned long long x) : v(x) {}
    Px(const Px &o) : v(o.v) { note(&o, false, false); }
    Px &operator=(const Px &o) { note(&o, false, false); note(this, true, false); v = o.v; return *this; }
    bool operator!=(const Px &o) const { note(this, false, false); note(&o, false, false); return v != o.v; }
};
static Px sm_ld_relaxed(const Px *p) { note(p, false, true); return Px(p->v); }
static void sm_st_relaxed(Px *p, const Px &v) { note(p, true, true); p->v = v.v; }
static Px __shfl_up_sync(uint32_t, const Px &v, int n) {
    const int l = H.cur % 32;
    return Px(H.warp_meet(v.v)[l < n ? l : l - n]);
}
static Px __shfl_down_sync(uint32_t, const Px &v, int n) {
    const int l = H.cur % 32;
    return Px(H.warp_meet(v.v)[l + n > 31 ? l : l + n]);
}
static void sm_ld4(const Px *p, Px (&q)[4]) { for (int i = 0; i < 4; i++) q[i] = p[i]; }

constexpr unsigned long long kFar = 1ull << 62, kWall = ~0ull, kStep = 1ull << 32;
static unsigned long long step(unsigned long long own, unsigned long long q) {
    return own == kWall || q >= kFar ? own : std::min(own, q + kStep);
}
struct TestOp {
    using Px = ::Px;
    struct Aux {};
    struct RowAux {};
    struct Ctx {};
    static RowAux row_aux(const Aux &, int, int) { return RowAux{}; }
    static Px none() { return Px(kWall); }
    static Px load(const ImageView &im, size_t e) { return Px(im.J[e]); }
    static void store(const ImageView &im, size_t e, const Px &v) { note(&v, false, false); im.J[e] = v.v; }
    static void load_aux(Aux &, const ImageView &, const Ctx &, int, int, int, int) {}
    static uint32_t halo_aux(const Aux &, int, int) { return 0; }
    template <int CONN>
    static bool row(const Px (&q)[4], const Px (&p)[4], const RowAux &, int, Px &e, Px &o) {
        unsigned long long v = step(step(step(q[1].v, q[0].v), q[2].v), p[1].v), u = step(q[2].v, p[2].v);
        if (CONN == 8) {
            v = step(step(v, p[0].v), p[2].v);
            u = step(step(u, p[1].v), p[3].v);
        }
        e.v = v;
        o.v = step(step(u, q[3].v), v);
        return e.v != q[1].v || o.v != q[2].v;
    }
    static bool changes(const Px &h, uint32_t, const Px (&q)[3], int n) {
        const unsigned long long v = h.v;
        note(&h, false, false);
        unsigned long long r = v;
        for (int k = 0; k < n; k++) r = step(r, q[k].v);
        return r != v;
    }
    static bool changes_own(const Px &v, const Aux &, const Ctx &, int, int, const Px (&q)[3], int n) {
        return changes(v, 0, q, n);
    }
};

// The engine of one CTA: a list of tiles. While a tile is held, now and then what another CTA could
// do happens to pixels beside it: they take their final values, their tile is to be visited, and
// the held tile goes another round.
namespace iwpp {
static std::vector<uint32_t> todo;
static std::vector<char> queued, visited;
static std::vector<unsigned long long> final_values;
uint32_t acquire_tile(const EngineArgs &, bool &first, unsigned long long &, int lane) {
    uint32_t t = kDone;
    if (lane == 0 && !todo.empty()) {
        const size_t k = H.random() % todo.size();
        t = todo[k];
        todo.erase(todo.begin() + k);
        queued[t] = 0;
    }
    t = __shfl_sync(~0u, t, 0);
    first = t != kDone && !visited[t];
    __syncwarp();
    if (lane == 0 && t != kDone) visited[t] = 1;
    return t;
}
void notify_tile(const EngineArgs &, uint32_t t) {
    if (!queued[t]) todo.push_back(t);
    queued[t] = 1;
}
bool finish_tile(const EngineArgs &a, uint32_t t, int lane) {
    const ImageView &im = a.img0;
    uint32_t redo = 0;
    if (lane == 0 && H.random() % 2) {
        const int y0 = (int)(t / im.tiles_x) * 64 - 1, x0 = (int)(t % im.tiles_x) * 64 - 1;
        for (int k = 0; k < 6; k++) {
            const int along = (int)(H.random() % 66), side = (int)(H.random() % 4);
            const int y = side < 2 ? y0 + 65 * side : y0 + along, x = side < 2 ? x0 + along : x0 + 65 * (side - 2);
            if (y < 0 || x < 0 || y >= im.H || x >= im.W || im.J[(size_t)y * im.W + x] == final_values[(size_t)y * im.W + x])
                continue;
            im.J[(size_t)y * im.W + x] = final_values[(size_t)y * im.W + x];
            const uint32_t u = (uint32_t)(y / 64 * im.tiles_x + x / 64);
            visited[u] = 0;
            notify_tile(a, u);
            redo = 1;
        }
    }
    return __shfl_sync(~0u, redo, 0) != 0;
}
}  // namespace iwpp

template <int CONN>
static int one(int rows, int cols, int walls, uint32_t seed) {
    static SmemTile<TestOp> S;
    tile_begin = (const char *)&S.v;
    tile_end = tile_begin + sizeof(S.v);
    H.rng = seed * 7919u + 3u;
    std::vector<unsigned long long> J((size_t)rows * cols);
    for (auto &v : J) v = (int)(H.random() % 100) < walls ? kWall : kFar;
    for (int k = 0; k <= rows * cols / 3000; k++) J[H.random() % J.size()] = 1 + H.random() % 5;
    final_values = J;
    for (bool ch = true; ch;) {
        ch = false;
        for (int pass = 0; pass < 2; pass++)
            for (int k = 0; k < rows * cols; k++) {
                const int i = pass ? rows * cols - 1 - k : k, y = i / cols, x = i % cols;
                for (int dy = -1; dy <= 1; dy++)
                    for (int dx = -1; dx <= 1; dx++) {
                        if ((CONN == 4 && dy && dx) || y + dy < 0 || x + dx < 0 || y + dy >= rows || x + dx >= cols) continue;
                        const unsigned long long n = step(final_values[i], final_values[(y + dy) * cols + x + dx]);
                        ch |= n != final_values[i];
                        final_values[i] = n;
                    }
            }
    }
    EngineArgs a = {};
    a.img0 = {J.data(), rows, cols, (cols + 63) / 64, (rows + 63) / 64};
    const uint32_t nt = (uint32_t)(a.img0.tiles_x * a.img0.tiles_y);
    queued.assign(nt, 0);
    visited.assign(nt, 0);
    todo.clear();
    for (int i = 0; i < rows * cols; i++)
        if (J[i] < kFar) notify_tile(a, (uint32_t)(i / cols / 64 * a.img0.tiles_x + i % cols / 64));
    logs.clear();
    H.run(kSmThreads, seed, [&] { sm_drain<TestOp, CONN>(a, TestOp::Ctx{}, S); });
    if (J != final_values) printf("conn %d %d x %d seed %u: another result\n", CONN, rows, cols, seed);
    return J != final_values;
}

int main(int argc, char **) {
    int bad = 0;
    const int sizes[][2] = {{65, 70}, {1, 1}, {64, 64}, {7, 200}, {200, 9}, {130, 150}};
    for (auto &s : sizes) {
        if (argc > 1 && &s != sizes) break;   // any argument: the first size only
        for (int walls : {0, 40}) {
            bad += one<8>(s[0], s[1], walls / 2, 1u + walls);
            bad += one<4>(s[0], s[1], walls / 2, 2u + walls);
        }
    }
    printf("%d wrong results, races: %ld between warps, within one %ld and %ld\n", bad, races[0], races[1], races[2]);
    return (bad ? 1 : 0) | (races[0] ? 2 : 0) | (races[1] ? 4 : 0) | (races[2] ? 8 : 0);
}
