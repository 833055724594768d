// What iwpp_smemtile.cuh takes from the tile engine, for one CTA on the host.
#pragma once
#include "host_cta.h"

namespace iwpp {
constexpr uint32_t kDone = 0xFFFFFFFFu;
struct ImageView {
    unsigned long long *J;
    int H, W, tiles_x, tiles_y;
};
struct EngineArgs { ImageView img0; };
struct VisitStats { uint32_t visits, pops, seeds, waves; };
uint32_t acquire_tile(const EngineArgs &a, bool &first, unsigned long long &idle, int lane);
void notify_tile(const EngineArgs &a, uint32_t t);
bool finish_tile(const EngineArgs &a, uint32_t t, int lane);
inline void flush_stats(const EngineArgs &, const VisitStats &, unsigned long long, unsigned long long, int) {}
inline unsigned long long globaltimer_ns() { return 0; }
}  // namespace iwpp
