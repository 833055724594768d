// One CTA of device code on the host: every thread is a fiber, warp collectives and barriers are
// rendezvous, and between rendezvous the warps run in random order. It counts the warp and CTA
// barriers a thread has passed, so that a test can tell which accesses to shared memory are ordered.
#pragma once
#include <ucontext.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>

#define __device__
#define __forceinline__ inline

struct HostCta {
    struct Thread {
        ucontext_t ctx;
        std::vector<char> stack;
        bool done = false;
        unsigned cta_epoch = 0, warp_epoch = 0;   // barriers passed
    };
    struct Meet {
        int arrived = 0;
        unsigned gen = 0;
        uint64_t in[1024], out[1024];
    };
    std::vector<Thread> th;
    std::vector<Meet> warp;
    Meet cta;
    ucontext_t main;
    int cur = 0;
    uint32_t rng = 1;
    std::function<void()> body;
    uint32_t random() { return (rng = rng * 1664525u + 1013904223u) >> 8; }
    void yield() { swapcontext(&th[cur].ctx, &main); }
    // Everybody's value once all n members have given theirs (valid until this thread's next meeting).
    const uint64_t *meet(Meet &m, int at, int n, uint64_t v) {
        m.in[at] = v;
        const unsigned g = m.gen;
        if (++m.arrived == n) {
            std::copy(m.in, m.in + n, m.out);
            m.arrived = 0;
            m.gen++;
        } else {
            while (m.gen == g) yield();
        }
        return m.out;
    }
    const uint64_t *warp_meet(uint64_t v) { return meet(warp[cur / 32], cur % 32, 32, v); }
    void run(int n, uint32_t seed, std::function<void()> fn);
};
inline HostCta H;
inline void host_thread() {
    H.body();
    H.th[H.cur].done = true;
    swapcontext(&H.th[H.cur].ctx, &H.main);
}
inline void HostCta::run(int n, uint32_t seed, std::function<void()> fn) {
    body = fn;
    rng = seed;
    th.clear();
    th.resize(n);
    warp.clear();
    warp.resize((n + 31) / 32);
    cta = Meet();
    for (Thread &t : th) {
        t.stack.resize(128 << 10);
        getcontext(&t.ctx);
        t.ctx.uc_stack.ss_sp = t.stack.data();
        t.ctx.uc_stack.ss_size = t.stack.size();
        t.ctx.uc_link = &main;
        makecontext(&t.ctx, host_thread, 0);
    }
    for (long rounds = 0;; rounds++) {
        if (rounds > 50000000) { printf("the CTA does not end\n"); exit(3); }
        if (std::all_of(th.begin(), th.end(), [](const Thread &t) { return t.done; })) break;
        const int w = (int)(random() % warp.size());   // a warp, its threads up to their next meeting
        for (int i = 32 * w; i < std::min(n, 32 * w + 32); i++)
            if (!th[i].done) { cur = i; swapcontext(&main, &th[i].ctx); }
    }
}

struct Dim { unsigned x, y, z; };
#define threadIdx (Dim{(unsigned)H.cur, 0u, 0u})
inline uint32_t __ballot_sync(uint32_t, bool p) {
    const uint64_t *o = H.warp_meet(p);
    uint32_t r = 0;
    for (int i = 0; i < 32; i++) r |= (uint32_t)o[i] << i;
    return r;
}
inline bool __any_sync(uint32_t m, bool p) { return __ballot_sync(m, p) != 0; }
inline uint32_t __shfl_sync(uint32_t, uint32_t v, int s) { return (uint32_t)H.warp_meet(v)[s]; }
// (votes and shuffles order no memory accesses: only the barriers count)
inline void __syncwarp() { H.warp_meet(0); H.th[H.cur].warp_epoch++; }
inline bool __syncthreads_or(bool p) {
    const int n = (int)H.th.size();
    const uint64_t *o = H.meet(H.cta, H.cur, n, p);
    bool r = false;
    for (int i = 0; i < n; i++) r |= o[i] != 0;
    H.th[H.cur].cta_epoch++;
    return r;
}
inline void __syncthreads() { __syncthreads_or(false); }
inline void __threadfence() {}
template <class T> T atomicOr(T *p, T v) { const T o = *p; *p = o | v; return o; }
inline int __ffs(uint32_t v) { return __builtin_ffs((int)v); }
inline int __clz(uint32_t v) { return v ? __builtin_clz(v) : 32; }
inline unsigned long long __cvta_generic_to_shared(const void *p) { return (unsigned long long)(uintptr_t)p; }
struct uint2 { uint32_t x, y; };
struct ulonglong2 { unsigned long long x, y; };
using std::max;
using std::min;
