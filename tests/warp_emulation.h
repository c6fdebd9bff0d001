// Host stand-ins for the CUDA intrinsics of the device headers in csrc: the lanes of one or
// more warps run as fibers of one thread, so that device functions run on the CPU as they are
// written (asm statements are replaced textually, see warp_emulation.py).
//
// A lane runs until it meets a warp collective or a barrier.  A warp's collective completes
// once all 32 lanes have reached it; a barrier once all warps have.  Which warp runs between
// barriers is the schedule's choice: 0 runs the warps in order (warp 0 as far ahead as barriers
// let it), 1 in the opposite order, others switch pseudo-randomly after each collective.
// Warps that wait for each other at different points are reported as a deadlock.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <functional>
#include <vector>

#ifndef __noinline__
#define __noinline__
#endif
using std::isfinite;
using std::max;
using std::min;

namespace emu {

enum { kRun, kWarp, kBar, kDone };
struct Lane {
    ucontext_t ctx;
    int state = kRun;
    uint64_t in = 0;
    std::vector<char> stack;
};
struct Block {
    std::vector<Lane> lanes;
    ucontext_t sched;
    int cur = 0;
    std::function<void(int)> body;
    bool deadlock = false;
};
extern Block *blk;

inline void yield(int state) {
    Block *b = blk;
    Lane &l = b->lanes[b->cur];
    l.state = state;
    swapcontext(&l.ctx, &b->sched);
}
// every lane's value of its warp, at a point all 32 lanes reach
inline const uint64_t *exchange(uint64_t v, uint64_t *copy) {
    Block *b = blk;
    const int me = b->cur;
    b->lanes[me].in = v;
    yield(kWarp);
    for (int i = 0; i < 32; ++i) copy[i] = b->lanes[me / 32 * 32 + i].in;
    yield(kWarp);  // all have copied before anyone's next value
    return copy;
}
inline int lane_id() { return blk->cur & 31; }

inline void entry() {
    Block *b = blk;
    b->body(b->cur);
    yield(kDone);
}

// Runs body(thread) on 32 warps threads; false when warps deadlocked.
inline bool run(int warps, unsigned schedule, std::function<void(int)> body) {
    Block b;
    blk = &b;
    b.body = body;
    b.lanes.resize(32 * warps);
    for (auto &l : b.lanes) {
        l.stack.resize(256 << 10);
        getcontext(&l.ctx);
        l.ctx.uc_stack.ss_sp = l.stack.data();
        l.ctx.uc_stack.ss_size = l.stack.size();
        l.ctx.uc_link = &b.sched;
        makecontext(&l.ctx, entry, 0);
    }
    uint64_t rnd = schedule * 0x9E3779B97F4A7C15ull + 1;
    for (;;) {
        bool progress = false, all_done = true, all_bar = true;
        std::vector<int> order(warps);
        for (int w = 0; w < warps; ++w) order[w] = schedule == 1 ? warps - 1 - w : w;
        if (schedule > 1) {
            rnd = rnd * 6364136223846793005ull + 1442695040888963407ull;
            std::rotate(order.begin(), order.begin() + (int)((rnd >> 33) % warps), order.end());
        }
        for (int w : order) {
            Lane *l = &b.lanes[32 * w];
            for (;;) {
                bool ran = false;
                for (int i = 0; i < 32; ++i)
                    if (l[i].state == kRun) {
                        b.cur = 32 * w + i;
                        swapcontext(&b.sched, &l[i].ctx);
                        ran = true;
                    }
                int at = 0;
                for (int i = 0; i < 32; ++i) at += l[i].state == kWarp;
                if (at == 32) {
                    for (int i = 0; i < 32; ++i) l[i].state = kRun;
                    progress = true;
                    if (schedule > 1) break;
                    continue;
                }
                progress |= ran;
                if (!ran) break;
            }
            if (schedule > 1 && progress) break;
        }
        for (auto &l : b.lanes) {
            all_done &= l.state == kDone;
            all_bar &= l.state == kBar;
        }
        if (all_done) break;
        if (all_bar) {
            for (auto &l : b.lanes) l.state = kRun;
            progress = true;
        }
        if (!progress) {
            b.deadlock = true;
            break;
        }
    }
    blk = nullptr;
    return !b.deadlock;
}

inline float rcp(float x) { return 1.0f / x; }
inline void bar() { yield(kBar); }

}  // namespace emu

static uint3 threadIdx, blockIdx;
static dim3 blockDim(1), gridDim(1);

inline void __syncwarp() {
    uint64_t c[32];
    emu::exchange(0, c);
}
inline unsigned __reduce_or_sync(unsigned, unsigned v) {
    uint64_t c[32];
    emu::exchange(v, c);
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r |= (unsigned)c[i];
    return r;
}
inline unsigned __reduce_add_sync(unsigned, unsigned v) {
    uint64_t c[32];
    emu::exchange(v, c);
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r += (unsigned)c[i];
    return r;
}
template <class T>
inline T __reduce_max_sync(unsigned, T v) {
    uint64_t c[32];
    emu::exchange((uint64_t)v, c);
    T r = (T)c[0];
    for (int i = 1; i < 32; ++i) r = std::max(r, (T)c[i]);
    return r;
}
template <class T>
inline T __reduce_min_sync(unsigned, T v) {
    uint64_t c[32];
    emu::exchange((uint64_t)v, c);
    T r = (T)c[0];
    for (int i = 1; i < 32; ++i) r = std::min(r, (T)c[i]);
    return r;
}
template <class T>
inline T shfl_from(T v, int src) {
    uint64_t u = 0, c[32];
    memcpy(&u, &v, sizeof v);
    emu::exchange(u, c);
    u = c[src & 31];
    memcpy(&v, &u, sizeof v);
    return v;
}
template <class T>
inline T __shfl_xor_sync(unsigned, T v, int o) {
    return shfl_from(v, emu::lane_id() ^ o);
}
template <class T>
inline T __shfl_down_sync(unsigned, T v, int o) {
    const int l = emu::lane_id();
    return shfl_from(v, l + o < 32 ? l + o : l);
}
inline int __any_sync(unsigned, int p) { return __reduce_or_sync(0, p != 0) != 0; }
inline int __all_sync(unsigned, int p) { return !__any_sync(0, !p); }

inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
    s &= 31;
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
inline int __mulhi(int a, int b) { return (int)(((long long)a * b) >> 32); }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
inline long long __double_as_longlong(double x) {
    long long r;
    memcpy(&r, &x, 8);
    return r;
}
inline double __longlong_as_double(long long x) {
    double r;
    memcpy(&r, &x, 8);
    return r;
}
inline int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
inline int __double2loint(double x) { return (int)__double_as_longlong(x); }
inline double __hiloint2double(int h, int l) { return __longlong_as_double(((long long)h << 32) | (unsigned)l); }
inline unsigned __float_as_uint(float x) {
    unsigned r;
    memcpy(&r, &x, 4);
    return r;
}
inline float __uint_as_float(unsigned x) {
    float r;
    memcpy(&r, &x, 4);
    return r;
}
inline unsigned __byte_perm(unsigned a, unsigned b, unsigned s) {
    const unsigned long long v = ((unsigned long long)b << 32) | a;
    unsigned r = 0;
    for (int i = 0; i < 4; ++i) r |= (unsigned)((v >> (8 * ((s >> (4 * i)) & 7))) & 0xff) << (8 * i);
    return r;
}
template <class T>
inline T atomicOr(T *p, T v) {
    const T o = *p;
    *p |= v;
    return o;
}
