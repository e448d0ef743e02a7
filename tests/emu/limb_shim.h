// The shuffles of the limb-lane engine for the host build: groups of 16 lanes, every lane of the
// block calling (the values pass through one shared array between two barriers over all lanes).
#pragma once
#include "lane_shim.h"

static uint32_t g_group_xchg[1024];
static inline uint32_t emu_group_xchg(uint32_t v, unsigned src) {
    g_group_xchg[threadIdx.x] = v;
    g_lanes->arrive_and_wait();
    const uint32_t r = g_group_xchg[src];
    g_lanes->arrive_and_wait();
    return r;
}
static inline int __shfl_up_sync(unsigned mask, int v, unsigned d, int width) {
    if (mask != 0xffffffffu || width != 16) std::abort();
    const unsigned L = threadIdx.x, l = L & 15;
    return (int)emu_group_xchg((uint32_t)v, l >= d ? L - d : L);
}
static inline uint32_t __shfl_sync(unsigned mask, uint32_t v, int src, int width) {
    if (mask != 0xffffffffu || width != 16) std::abort();
    return emu_group_xchg(v, (threadIdx.x & ~15u) + (unsigned)src);
}
