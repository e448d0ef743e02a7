// Warp-level synchronisation of the limb-lane engine for the host build: __syncwarp and the shuffles on
// groups of 16 lanes as a barrier over the lanes of one warp (warps of a block may take different paths
// between block barriers), the shuffled values through one shared array.
#pragma once
#include "lane_shim.h"

static std::barrier<>* g_warp[32] = {};
static uint32_t g_group_xchg[1024];
static inline void emu_setup_warps(int n) {
    for (int w = 0; w < 32; w++) {
        delete g_warp[w];
        g_warp[w] = 32 * w < n ? new std::barrier<>(n - 32 * w < 32 ? n - 32 * w : 32) : nullptr;
    }
}
static inline void emu_warp_sync() { g_warp[threadIdx.x >> 5]->arrive_and_wait(); }
#define __syncwarp emu_warp_sync
static inline uint32_t emu_group_xchg(uint32_t v, unsigned src) {
    g_group_xchg[threadIdx.x] = v;
    emu_warp_sync();
    const uint32_t r = g_group_xchg[src];
    emu_warp_sync();
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
