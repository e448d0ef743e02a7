// Host build of the Montgomery products of Fq and Fr (fp.cuh) for CPU tests.
#include "lane_shim.h"
#include "fp.cuh"

extern "C" void emu_fq_mul(const uint32_t* a, const uint32_t* b, uint32_t* r) {
    fq x, y;
    std::memcpy(x.v, a, sizeof x.v);
    std::memcpy(y.v, b, sizeof y.v);
    const fq z = fq_mul(x, y);
    std::memcpy(r, z.v, sizeof z.v);
}
extern "C" void emu_fr_mul(const uint32_t* a, const uint32_t* b, uint32_t* r) {
    fr x, y;
    std::memcpy(x.v, a, sizeof x.v);
    std::memcpy(y.v, b, sizeof y.v);
    const fr z = fr_mul(x, y);
    std::memcpy(r, z.v, sizeof z.v);
}
