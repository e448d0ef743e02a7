// Host build of the limb-lane engine (limb.cuh, limb12.cuh): every lane of a block as a host thread.
// Field elements cross as canonical big-endian bytes (Fq12 576 in the tower order of the serialisation).
#include "limb_shim.h"
#include "pairing.cuh"
#include "limb12.cuh"
#include "limb_ec.cuh"
#include "limb_miller.cuh"

#include <vector>

namespace {
fq be_fq(const uint8_t* b) {
    fq a;
    for (int j = 0; j < 12; j++) {
        const uint8_t* p = b + 44 - 4 * j;
        a.v[j] = ((uint32_t)p[0] << 24) | ((uint32_t)p[1] << 16) | ((uint32_t)p[2] << 8) | p[3];
    }
    return fq_to_mont(a);
}
template <typename Fn>
void lanes(int n, Fn fn) {
    std::barrier<> bar(n);
    g_lanes = &bar;
    emu_setup_quads(n);
    emu_setup_warps(n);
    std::vector<std::thread> th;
    for (int lane = 0; lane < n; lane++) th.emplace_back([&, lane] { threadIdx.x = lane; fn(); });
    for (auto& t : th) t.join();
}
int tower_pos(int k) { return (k & 1) ? 3 + (k >> 1) : (k >> 1); }
L12 g_w;
LimbEc g_ec;
LimbMiller g_m;
LimbEc2 g_ec2;
}  // namespace

extern "C" {
// sum of nt products (12 little-endian words per operand, not Montgomery form) times 2^-390 mod p
void emu_limb_dot3(const uint32_t* x, const uint32_t* y, uint32_t* out) {
    lanes(16, [&] {
        const LimbLane k = limb_lane();
        alignas(16) static int32_t win[3][LIMB_WIN], u[16], r[16], row[3][LIMB_ROW];
        const int32_t *w[3] = {win[0], win[1], win[2]}, *y3[3] = {row[0], row[1], row[2]};
        for (int t = 0; t < 3; t++) {
            limb_put_window(win[t], k.l, limb_of_words(x + 12 * t, k.l));
            limb_put(row[t], k.l, limb_of_words(y + 12 * t, k.l));
        }
        __syncwarp();
        int64_t lo, hi;
        limb_dot<3>(k, lo, hi, y3, w);
        limb_put(r, k.l, limb_carry(limb_reduce(k, lo, hi, u), k.l));
        __syncwarp();
        if (k.l == 0) {
            const fq v = limb_canon(r);
            for (int j = 0; j < 12; j++) out[j] = v.v[j];
        }
    });
}
void emu_limb_final_exp(const uint8_t* f_be, uint8_t* out) {
    lanes(L12_THREADS, [&] {
        const L12Lane c = l12_lane();
        const int pos = 2 * tower_pos(c.kc) + c.e;
        l12_load(g_w, c, g_w.v[0], g_w.v[1], be_fq(f_be + 48 * pos));
        l12_final_exp(g_w);
        const fq v = l12_store(g_w, c, g_w.v[L12_FE_RESULT], g_w.v[0]);
        if (c.k.l == 0) fq_to_be(out + 48 * pos, v);
    });
}
// k P (96 bytes in and out, k as 8 little-endian words)
void emu_limb_g1_mul(const uint8_t* p, const uint32_t* k, uint8_t* out) {
    g1a P;
    P.x = be_fq(p);
    P.y = be_fq(p + 48);
    g1j r;
    lanes(LEC_THREADS, [&] {
        const LecLane c = lec_lane();
        lec_g1_mul(g_ec, c, P, k);
        const fq v = lec_jacobian(g_ec, c);
        if (c.k.l == 0 && c.slot < 3) (c.slot == 0 ? r.X : c.slot == 1 ? r.Y : r.Z) = v;
    });
    g1a a;
    jac_to_affine(a.x, a.y, r);
    fq_to_be(out, a.x);
    fq_to_be(out + 48, a.y);
}
// k P + Q on G2 (192 bytes each)
void emu_limb_g2_mul_add(int pre, const uint8_t* p, const uint32_t* k, const uint8_t* q, uint8_t* out) {
    auto pt = [](const uint8_t* b) {
        g2a P;
        P.x.c0 = be_fq(b); P.x.c1 = be_fq(b + 48); P.y.c0 = be_fq(b + 96); P.y.c1 = be_fq(b + 144);
        return P;
    };
    const g2a P = pt(p), Q = pt(q);
    lanes(LEC2_THREADS, [&] {
        const Lec2Lane c = lec2_lane();
        if (pre) {
            static int32_t T[LEC2_PRE_INTS];
            lec2_pre(g_ec2, c, P, T);
            __syncthreads();
            lec2_g2_mul_pre(g_ec2, c, T, k);
        } else {
            lec2_g2_mul(g_ec2, c, P, k);
        }
        lec2_add_affine(g_ec2, c, Q);
        const fq v = lec2_affine(g_ec2, c);
        if (c.k.l == 0 && c.slot < 4) fq_to_be(out + 48 * c.slot, v);
    });
}
// k P + Q on G1, affine
void emu_limb_g1_mul_add(int pre, const uint8_t* p, const uint32_t* k, const uint8_t* q, uint8_t* out) {
    g1a P, Q;
    P.x = be_fq(p); P.y = be_fq(p + 48); Q.x = be_fq(q); Q.y = be_fq(q + 48);
    lanes(LEC_THREADS, [&] {
        const LecLane c = lec_lane();
        if (pre) {
            static int32_t T[LEC_PRE_INTS];
            lec_pre(g_ec, c, P, T);
            __syncthreads();
            lec_g1_mul_pre(g_ec, c, T, k);
        } else {
            lec_g1_mul(g_ec, c, P, k);
        }
        lec_add_affine(g_ec, c, Q);
        const fq v = lec_affine(g_ec, c);
        if (c.k.l == 0 && c.slot < 2) fq_to_be(out + 48 * c.slot, v);
    });
}
void emu_limb_miller(const uint8_t* p, const uint8_t* q, uint8_t* out) {
    g1a P;
    P.x = be_fq(p); P.y = be_fq(p + 48);
    g2a Q;
    Q.x.c0 = be_fq(q); Q.x.c1 = be_fq(q + 48); Q.y.c0 = be_fq(q + 96); Q.y.c1 = be_fq(q + 144);
    lanes(LM_THREADS, [&] {
        const LmLane c = lm_lane();
        const fq v = lm_miller(g_m, c, P, Q);
        if (!c.point && c.k.l == 0) fq_to_be(out + 48 * (2 * tower_pos(c.kc) + c.e), v);
    });
}
}
