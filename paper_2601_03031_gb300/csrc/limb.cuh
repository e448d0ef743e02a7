// Fq arithmetic with one limb per lane, for latency: sums of products of Fq values on 16 lanes each.
//
// A product per lane is a chain of 300 multiply-adds (fp.cuh), about 2.0 k cycles for a warp however idle
// the GPU is, and every addition around it another 24 carries.  Here a value is 15 signed limbs of 26 bits
// on 15 of the 16 lanes of a slot, so an addition is one instruction without carries, and a lane forms
// one column of a product with 15 multiply-adds into a 64-bit sum.  What is computed is
//     out = sum_{t < n} x_t y_t  2^-390  +  addend   (mod p)
// with one reduction for the whole sum, so that an Fq12 operation needs no recombination of products
// afterwards: every output component is one such sum.
//   columns:   lane l holds T_l and T_{15 + l} of T = sum_t x_t y_t.  At step s it multiplies x's limb
//              (l - s) mod 15 by y's limb s; the sum after step l is T_l, what is added later T_{15 + l}.
//              x is read from a window of 30 words (its limbs twice), y by broadcast.
//   reduction: the 13 lowest columns, their carries passed one and two lanes up (27-bit limbs u_k
//              then), are folded by c_k = 2^(26 k - 338) mod p: S = (T >> 338) + sum_k u_k c_k; a
//              two-limb Montgomery step, m = -S p^-1 mod 2^52, gives out = (S + m p) / 2^52.  Lane l
//              forms column l + 2 of S, which is its own T_{15 + l} and lands in its own output column;
//              lanes 13 and 14, whose own low columns are T_13 and T_14, form S's columns 0 and 1.
// Bounds: limbs are at most 27 bits (signed), sums of two 28; every column stays below 2^63 for
// 15 n 2^(bits of x's and y's limbs) < 2^63.  The value lies in (-d, p + d), d = sum |x_t y_t| / 2^390
// (p^2 / 2^390 is p / 632): it is not canonical, limb_canon makes it so.  An addend is not reduced with
// the sum, so one that depends on the value before it has to be brought near zero first (limb_near_zero).
#pragma once
#include "fp.cuh"

constexpr int LIMB_BITS = 26, LIMB_N = 15, LIMB_MASK = (1 << LIMB_BITS) - 1;
constexpr int LIMB_ROW = 16;       // words of a value (the 16th unused): 16-byte aligned for broadcasts
constexpr int LIMB_WIN = 32;       // words of a window: the limbs twice

struct LimbLane {
    int l;                         // lane of the slot, 0 .. 15 (lane 15 holds nothing)
    int32_t c[13];                 // fold constants of this lane's column of S
    int32_t pa, pb, pl;            // p's limbs l + 2, l + 1 and l
    uint32_t at[LIMB_N];           // all-ones at s = l: takes the sum after step l in one logic
                                   // instruction per word (a compare and two selects cost 6 cycles)
};

FPG_DEV LimbLane limb_lane() {
    LimbLane k;
    k.l = (int)(threadIdx.x & 15);
#pragma unroll
    for (int i = 0; i < 13; i++) k.c[i] = LIMB_FOLD[k.l][i];
    k.pa = LIMB_P[k.l][0];
    k.pb = LIMB_P[k.l][1];
    k.pl = LIMB_P[k.l][2];
#pragma unroll
    for (int s = 0; s < LIMB_N; s++) {
        k.at[s] = s == k.l ? 0xffffffffu : 0u;
#ifndef FPG_PRIMITIVES_EXTERNAL
        asm volatile("" : "+r"(k.at[s]));      // kept in a register, not formed again at each use
#endif
    }
    return k;
}

// limb l of a 12-word value (the words at x)
FPG_DEV int32_t limb_of_words(const uint32_t* x, int l) {
    const int w = LIMB_BITS * l >> 5, o = LIMB_BITS * l & 31;
    if (l >= LIMB_N) return 0;
    return (int32_t)(__funnelshift_r(x[w], w + 1 < 12 ? x[w + 1] : 0, o) & LIMB_MASK);
}

// a value's limb into its row / window
FPG_DEV void limb_put(int32_t* row, int l, int32_t v) { row[l] = l < LIMB_N ? v : 0; }
FPG_DEV void limb_put_window(int32_t* win, int l, int32_t v) {
    if (l < LIMB_N) {
        win[l] = v;
        win[LIMB_N + l] = v;
    }
}

struct alignas(16) limb4 { int32_t x[4]; };

// T_l (lo) and T_{15 + l} (hi) of sum_t x_t y_t: the y_t's rows at y[t], the x_t's windows at win[t]
template <int NT>
FPG_DEV void limb_dot(const LimbLane& k, int64_t& lo, int64_t& hi, const int32_t* const (&y)[NT],
                      const int32_t* const (&win)[NT]) {
    int64_t acc = 0;
    uint32_t klo = 0, khi = 0;
    const int32_t* x[NT];
#pragma unroll
    for (int t = 0; t < NT; t++) x[t] = win[t] + LIMB_N + k.l;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        limb4 v[NT];
#pragma unroll
        for (int t = 0; t < NT; t++) v[t] = reinterpret_cast<const limb4*>(y[t])[q];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int s = 4 * q + r;
            if (s == LIMB_N) break;
#pragma unroll
            for (int t = 0; t < NT; t++) acc += (int64_t)x[t][-s] * v[t].x[r];
            klo |= (uint32_t)acc & k.at[s];
            khi |= (uint32_t)((uint64_t)acc >> 32) & k.at[s];
        }
    }
    lo = (int64_t)(((uint64_t)khi << 32) | klo);
    hi = acc - lo;
}

// column l of the reduced value, before its carries; u: 16 words of this slot.  All lanes of the warp.
FPG_DEV int64_t limb_reduce(const LimbLane& k, int64_t lo, int64_t hi, int32_t* u) {
    const int l = k.l;
    const bool low = l < 13;
    const int32_t c1 = low ? (int32_t)(lo >> LIMB_BITS) & LIMB_MASK : 0, c2 = low ? (int32_t)(lo >> (2 * LIMB_BITS)) : 0;
    const int32_t d1 = __shfl_up_sync(0xffffffffu, c1, 1, 16), d2 = __shfl_up_sync(0xffffffffu, c2, 2, 16);
    const int64_t U = (low ? lo & LIMB_MASK : lo) + (l >= 1 ? d1 : 0) + (l >= 2 ? d2 : 0);
    u[l] = (int32_t)U;
    __syncwarp();
    int64_t S = low ? hi : U;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const limb4 v = reinterpret_cast<const limb4*>(u)[q];
#pragma unroll
        for (int r = 0; r < 4; r++)
            if (4 * q + r < 13) S += (int64_t)v.x[r] * k.c[4 * q + r];
    }
    const uint32_t s0l = __shfl_sync(0xffffffffu, (uint32_t)S, 13, 16);
    const uint32_t s0h = __shfl_sync(0xffffffffu, (uint32_t)((uint64_t)S >> 32), 13, 16);
    const uint32_t s1l = __shfl_sync(0xffffffffu, (uint32_t)S, 14, 16);
    const uint32_t s1h = __shfl_sync(0xffffffffu, (uint32_t)((uint64_t)S >> 32), 14, 16);
    const int64_t S0 = (int64_t)(((uint64_t)s0h << 32) | s0l), S1 = (int64_t)(((uint64_t)s1h << 32) | s1l);
    const uint64_t m = ((uint64_t)S0 + ((uint64_t)S1 << LIMB_BITS)) * LIMB_PINV52;
    const int32_t m0 = (int32_t)m & LIMB_MASK, m1 = (int32_t)(m >> LIMB_BITS) & LIMB_MASK;
    // columns 0 and 1 of S + m p are a multiple of 2^52; its quotient is the carry into column 2
    const int64_t e = (S0 + (int64_t)m0 * LIMB_P0) >> LIMB_BITS;
    const int64_t f = (S1 + e + (int64_t)m0 * LIMB_P1 + (int64_t)m1 * LIMB_P0) >> LIMB_BITS;
    return (low ? S : hi) + (int64_t)m0 * k.pa + (int64_t)m1 * k.pb + (l == 0 ? f : 0);
}

// this lane's limb from the columns o (carries passed one and two lanes up, the top limb takes the rest)
FPG_DEV int32_t limb_carry(int64_t o, int l) {
    const int32_t c1 = l < 13 ? (int32_t)(o >> LIMB_BITS) & LIMB_MASK : (int32_t)(o >> LIMB_BITS);
    const int32_t c2 = l < 13 ? (int32_t)(o >> (2 * LIMB_BITS)) : 0;
    const int32_t d1 = __shfl_up_sync(0xffffffffu, c1, 1, 16), d2 = __shfl_up_sync(0xffffffffu, c2, 2, 16);
    return (int32_t)(l < 14 ? o & LIMB_MASK : o) + (l >= 1 ? d1 : 0) + (l >= 2 ? d2 : 0);
}

// this lane's limb of a value minus the multiple of p nearest to it, judged by its top limb (bits from
// 364 on; p >> 364 is 106513): within p / 2 of zero and a 2^-16th
FPG_DEV int32_t limb_near_zero(const LimbLane& k, const int32_t* row) {
    const int32_t q = (int32_t)(((int64_t)row[LIMB_N - 1] * LIMB_PTOP_INV + (1ll << 31)) >> 32);
    return row[k.l] - q * k.pl;
}

// the canonical 12 words of a value in (-p, 2 p) from its row (one lane)
FPG_DEV fq limb_canon(const int32_t* row) {
    uint32_t w[13];
    uint64_t buf = 0;
    int64_t c = 0;
    int nb = 0, k = 0;
#pragma unroll
    for (int i = 0; i < LIMB_N; i++) {                      // the value plus p, packed
        c += (int64_t)row[i] + LIMB_P[i][2];
        buf |= (uint64_t)(i < LIMB_N - 1 ? c & LIMB_MASK : c) << nb;
        c >>= LIMB_BITS;
        nb += LIMB_BITS;
        if (nb >= 32) {
            w[k++] = (uint32_t)buf;
            buf >>= 32;
            nb -= 32;
        }
    }
    fq v;
#pragma unroll
    for (int i = 0; i < 12; i++) v.v[i] = w[i];
#pragma unroll
    for (int r = 0; r < 2; r++) {                           // < 3 p: at most two subtractions
        fq t;
        t.v[0] = ptx::sub_cc(v.v[0], FQ_P[0]);
#pragma unroll
        for (int i = 1; i < 12; i++) t.v[i] = ptx::subc_cc(v.v[i], FQ_P[i]);
        v = fq_select(ptx::subc(0, 0) != 0, v, t);
    }
    return v;
}
