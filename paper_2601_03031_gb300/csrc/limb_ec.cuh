// G1 and G2 with one limb per lane (limb.cuh), for latency.  G1: one scalar multiplication on 96 threads,
// six slots of 16 lanes.
//
// Points are homogeneous projective and every operation uses the complete formulas of Renes, Costello
// and Batina (EUROCRYPT 2016) for a = 0 and b3 = 3 b = 12, in two levels of sums of products:
//   level 1:  t0 = 3 X1 X2, t1 = Y1 Y2, t2 = b3 Z1 Z2, t3 = X1 Y2 + X2 Y1, t4 = Y1 Z2 + Y2 Z1,
//             t5 = b3 (X1 Z2 + X2 Z1)                              one slot each
//   level 2:  X3 = t3 (t1 - t2) - t4 t5,  Y3 = (t1 + t2)(t1 - t2) + t0 t5,  Z3 = t4 (t1 + t2) + t0 t3
// and a doubling (level 1 with both points equal, so t3 = 2 X Y, t4 = 2 Y Z)
//             X3 = t3 (t1 - 3 t2),  Y3 = (t1 - 3 t2)(t1 + t2) + 8 t1 t2,  Z3 = 4 t1 t4.
// On an 8-lane group with one Fq product per lane (group_ec.cuh) an operation is two rounds of products
// and about twenty field additions in sequence, 8.6 k cycles; here the additions are lane-wise.
// A multiplication by k: GLV halves k0, k1 (curve.cuh) in width-4 NAF, P, 3P, 5P, 7P, one accumulator:
// 128 doublings and ~51 additions.  Alone on the GPU's idle SMs it takes 0.19 ms (8-lane groups: 0.78),
// about 2.2 k cycles per operation, half of it in the two reductions.  It issues more than a group does, so with
// many of them the groups win.  A launch of n multiplications, two per block / one per block / groups, in ms:
// 512: 0.26 / 0.26 / 0.79, 1024: 0.42 / 0.51 / 0.79, 2048: 0.74 / 0.97 / 0.79, 4096: 1.39 / 1.76 / 0.99,
// 8192: 2.62 / 3.43 / 1.97, 65536: 20.4 / 26.6 / 13.4.
#pragma once
#include "group_ec.cuh"
#include "limb.cuh"

constexpr int LEC_THREADS = 96, LEC_DIGITS = 132;
// G1 multiplications up to which a launch of them runs two to a block with one limb per lane, above it on 8-lane
// groups (the figures above: 2048 take 0.74 and 0.79 ms, 3072 take 1.11 and 0.99)
constexpr uint64_t LEC_MULS_MAX = 2048;

struct LimbEc {
    alignas(16) int32_t acc[3][LIMB_WIN];          // X, Y, Z of the accumulator, each as a window
    alignas(16) int32_t two[3][LIMB_WIN];          // 2P while the table is built
    alignas(16) int32_t tab[4][4][LIMB_WIN];       // (2 i + 1) P: X, Y, -Y, Z
    alignas(16) int32_t phix[4][LIMB_WIN];         // omega X of the entries: -phi((x, y)) = (omega x, -y)
    alignas(16) int32_t t[6][LIMB_ROW];
    alignas(16) int32_t priv[3][2 * LIMB_WIN + 2 * LIMB_ROW + 16];   // (an odd multiple of 16 words)
    alignas(16) int32_t u[6][LIMB_ROW];
    alignas(16) int32_t zero[LIMB_WIN], one[LIMB_WIN], back[LIMB_WIN], omega[LIMB_WIN];
    fq x[2];
    signed char d[2][LEC_DIGITS];
    int nops;
    unsigned char ops[192];
};

// Barrier of a multiplication's 96 threads: a block may hold several, each on three whole warps.
FPG_DEV int lec_thread() { return (int)(threadIdx.x % LEC_THREADS); }
FPG_DEV void lec_sync() {
#ifdef FPG_PRIMITIVES_EXTERNAL
    __syncthreads();
#else
    asm volatile("bar.sync %0, 96;" ::"r"(1 + (int)(threadIdx.x / LEC_THREADS)) : "memory");
#endif
}

struct LecLane {
    LimbLane k;
    int slot;
    int i, j, scale;                               // level 1: coordinates and factor
};
FPG_DEV LecLane lec_lane() {
    LecLane c;
    c.k = limb_lane();
    const int s = lec_thread() >> 4;
    c.slot = s;
    c.i = s < 3 ? s : s == 4 ? 1 : 0;
    c.j = s < 3 ? s : s == 3 ? 1 : 2;
    c.scale = s == 0 ? 3 : (s == 2 || s == 5) ? 12 : 1;
    return c;
}

// one product x y (x a window, y a row) with one reduction
FPG_DEV int32_t lec_mul1(LimbEc& S, const LecLane& c, const int32_t* y, const int32_t* x) {
    const int32_t *row[1] = {y}, *win[1] = {x};
    int64_t lo, hi;
    limb_dot<1>(c.k, lo, hi, row, win);
    return limb_carry(limb_reduce(c.k, lo, hi, S.u[c.slot]), c.k.l);
}

// acc <- acc + Q for Q's windows qx, qy, qz, or 2 acc for DBL (the windows are then acc's own)
template <bool DBL>
FPG_DEV void lec_step_on(LimbEc& S, const LecLane& c, int32_t (*acc)[LIMB_WIN], const int32_t* qx, const int32_t* qy,
                         const int32_t* qz) {
    const int l = c.k.l, s = c.slot;
    {
        const int32_t* qi = c.i == 0 ? qx : c.i == 1 ? qy : qz;
        const int32_t* qj = c.j == 0 ? qx : c.j == 1 ? qy : qz;
        int64_t lo, hi;
        if (s < 2) {                               // warp 0: squares of coordinates, one product each
            const int32_t *row[1] = {acc[c.i]}, *win[1] = {qi};
            limb_dot<1>(c.k, lo, hi, row, win);
        } else {
            const int32_t *row[2] = {acc[c.i], acc[c.j]}, *win[2] = {qj, s == 2 ? S.zero : qi};
            limb_dot<2>(c.k, lo, hi, row, win);
        }
        lo *= c.scale;
        hi *= c.scale;
        limb_put(S.t[s], l, limb_carry(limb_reduce(c.k, lo, hi, S.u[s]), l));
    }
    lec_sync();
    if (s < 4) {                                   // warps 0 and 1; slot 3 repeats slot 2 and stores nothing
        const int q = s < 3 ? s : 2;
        int32_t* p = S.priv[q];
        int32_t* rows = p + 2 * LIMB_WIN;
        const int32_t t1 = S.t[1][l], t2 = S.t[2][l];
        if (s < 3) {
            if (DBL) {
                limb_put_window(p, l, q < 2 ? t1 - 3 * t2 : 4 * t1);
                limb_put_window(p + LIMB_WIN, l, q == 1 ? t2 : 0);
                rows[LIMB_ROW + l] = 8 * t1;
            } else {
                limb_put_window(p, l, q < 2 ? t1 - t2 : t1 + t2);
                limb_put_window(p + LIMB_WIN, l, q == 0 ? -S.t[4][l] : S.t[0][l]);
            }
            rows[l] = t1 + t2;
        }
        __syncwarp();
        const int32_t *row[2] = {q == 0 ? S.t[3] : q == 1 ? rows : S.t[4], DBL ? rows + LIMB_ROW : q < 2 ? S.t[5] : S.t[3]},
                      *win[2] = {p, p + LIMB_WIN};
        int64_t lo, hi;
        limb_dot<2>(c.k, lo, hi, row, win);
        const int32_t v = limb_carry(limb_reduce(c.k, lo, hi, S.u[s]), l);
        if (s < 3) limb_put_window(acc[s], l, v);
    }
    lec_sync();
}

template <bool DBL>
FPG_DEV void lec_step(LimbEc& S, const LecLane& c, const int32_t* qx, const int32_t* qy, const int32_t* qz) {
    lec_step_on<DBL>(S, c, S.acc, qx, qy, qz);
}

// the width-4 NAF of a 128-bit k, least significant first, into the zeroed d (one lane)
FPG_DEV void lec_naf(signed char* d, const uint32_t* k) {
    uint64_t lo = ((uint64_t)k[1] << 32) | k[0], hi = ((uint64_t)k[3] << 32) | k[2];
    uint32_t ex = 0;                               // bit 128
    for (int i = 0; lo | hi | ex;) {
        int sh = 1;
        if (lo & 1) {
            int v = (int)(lo & 15);
            if (v >= 8) {
                v -= 16;
                const uint64_t n = lo + (uint64_t)(-v);
                if (n < lo && ++hi == 0) ex = 1;
                lo = n;
            } else {
                lo -= (uint64_t)v;
            }
            d[i] = (signed char)v;
            sh = 4;
        }
        i += sh;
        lo = (lo >> sh) | (hi << (64 - sh));
        hi = (hi >> sh) | ((uint64_t)ex << (64 - sh));
        ex = 0;
    }
}

// constant windows and an affine P (Montgomery residues, (0, 0) the identity) into the accumulator and the
// table's first entry
FPG_DEV void lec_enter(LimbEc& S, const LecLane& c, const g1a& P) {
    const int l = c.k.l, s = c.slot;
    if (s == 0) limb_put_window(S.zero, l, 0);
    if (s == 1) limb_put_window(S.one, l, LIMB_FROB2[0][l]);
    if (s == 2) limb_put_window(S.back, l, LIMB_CONV[1][l]);
    if (s == 3) limb_put_window(S.omega, l, LIMB_OMEGA[l]);
    // x, y times 2^396 2^-390: from residues times 2^384 to the engine's form
    if (s < 2) limb_put_window(S.acc[s], l, LIMB_CONV[0][l]);
    limb_put(S.t[s], l, s < 2 ? limb_of_words(s == 0 ? P.x.v : P.y.v, l) : 0);
    lec_sync();
    const bool inf = g1a_is_inf(P);
    int32_t v = lec_mul1(S, c, S.t[s], S.acc[s < 2 ? s : 0]);
    const int32_t one = LIMB_FROB2[0][l];
    if (s == 1 && inf) v = one;                    // the identity is (0 : 1 : 0)
    lec_sync();                                    // reads of S.acc are over
    if (s == 2) v = inf ? 0 : one;
    if (s < 3) {
        limb_put_window(S.acc[s], l, v);
        limb_put_window(S.tab[0][s == 2 ? 3 : s], l, v);
        if (s == 1) limb_put_window(S.tab[0][2], l, -v);
    }
    lec_sync();
}
// the digits of the GLV halves of a canonical k < r (8 words) into S.d (visible after the next barrier)
FPG_DEV void lec_digits(LimbEc& S, const LecLane& c, const uint32_t* kw) {
    for (int i = lec_thread(); i < 2 * LEC_DIGITS; i += LEC_THREADS) (&S.d[0][0])[i] = 0;
    lec_sync();
    if (c.k.l == 0 && (c.slot == 0 || c.slot == 2)) {   // one lane of warps 0 and 1
        uint32_t k1[5], k0[4];
        div_by_const<4, 5>(k1, k0, kw, GLV_D, GLV_BARRETT);
        lec_naf(S.d[c.slot >> 1], c.slot ? k1 : k0);
    }
    __syncwarp();
}
// from P in the accumulator and the table's first entry: 2P in S.two, 3P = 2P + P, 5P = 3P + 2P,
// 7P = 5P + 2P in the table, and omega X of the four entries
FPG_DEV void lec_table(LimbEc& S, const LecLane& c) {
    const int l = c.k.l, s = c.slot;
    lec_step<true>(S, c, S.acc[0], S.acc[1], S.acc[2]);
    if (s < 3) limb_put_window(S.two[s], l, S.acc[s][l]);
    lec_sync();
    for (int e = 1; e < 4; e++) {
        if (e == 1) lec_step<false>(S, c, S.tab[0][0], S.tab[0][1], S.tab[0][3]);
        else lec_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
        if (s < 3) {
            const int32_t v = S.acc[s][l];
            limb_put_window(S.tab[e][s == 2 ? 3 : s], l, v);
            if (s == 1) limb_put_window(S.tab[e][2], l, -v);
        }
        lec_sync();
    }
    const int32_t v = lec_mul1(S, c, S.tab[s < 4 ? s : 0][0], S.omega);
    if (s < 4) limb_put_window(S.phix[s], l, v);
    lec_sync();
}
FPG_DEV void lec_set_identity(LimbEc& S, const LecLane& c) {
    if (c.slot < 3) limb_put_window(S.acc[c.slot], c.k.l, c.slot == 1 ? LIMB_FROB2[0][c.k.l] : 0);
    lec_sync();
}

// S.acc <- k P for a canonical k < r (8 words) and an affine P
FPG_DEV void lec_g1_mul(LimbEc& S, const LecLane& c, const g1a& P, const uint32_t* kw) {
    lec_digits(S, c, kw);
    lec_enter(S, c, P);
    lec_table(S, c);
    lec_set_identity(S, c);
    int i = LEC_DIGITS - 1;
    while (i >= 0 && !S.d[0][i] && !S.d[1][i]) i--;
    for (bool first = true; i >= 0; i--) {
        if (!first) lec_step<true>(S, c, S.acc[0], S.acc[1], S.acc[2]);
        first = false;
        for (int h = 0; h < 2; h++) {
            const int d = S.d[h][i];
            if (!d) continue;
            const int e = (d < 0 ? -d : d) >> 1;
            // the half k1 multiplies -phi(P) = (omega x, -y)
            lec_step<false>(S, c, h ? S.phix[e] : S.tab[e][0], S.tab[e][(d < 0) != (h == 1) ? 2 : 1], S.tab[e][3]);
        }
    }
}

// ---- Bases known before their scalar: the chain of doublings is cut into LEC_CUTS pieces.  The tables of
// 2^(CH i) P, i < 4, are formed ahead (lec_pre, lec2_pre: limbs in global memory), and k P is then one
// chain of CH doublings in which every piece's digits are added: ~83 (G1, CH = 32) or ~68 operations (G2,
// CH = 16) instead of ~182 and ~121.  The order of operations is listed first, so that the next table
// entry's limbs are loaded while an operation runs.
constexpr int LEC_CUTS = 4, LEC_CH = 32, LEC2_CH = 16;
constexpr int LEC_PRE_INTS = LEC_CUTS * 4 * 4 * LIMB_ROW;        // (cut, entry, X Y Z omega-X)
constexpr int LEC2_PRE_INTS = LEC_CUTS * 16 * 6 * LIMB_ROW;      // (cut, 4 h + entry, X Y Z parts)

// operations in order: 0 a doubling, else 0x80 | sign 0x40 | (cut, half or digit string h, entry); at most
// one digit in any four of a string is nonzero, so there are at most 2 33 + 36 (G1), 4 17 + 20 (G2).  One lane.
template <int NH, int CH, int LIM>
FPG_DEV int lec_list(unsigned char* ops, const signed char (*d)[LEC_DIGITS]) {
    int n = 0;
    for (int pos = LIM - 1 - 3 * CH; pos >= 0; pos--) {
        if (n) ops[n++] = 0;
#pragma unroll
        for (int q = 0; q < LEC_CUTS * NH; q++) {
            const int cut = q / NH, h = q % NH;
            if (pos >= CH && cut < LEC_CUTS - 1) continue;
            const int v = d[h][CH * cut + pos];
            if (v) ops[n++] = (unsigned char)(0x80 | (v < 0 ? 0x40 : 0) | (cut << 4) | (h << 2) | ((v < 0 ? -v : v) >> 1));
        }
    }
    return n;
}

FPG_DEV void lec_pre(LimbEc& S, const LecLane& c, const g1a& P, int32_t* T) {
    const int l = c.k.l, s = c.slot;
    lec_enter(S, c, P);
    for (int cut = 0; cut < LEC_CUTS; cut++) {
        lec_table(S, c);
        if (s < 4)
            for (int e = 0; e < 4; e++) {
                const int32_t* w = s == 3 ? S.phix[e] : S.tab[e][s == 2 ? 3 : s];
                T[((cut * 4 + e) * 4 + s) * LIMB_ROW + l] = l < LIMB_N ? w[l] : 0;
            }
        if (cut == LEC_CUTS - 1) break;
        if (s < 3) limb_put_window(S.acc[s], l, S.two[s][l]);
        lec_sync();
        for (int i = 1; i < LEC_CH; i++) lec_step<true>(S, c, S.acc[0], S.acc[1], S.acc[2]);
        if (s < 3) {
            const int32_t v = S.acc[s][l];
            limb_put_window(S.tab[0][s == 2 ? 3 : s], l, v);
            if (s == 1) limb_put_window(S.tab[0][2], l, -v);
        }
        lec_sync();
    }
}
// S.acc <- k P from lec_pre's tables of P
FPG_DEV void lec_g1_mul_pre(LimbEc& S, const LecLane& c, const int32_t* T, const uint32_t* kw) {
    const int l = c.k.l, s = c.slot;
    if (s == 5) limb_put_window(S.zero, l, 0);
    if (s == 4) limb_put_window(S.back, l, LIMB_CONV[1][l]);
    lec_digits(S, c, kw);
    lec_sync();
    if (lec_thread() == 0) S.nops = lec_list<2, LEC_CH, LEC_DIGITS>(S.ops, S.d);
    lec_set_identity(S, c);
    auto limb = [&](int op) -> int32_t {           // slot s < 3's coordinate of the entry
        const int h = (op >> 2) & 1, row = ((op >> 4) & 3) * 16 + (op & 3) * 4 + (s == 0 && h ? 3 : s < 3 ? s : 0);
        const int32_t v = T[row * LIMB_ROW + l];
        return s == 1 && (((op & 0x40) != 0) != (h == 1)) ? -v : v;
    };
    const int n = S.nops;
    int32_t next = n && S.ops[0] ? limb(S.ops[0]) : 0;
    for (int i = 0; i < n; i++) {
        const int op = S.ops[i], nx = i + 1 < n ? S.ops[i + 1] : 0;
        if (op) {
            if (s < 3) limb_put_window(S.two[s], l, next);
            lec_sync();
        }
        if (nx) next = limb(nx);
        if (op) lec_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
        else lec_step<true>(S, c, S.acc[0], S.acc[1], S.acc[2]);
    }
}

// S.acc as Jacobian (X Z, Y Z^2, Z) residues times 2^384: component s is returned on slot s's first lane
FPG_DEV fq lec_jacobian(LimbEc& S, const LecLane& c) {
    const int l = c.k.l, s = c.slot, q = s < 3 ? s : 0;
    int32_t v = lec_mul1(S, c, S.acc[q], q < 2 ? S.acc[2] : S.one);
    limb_put(S.t[s], l, v);
    __syncwarp();
    v = lec_mul1(S, c, S.t[s], s == 1 ? S.acc[2] : S.one);
    limb_put(S.t[s], l, v);
    __syncwarp();
    v = lec_mul1(S, c, S.t[s], S.back);
    limb_put(S.t[s], l, v);
    __syncwarp();
    fq r;
    fq_zero(r);
    if (l == 0 && s < 3) r = limb_canon(S.t[s]);
    return r;
}


// S.acc <- S.acc + P for an affine P
FPG_DEV void lec_add_affine(LimbEc& S, const LecLane& c, const g1a& P) {
    const int l = c.k.l, s = c.slot;
    const bool inf = g1a_is_inf(P);
    limb_put_window(S.two[s < 2 ? s : 2], l, LIMB_CONV[0][l]);
    limb_put(S.t[s], l, s < 2 ? limb_of_words(s == 0 ? P.x.v : P.y.v, l) : 0);
    __syncwarp();
    int32_t v = lec_mul1(S, c, S.t[s], S.two[s < 2 ? s : 2]);
    if (s == 2) v = inf ? 0 : LIMB_FROB2[0][l];
    if (s == 1 && inf) v = LIMB_FROB2[0][l];
    lec_sync();
    if (s < 3) limb_put_window(S.two[s], l, v);
    lec_sync();
    lec_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
}

// S.acc as an affine point, x on slot 0's and y on slot 1's first lane; the identity is (0, 0) (the
// inverse of zero is zero).  The inversion runs on the quad of the first four lanes.
FPG_DEV fq lec_affine(LimbEc& S, const LecLane& c) {
    const int l = c.k.l, s = c.slot, q = s < 2 ? s : 0;
    limb_put(S.t[s], l, lec_mul1(S, c, S.acc[2], S.back));
    __syncwarp();
    if (lec_thread() == 0) S.x[0] = limb_canon(S.t[0]);
    lec_sync();
    if (lec_thread() < 4) {
        const fq zi = fq_inv_quad(S.x[0]);
        if (lec_thread() == 0) S.x[1] = zi;
    }
    lec_sync();
    limb_put(S.t[s], l, limb_of_words(S.x[1].v, l));
    if (s == 0) limb_put_window(S.two[0], l, LIMB_CONV[0][l]);
    lec_sync();
    const int32_t zi = lec_mul1(S, c, S.t[s], S.two[0]);
    if (s == 0) limb_put_window(S.two[1], l, zi);
    lec_sync();
    int32_t v = lec_mul1(S, c, S.acc[q], S.two[1]);
    limb_put(S.t[s], l, v);
    __syncwarp();
    v = lec_mul1(S, c, S.t[s], S.back);
    limb_put(S.t[s], l, v);
    __syncwarp();
    fq r;
    fq_zero(r);
    if (l == 0 && s < 2) r = limb_canon(S.t[s]);
    return r;
}

// ---------------------------------------------------------------------------------------
// G2 on a block of 192 threads: slot 2 q + e holds part e of an Fq2 value.  The same formulas with
// b3 = 12 xi, xi = 1 + u; a product of Fq2 values is two products per part, (re) a0 b0 - a1 b1, (im)
// a0 b1 + a1 b0, with the signs and xi's factor taken by the rows (a0, a1, -a1 and, for xi a, a0 - a1,
// a0 + a1, -(a0 + a1)), so that a table point is only its six windows and -Y's two.
//   level 1:  t0 = 3 X1 X2, t1 = Y1 Y2, t2 = 6 xi Z1 Z2, t3 = X1 Y2 + X2 Y1, t4 = Y1 Z2 + Y2 Z1,
//             t5 = 4 xi (X1 Z2 + X2 Z1)    (factors that keep the columns below 2^63)
//   level 2:  X3 = t3 (t1 - 2 t2) - 3 t4 t5,  Y3 = (t1 + 2 t2)(t1 - 2 t2) + 3 t0 t5,
//             Z3 = t4 (t1 + 2 t2) + t0 t3
//   doubling: X3 = t3 (t1 - 6 t2),  Y3 = (t1 + 2 t2)(t1 - 6 t2) + (8 t1)(2 t2),  Z3 = t4 (4 t1).
// A multiplication by k: four GLS digits of 64 bits in width-4 NAF over (2 i + 1) P, i < 4, and their
// images under -psi, psi^2, -psi^3: 64 doublings and ~51 additions.
// ---------------------------------------------------------------------------------------
constexpr int LEC2_THREADS = 192;
// rows of an accumulator coordinate: a0, a1, -a1 and xi's a0 - a1, a0 + a1, -(a0 + a1)
constexpr int LR_0 = 0, LR_1 = 1, LR_N1 = 2, LR_D = 3, LR_S = 4, LR_NS = 5;
constexpr int LEC2_PAIR = 2 * LIMB_WIN + 16;       // the windows of an Fq2 value: part 1's 16 banks apart

struct LimbEc2 {
    alignas(16) int32_t acc[3][6][LIMB_ROW];       // the accumulator's rows
    alignas(16) int32_t win[3][LEC2_PAIR];         // and windows
    alignas(16) int32_t two[3][LEC2_PAIR];         // windows of 2P while the table is built
    alignas(16) int32_t tab[16][4][LEC2_PAIR];     // windows of entry 4 i + e: X, Y, -Y, Z of (2 e + 1) B_i
    alignas(16) int32_t t[6][3][LIMB_ROW];         // level 1: parts 0, 1 and -(part 1)
    alignas(16) int32_t b[3][2][LEC2_PAIR];        // level 2: windows of the second factors
    alignas(16) int32_t a[2][3][LIMB_ROW];         // level 2: formed first factors of Y3 (t1 + 2 t2, 8 t1)
    alignas(16) int32_t u[12][LIMB_ROW];
    alignas(16) int32_t cst[12][2 * LIMB_WIN + 16];   // slots' constant windows
    fq x[6];
    signed char d[4][LEC_DIGITS];
    int nops;
    unsigned char ops[192];
};

FPG_DEV const int32_t* lec2_win(const int32_t* pair, int e) { return pair + (e ? LIMB_WIN + 16 : 0); }
FPG_DEV int32_t* lec2_win(int32_t* pair, int e) { return pair + (e ? LIMB_WIN + 16 : 0); }

struct Lec2Lane {
    LimbLane k;
    int slot, q, e;                                // level 1: t_q's part e
    int i, j, scale;                               // coordinates and factor
    bool xi;
};
// warps 0, 4 and 1, 5 share a sub-partition: t0, t1, t2 take two products, t3, t4, t5 four
FPG_DEV int lec2_q(int w) { return w < 2 ? w : w < 4 ? w + 1 : w == 4 ? 2 : 5; }
FPG_DEV Lec2Lane lec2_lane() {
    Lec2Lane c;
    c.k = limb_lane();
    c.slot = (int)(threadIdx.x >> 4);
    c.q = lec2_q((int)(threadIdx.x >> 5));
    c.e = c.slot & 1;
    c.i = c.q < 3 ? c.q : c.q == 4 ? 1 : 0;
    c.j = c.q < 3 ? c.q : c.q == 3 ? 1 : 2;
    c.scale = c.q == 0 ? 3 : c.q == 2 ? 6 : c.q == 5 ? 4 : 1;
    c.xi = c.q == 2 || c.q == 5;
    return c;
}

// part e's limb of coordinate i of the accumulator into its windows and rows (both slots of a warp)
FPG_DEV void lec2_put_acc(LimbEc2& S, int i, int e, int l, int32_t v) {
    int32_t(*r)[LIMB_ROW] = S.acc[i];
    limb_put_window(lec2_win(S.win[i], e), l, v);
    limb_put(r[e], l, v);
    __syncwarp();
    const int32_t a0 = r[0][l], a1 = r[1][l];
    if (e == 0) {
        limb_put(r[LR_D], l, a0 - a1);
        limb_put(r[LR_N1], l, -a1);
    } else {
        limb_put(r[LR_S], l, a0 + a1);
        limb_put(r[LR_NS], l, -a0 - a1);
    }
}

// NT / 2 Fq2 products' part e: first factors' rows (three each: part 0, part 1, -(part 1)), second
// factors' windows; column before the reduction
template <int NT>
FPG_DEV void lec2_dot(const Lec2Lane& c, int64_t& lo, int64_t& hi, const int32_t (*const (&a)[NT / 2])[LIMB_ROW],
                      const int32_t* const (&b)[NT / 2]) {
    const int32_t *row[NT], *win[NT];
#pragma unroll
    for (int t = 0; t < NT / 2; t++) {
        row[2 * t] = a[t][0];
        win[2 * t] = lec2_win(b[t], c.e);
        row[2 * t + 1] = a[t][c.e ? 1 : 2];
        win[2 * t + 1] = lec2_win(b[t], 1 - c.e);
    }
    limb_dot<NT>(c.k, lo, hi, row, win);
}

// acc <- acc + Q for Q's coordinates' windows, or 2 acc for DBL (the windows are then acc's own)
template <bool DBL>
FPG_DEV void lec2_step(LimbEc2& S, const Lec2Lane& c, const int32_t* qx, const int32_t* qy, const int32_t* qz) {
    const int l = c.k.l, s = c.slot;
    {
        const int32_t* qi = c.i == 0 ? qx : c.i == 1 ? qy : qz;
        const int32_t* qj = c.j == 0 ? qx : c.j == 1 ? qy : qz;
        // xi a's rows (a0 - a1, a0 + a1, -(a0 + a1)) follow a's three
        const int32_t(*pi)[LIMB_ROW] = S.acc[c.i] + (c.xi ? LR_D : LR_0);
        const int32_t(*pj)[LIMB_ROW] = S.acc[c.j] + (c.xi ? LR_D : LR_0);
        int64_t lo, hi;
        if (c.q < 3) {
            const int32_t(*a[1])[LIMB_ROW] = {pi};
            const int32_t* b[1] = {qi};
            lec2_dot<2>(c, lo, hi, a, b);
        } else {
            const int32_t(*a[2])[LIMB_ROW] = {pi, pj};
            const int32_t* b[2] = {qj, qi};
            lec2_dot<4>(c, lo, hi, a, b);
        }
        lo *= c.scale;
        hi *= c.scale;
        const int32_t v = limb_carry(limb_reduce(c.k, lo, hi, S.u[s]), l);
        limb_put(S.t[c.q][c.e], l, v);
        if (c.e) limb_put(S.t[c.q][2], l, -v);
    }
    __syncthreads();
    if (s < 6) {                                   // warps 0, 1, 2: X3, Y3, Z3
        const int q = s >> 1, e = c.e;
        const int32_t t1 = S.t[1][e][l], t2 = S.t[2][e][l];
        int32_t b1, b2 = 0;
        if (DBL) {
            const int32_t m6 = limb_carry((int64_t)t1 - 6 * (int64_t)t2, l), k8 = limb_carry(8 * (int64_t)t1, l);
            b1 = q < 2 ? m6 : 4 * t1;
            b2 = 2 * t2;
            if (q == 1) {
                limb_put(S.a[1][e], l, k8);
                if (e) limb_put(S.a[1][2], l, -k8);
            }
        } else {
            b1 = q < 2 ? t1 - 2 * t2 : t1 + 2 * t2;
            b2 = q == 0 ? -3 * S.t[4][e][l] : (q == 1 ? 3 : 1) * S.t[0][e][l];
        }
        limb_put_window(lec2_win(S.b[q][0], e), l, b1);
        limb_put_window(lec2_win(S.b[q][1], e), l, b2);
        if (q == 1) {
            limb_put(S.a[0][e], l, t1 + 2 * t2);
            if (e) limb_put(S.a[0][2], l, -t1 - 2 * t2);
        }
        __syncwarp();
        int64_t lo, hi;
        const int32_t(*a0)[LIMB_ROW] = q == 0 ? S.t[3] : q == 1 ? S.a[0] : S.t[4];
        if (DBL && q != 1) {
            const int32_t(*a[1])[LIMB_ROW] = {a0};
            const int32_t* b[1] = {S.b[q][0]};
            lec2_dot<2>(c, lo, hi, a, b);
        } else {
            const int32_t(*a[2])[LIMB_ROW] = {a0, DBL ? S.a[1] : q < 2 ? S.t[5] : S.t[3]};
            const int32_t* b[2] = {S.b[q][0], S.b[q][1]};
            lec2_dot<4>(c, lo, hi, a, b);
        }
        lec2_put_acc(S, q, e, l, limb_carry(limb_reduce(c.k, lo, hi, S.u[s]), l));
    }
    __syncthreads();
}

// the Fq2 product of rows a (three) and windows b, part c.e (both slots of a warp)
FPG_DEV int32_t lec2_mul(LimbEc2& S, const Lec2Lane& c, const int32_t (*a)[LIMB_ROW], const int32_t* b) {
    const int32_t(*aa[1])[LIMB_ROW] = {a};
    const int32_t* bb[1] = {b};
    int64_t lo, hi;
    lec2_dot<2>(c, lo, hi, aa, bb);
    return limb_carry(limb_reduce(c.k, lo, hi, S.u[c.slot]), c.k.l);
}
// one product of a row and a window
FPG_DEV int32_t lec2_mul1(LimbEc2& S, const Lec2Lane& c, const int32_t* y, const int32_t* x) {
    const int32_t *row[1] = {y}, *win[1] = {x};
    int64_t lo, hi;
    limb_dot<1>(c.k, lo, hi, row, win);
    return limb_carry(limb_reduce(c.k, lo, hi, S.u[c.slot]), c.k.l);
}
// component s of an affine point (x0, x1, y0, y1; s < 4) from a residue times 2^384, on slot s
FPG_DEV int32_t lec2_load(LimbEc2& S, const Lec2Lane& c, const fq& w) {
    const int l = c.k.l, s = c.slot;
    int32_t* p = S.cst[s];
    limb_put_window(p, l, LIMB_CONV[0][l]);
    limb_put(p + LIMB_WIN, l, s < 4 ? limb_of_words(w.v, l) : 0);
    __syncwarp();
    const int32_t v = lec2_mul1(S, c, p + LIMB_WIN, p);
    __syncwarp();
    return v;
}
// the component of an affine point that slot s loads
FPG_DEV const fq& lec2_comp(const g2a& P, int s) { return s == 0 ? P.x.c0 : s == 1 ? P.x.c1 : s == 2 ? P.y.c0 : P.y.c1; }

// an affine P into the accumulator and the table's first entry
FPG_DEV void lec2_enter(LimbEc2& S, const Lec2Lane& c, const g2a& P) {
    const int l = c.k.l, s = c.slot;
    const bool inf = g2a_is_inf(P);
    const int32_t one = LIMB_FROB2[0][l];
    int32_t v = lec2_load(S, c, lec2_comp(P, s));
    if (s >= 4) v = s == 4 && !inf ? one : 0;      // Z = 1, or (0 : 1 : 0)
    if (s == 2 && inf) v = one;
    if (s < 6) {
        const int i = s >> 1;
        lec2_put_acc(S, i, c.e, l, v);
        limb_put_window(lec2_win(S.tab[0][i == 2 ? 3 : i], c.e), l, v);
        if (i == 1) limb_put_window(lec2_win(S.tab[0][2], c.e), l, -v);
    }
    __syncthreads();
}
// the digits of the four GLS parts of a canonical k < r (visible after the next barrier)
FPG_DEV void lec2_digits(LimbEc2& S, const Lec2Lane& c, const uint32_t* kw) {
    const int s = c.slot;
    for (int i = (int)threadIdx.x; i < 4 * LEC_DIGITS; i += LEC2_THREADS) (&S.d[0][0])[i] = 0;
    __syncthreads();
    if (c.k.l == 0 && c.e == 0 && s < 8) {         // one lane of warps 0 .. 3
        uint32_t dg[4][2], w[4] = {0, 0, 0, 0};
        gls_digits(dg, kw);
        const int h = s >> 1;
        w[0] = h == 0 ? dg[0][0] : h == 1 ? dg[1][0] : h == 2 ? dg[2][0] : dg[3][0];
        w[1] = h == 0 ? dg[0][1] : h == 1 ? dg[1][1] : h == 2 ? dg[2][1] : dg[3][1];
        lec_naf(S.d[h], w);
    }
    __syncwarp();
}
// from P in the accumulator and the table's first entry: 2P in S.two, 3P, 5P, 7P, and the four entries'
// images B_{i + 1} = -psi(B_i)
FPG_DEV void lec2_table(LimbEc2& S, const Lec2Lane& c) {
    const int l = c.k.l, s = c.slot;
    lec2_step<true>(S, c, S.win[0], S.win[1], S.win[2]);
    if (s < 6) limb_put_window(lec2_win(S.two[s >> 1], c.e), l, S.acc[s >> 1][c.e][l]);
    __syncthreads();
    for (int m = 1; m < 4; m++) {
        if (m == 1) lec2_step<false>(S, c, S.tab[0][0], S.tab[0][1], S.tab[0][3]);
        else lec2_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
        if (s < 6) {
            const int i = s >> 1;
            const int32_t w = S.acc[i][c.e][l];
            limb_put_window(lec2_win(S.tab[m][i == 2 ? 3 : i], c.e), l, w);
            if (i == 1) limb_put_window(lec2_win(S.tab[m][2], c.e), l, -w);
        }
        __syncthreads();
    }
    // -psi: (cx conj(X) : -cy conj(Y) : conj(Z)); conj(a) g: a0 g0 + a1 g1, a0 g1 - a1 g0.
    // Warp w: entry w / 2 of a pass's three, X or Y by w % 2
    const int w = s >> 1, xy = w & 1;
    const int32_t g0 = LIMB_PSI[2 * xy][l], g1 = LIMB_PSI[2 * xy + 1][l];
    int32_t* cw = S.cst[s];
    limb_put_window(cw, l, c.e ? g1 : g0);
    limb_put_window(cw + LIMB_WIN, l, c.e ? -g0 : g1);
    __syncwarp();
    for (int i = 0; i < 3; i++) {
        for (int pass = 0; pass < 2; pass++) {
            const int m = 3 * pass + (w >> 1), mm = m < 4 ? m : 0;
            const int32_t(*src)[LEC2_PAIR] = S.tab[4 * i + mm];
            const int32_t *row[2] = {lec2_win(src[xy], 0), lec2_win(src[xy], 1)}, *win[2] = {cw, cw + LIMB_WIN};
            int64_t lo, hi;
            limb_dot<2>(c.k, lo, hi, row, win);
            const int32_t x = limb_carry(limb_reduce(c.k, lo, hi, S.u[s]), l);
            if (m < 4) {
                int32_t(*dst)[LEC2_PAIR] = S.tab[4 * i + 4 + m];
                limb_put_window(lec2_win(dst[xy], c.e), l, xy ? -x : x);
                if (xy) limb_put_window(lec2_win(dst[2], c.e), l, x);
                else {
                    const int32_t z = lec2_win(src[3], c.e)[l];
                    limb_put_window(lec2_win(dst[3], c.e), l, c.e ? -z : z);
                }
            }
        }
        __syncthreads();
    }
}
FPG_DEV void lec2_set_identity(LimbEc2& S, const Lec2Lane& c) {
    if (c.slot < 6) lec2_put_acc(S, c.slot >> 1, c.e, c.k.l, c.slot == 2 ? LIMB_FROB2[0][c.k.l] : 0);
    __syncthreads();
}

// S.acc <- k P for a canonical k < r (8 words) and an affine P (Montgomery residues, (0, 0) the identity)
FPG_DEV void lec2_g2_mul(LimbEc2& S, const Lec2Lane& c, const g2a& P, const uint32_t* kw) {
    lec2_digits(S, c, kw);
    lec2_enter(S, c, P);
    lec2_table(S, c);
    lec2_set_identity(S, c);
    int i = LEC_DIGITS - 1;
    while (i >= 0 && !S.d[0][i] && !S.d[1][i] && !S.d[2][i] && !S.d[3][i]) i--;
    for (bool first = true; i >= 0; i--) {
        if (!first) lec2_step<true>(S, c, S.win[0], S.win[1], S.win[2]);
        first = false;
        for (int h = 0; h < 4; h++) {
            const int d = S.d[h][i];
            if (!d) continue;
            const int32_t(*t)[LEC2_PAIR] = S.tab[4 * h + ((d < 0 ? -d : d) >> 1)];
            lec2_step<false>(S, c, t[0], t[d < 0 ? 2 : 1], t[3]);
        }
    }
}

// tables of 2^(16 i) P, i < 4 (see lec_pre)
FPG_DEV void lec2_pre(LimbEc2& S, const Lec2Lane& c, const g2a& P, int32_t* T) {
    const int l = c.k.l, s = c.slot;
    lec2_enter(S, c, P);
    for (int cut = 0; cut < LEC_CUTS; cut++) {
        lec2_table(S, c);
        if (s < 6)
            for (int e = 0; e < 16; e++) {
                const int i = s >> 1;
                T[((cut * 16 + e) * 6 + s) * LIMB_ROW + l] = l < LIMB_N ? lec2_win(S.tab[e][i == 2 ? 3 : i], c.e)[l] : 0;
            }
        if (cut == LEC_CUTS - 1) break;
        if (s < 6) lec2_put_acc(S, s >> 1, c.e, l, lec2_win(S.two[s >> 1], c.e)[l]);
        __syncthreads();
        for (int i = 1; i < LEC2_CH; i++) lec2_step<true>(S, c, S.win[0], S.win[1], S.win[2]);
        if (s < 6) {
            const int i = s >> 1;
            const int32_t v = S.acc[i][c.e][l];
            limb_put_window(lec2_win(S.tab[0][i == 2 ? 3 : i], c.e), l, v);
            if (i == 1) limb_put_window(lec2_win(S.tab[0][2], c.e), l, -v);
        }
        __syncthreads();
    }
}
// S.acc <- k P from lec2_pre's tables of P
FPG_DEV void lec2_g2_mul_pre(LimbEc2& S, const Lec2Lane& c, const int32_t* T, const uint32_t* kw) {
    const int l = c.k.l, s = c.slot;
    lec2_digits(S, c, kw);
    __syncthreads();
    if (threadIdx.x == 0) S.nops = lec_list<4, LEC2_CH, 68>(S.ops, S.d);
    lec2_set_identity(S, c);
    auto limb = [&](int op) -> int32_t {           // slot s < 6's part of the entry
        const int32_t v = T[((((op >> 4) & 3) * 16 + (op & 15)) * 6 + (s < 6 ? s : 0)) * LIMB_ROW + l];
        return (s >> 1) == 1 && (op & 0x40) ? -v : v;
    };
    const int n = S.nops;
    int32_t next = n && S.ops[0] ? limb(S.ops[0]) : 0;
    for (int i = 0; i < n; i++) {
        const int op = S.ops[i], nx = i + 1 < n ? S.ops[i + 1] : 0;
        if (op) {
            if (s < 6) limb_put_window(lec2_win(S.two[s >> 1], c.e), l, next);
            __syncthreads();
        }
        if (nx) next = limb(nx);
        if (op) lec2_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
        else lec2_step<true>(S, c, S.win[0], S.win[1], S.win[2]);
    }
}

// S.acc <- S.acc + P for an affine P
FPG_DEV void lec2_add_affine(LimbEc2& S, const Lec2Lane& c, const g2a& P) {
    const int l = c.k.l, s = c.slot;
    const bool inf = g2a_is_inf(P);
    const int32_t one = LIMB_FROB2[0][l];
    int32_t v = lec2_load(S, c, lec2_comp(P, s));
    if (s >= 4) v = s == 4 && !inf ? one : 0;
    if (s == 2 && inf) v = one;
    if (s < 6) limb_put_window(lec2_win(S.two[s >> 1], c.e), l, v);
    __syncthreads();
    lec2_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
}

// S.acc as an affine point, component s < 4 on slot s's first lane; the identity is (0, 0) (the inverse
// of zero is zero).  The inversion runs on the quad of lanes 0 .. 3 of the block.
FPG_DEV fq lec2_affine(LimbEc2& S, const Lec2Lane& c) {
    const int l = c.k.l, s = c.slot;
    int32_t* p = S.cst[s];
    auto to_words = [&](const int32_t* row) {      // residues times 2^384, on the slot's first lane
        limb_put_window(p, l, LIMB_CONV[1][l]);
        __syncwarp();
        const int32_t v = lec2_mul1(S, c, row, p);
        __syncwarp();
        limb_put(p, l, v);
        __syncwarp();
        fq r;
        fq_zero(r);
        if (l == 0) r = limb_canon(p);
        __syncwarp();
        return r;
    };
    const fq z = to_words(S.acc[2][c.e]);
    if (l == 0 && s < 2) S.x[s] = z;
    __syncthreads();
    if (threadIdx.x < 4) {
        const fq2 zz{S.x[0], S.x[1]};
        const fq2 zi = fq2_inv_quad(zz);
        if (threadIdx.x == 0) {
            S.x[2] = zi.c0;
            S.x[3] = zi.c1;
        }
    }
    __syncthreads();
    const int32_t v = lec2_load(S, c, S.x[2 + c.e]);        // slots 0 and 1 (and 2, 3 the same)
    if (s < 2) limb_put_window(lec2_win(S.two[0], c.e), l, v);
    __syncthreads();
    const int32_t w = lec2_mul(S, c, S.acc[s < 4 ? s >> 1 : 0], S.two[0]);
    limb_put(S.t[s >> 1][c.e], l, w);
    __syncwarp();
    return to_words(S.t[s >> 1][c.e]);
}
