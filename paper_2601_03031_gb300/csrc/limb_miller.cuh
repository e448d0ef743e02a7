// The Miller loop with one limb per lane (limb.cuh): a block of 352 threads per pair, 22 slots of 16
// lanes.  Twelve slots hold f's components (flat as Fq2[w]/(w^6 - xi)), ten the two parts of five Fq2
// values of the point's chain.  The formulas are those of miller_loop (pairing.cuh); the point runs a round
// ahead of f, so a doubling step is two rounds, each one sum of products per slot:
//   round 1:  g = f^2  |  from XX, YY, bz = 4 xi ZZ, YZ, XY of T:  X' = 2 XY (YY - 9 bz),
//             Y' = (YY + 9 bz)^2 - 108 bz^2, Z' = 8 YY YZ, and the line l0 = YY - 3 bz, l2 = -3 xP XX,
//             l3 = 2 yP YZ
//   round 2:  f = g (l0 + l2 w^2 + l3 w^3)  |  XX, YY, bz, YZ, XY of the new T
// and the five addition steps four rounds and a priming one.  Bound by issue: a round's 11 warps are three
// on most sub-partitions (2.8 k cycles per doubling step's round with one block on the SM, 0.205 ms for the
// loop; with one Fq product per lane and field additions between, 0.42 ms).
#pragma once
#include "limb12.cuh"
#include "pairing.cuh"

constexpr int LM_THREADS = 352;
constexpr int LM_PAIR = 2 * LIMB_WIN + 16;         // the windows of an Fq2 value: part 1's 16 banks apart

// Windows of NJ coefficients as the second factors of Fq12 products: b0, b0 - b1 of each, then, 16 banks
// apart, b1, -b1, b0 + b1, -(b0 + b1) of each.  lm_win: the one that multiplies part `part` of the
// first factor's coefficient for part e of the product (tw: times xi).
template <int NJ> struct LmWindows {
    static constexpr int W1 = 2 * NJ * LIMB_WIN + 16, WORDS = W1 + 4 * NJ * LIMB_WIN;
};
template <int NJ>
FPG_DEV int lm_win(int j, bool tw, int e, int part) {
    const int w0 = 2 * j * LIMB_WIN, w1 = LmWindows<NJ>::W1 + 4 * j * LIMB_WIN;
    if (part == 0) return e == 0 ? (tw ? w0 + LIMB_WIN : w0) : (tw ? w1 + 2 * LIMB_WIN : w1);
    return e == 0 ? (tw ? w1 + 3 * LIMB_WIN : w1 + LIMB_WIN) : (tw ? w0 + LIMB_WIN : w0);
}
// coefficient j's windows from its parts' limbs, the work of its two slots e = 0, 1
template <int NJ>
FPG_DEV void lm_put_windows(int32_t* w, int j, int e, int l, int32_t b0, int32_t b1) {
    int32_t* w0 = w + 2 * j * LIMB_WIN;
    int32_t* w1 = w + LmWindows<NJ>::W1 + 4 * j * LIMB_WIN;
    if (e == 0) {
        limb_put_window(w0, l, b0);
        limb_put_window(w0 + LIMB_WIN, l, b0 - b1);
        limb_put_window(w1 + 3 * LIMB_WIN, l, -b0 - b1);
    } else {
        limb_put_window(w1, l, b1);
        limb_put_window(w1 + LIMB_WIN, l, -b1);
        limb_put_window(w1 + 2 * LIMB_WIN, l, b0 + b1);
    }
}

struct LmFq2 {                                     // an Fq2 value as first and second factor of products
    alignas(16) int32_t r[3][LIMB_ROW];            // rows of a0, a1, -a1
    alignas(16) int32_t w[LM_PAIR];                // windows of a0, a1
};
struct LimbMiller {
    alignas(16) int32_t f[2][L12_VALUE];           // f and 2 f
    alignas(16) int32_t g[L12_VALUE];              // f^2
    alignas(16) int32_t fw[LmWindows<6>::WORDS];         // windows of f
    alignas(16) int32_t lw[LmWindows<3>::WORDS];         // windows of the line's l0, l2, l3
    alignas(16) int32_t lr[3][2][LIMB_ROW];        // the line's parts
    LmFq2 T[3];                                    // X, Y, Z
    alignas(16) int32_t zx[3][LIMB_ROW];           // xi Z's rows
    alignas(16) int32_t v[5][3][LIMB_ROW];         // XX, YY, bz, YZ, XY (rows as LmFq2)
    LmFq2 a[5];                                    // round 1's formed factors / an addition step's values
    LmFq2 b[4];
    alignas(16) int32_t ln[3][LIMB_ROW];           // -lambda's rows
    LmFq2 q[2];                                    // xQ, yQ
    alignas(16) int32_t cst[4][LIMB_WIN];          // -3 xP, 2 yP, -xP, yP
    alignas(16) int32_t u[22][LIMB_ROW];
};

FPG_DEV const int32_t* lm_w(const LmFq2& a, int e) { return a.w + (e ? LIMB_WIN + 16 : 0); }
// part e's limb of a value (each of its two slots its own part)
FPG_DEV void lm_put(LmFq2& a, int e, int l, int32_t v) {
    limb_put_window(a.w + (e ? LIMB_WIN + 16 : 0), l, v);
    limb_put(a.r[e], l, v);
    if (e) limb_put(a.r[2], l, -v);
}
FPG_DEV void lm_put_rows(int32_t (*r)[LIMB_ROW], int e, int l, int32_t v) {
    limb_put(r[e], l, v);
    if (e) limb_put(r[2], l, -v);
}

struct LmLane {
    LimbLane k;
    int slot, e;
    int kc;                       // f slots: component 2 kc + e; point slots: value 0 .. 4 (the warp)
    bool point, four;             // four: f^2's component is four pairs of coefficients, else three
    int sr[4], sw[8];             // f^2: rows of the pairs' first factors (part 0) and windows
    int gr[3], gw[6];             // f^2 * line: the same
};

FPG_DEV LmLane lm_lane() {
    LmLane c;
    c.k = limb_lane();
    const int s = (int)(threadIdx.x >> 4);
    c.slot = s;
    c.e = s & 1;
    c.point = s >= 12;
    // warps 0 .. 5 hold f's coefficients (3 and 4 pairs alternating over the sub-partitions), 6 .. 10 the point
    c.kc = c.point ? (s - 12) >> 1 : l12_coef(s >> 1);
    const int kc = c.point ? 0 : c.kc;
    c.four = (kc & 1) == 0;
    int n = 0;
#pragma unroll
    for (int t = 0; t < 4; t++) c.sr[t] = 0;
#pragma unroll
    for (int t = 0; t < 8; t++) c.sw[t] = 0;
    // unordered pairs i <= j with i + j = kc or kc + 6; i < j counts twice (rows of 2 f)
#pragma unroll
    for (int i = 0; i < 6; i++) {
#pragma unroll
        for (int j = 0; j < 6; j++) {
            if (j < i || (i + j != kc && i + j != kc + 6)) continue;
            const bool tw = i + j >= 6;
#pragma unroll
            for (int t = 0; t < 4; t++) {
                if (t != n) continue;
                c.sr[t] = (i < j ? L12_VALUE : 0) + 2 * i * LIMB_ROW;
                c.sw[2 * t] = lm_win<6>(j, tw, c.e, 0);
                c.sw[2 * t + 1] = lm_win<6>(j, tw, c.e, 1);
            }
            n++;
        }
    }
    // g_k l0 + g_{k-2} l2 + g_{k-3} l3, the last two times xi when the index wraps
#pragma unroll
    for (int t = 0; t < 3; t++) {
        const int d = t == 0 ? 0 : t + 1;
        const bool tw = kc < d;
        c.gr[t] = 2 * (tw ? kc - d + 6 : kc - d) * LIMB_ROW;
        c.gw[2 * t] = lm_win<3>(t, tw, c.e, 0);
        c.gw[2 * t + 1] = lm_win<3>(t, tw, c.e, 1);
    }
    return c;
}

FPG_DEV int32_t lm_finish(LimbMiller& S, const LmLane& c, int64_t lo, int64_t hi) {
    return limb_carry(limb_reduce(c.k, lo, hi, S.u[c.slot]), c.k.l);
}
// part e of NP products of Fq2 values: rows (part 0, part 1, -(part 1)) and windows
template <int NP>
FPG_DEV void lm_dot(const LmLane& c, int64_t& lo, int64_t& hi, const int32_t (*const (&a)[NP])[LIMB_ROW],
                    const LmFq2* const (&b)[NP]) {
    const int32_t *row[2 * NP], *win[2 * NP];
#pragma unroll
    for (int t = 0; t < NP; t++) {
        row[2 * t] = a[t][0];
        win[2 * t] = lm_w(*b[t], c.e);
        row[2 * t + 1] = a[t][c.e ? 1 : 2];
        win[2 * t + 1] = lm_w(*b[t], 1 - c.e);
    }
    limb_dot<2 * NP>(c.k, lo, hi, row, win);
}
FPG_DEV int32_t lm_mul(LimbMiller& S, const LmLane& c, const int32_t (*a)[LIMB_ROW], const LmFq2& b) {
    const int32_t(*aa[1])[LIMB_ROW] = {a};
    const LmFq2* bb[1] = {&b};
    int64_t lo, hi;
    lm_dot<1>(c, lo, hi, aa, bb);
    return lm_finish(S, c, lo, hi);
}
FPG_DEV int32_t lm_mul2(LimbMiller& S, const LmLane& c, const int32_t (*a0)[LIMB_ROW], const LmFq2& b0,
                        const int32_t (*a1)[LIMB_ROW], const LmFq2& b1) {
    const int32_t(*aa[2])[LIMB_ROW] = {a0, a1};
    const LmFq2* bb[2] = {&b0, &b1};
    int64_t lo, hi;
    lm_dot<2>(c, lo, hi, aa, bb);
    return lm_finish(S, c, lo, hi);
}
// a row times a constant's window
FPG_DEV int32_t lm_scale(LimbMiller& S, const LmLane& c, const int32_t* y, const int32_t* x) {
    const int32_t *row[1] = {y}, *win[1] = {x};
    int64_t lo, hi;
    limb_dot<1>(c.k, lo, hi, row, win);
    return lm_finish(S, c, lo, hi);
}
// the line's coefficient j (0: l0, 1: l2, 2: l3) from its parts' limbs, by the two slots of a warp
FPG_DEV void lm_put_line(LimbMiller& S, const LmLane& c, int j, int32_t v) {
    const int l = c.k.l;
    limb_put(S.lr[j][c.e], l, v);
    __syncwarp();
    const int32_t o = S.lr[j][1 - c.e][l];
    lm_put_windows<3>(S.lw, j, c.e, l, c.e ? o : v, c.e ? v : o);
}
// coordinate i of T; Z with xi Z's rows
FPG_DEV void lm_put_T(LimbMiller& S, const LmLane& c, int i, int32_t v) {
    const int l = c.k.l;
    lm_put(S.T[i], c.e, l, v);
    __syncwarp();
    if (i == 2) {
        const int32_t a0 = S.T[2].r[0][l], a1 = S.T[2].r[1][l];
        if (c.e == 0) limb_put(S.zx[0], l, a0 - a1);
        else {
            limb_put(S.zx[1], l, a0 + a1);
            limb_put(S.zx[2], l, -a0 - a1);
        }
    }
}
// f's component into its rows and windows
FPG_DEV void lm_put_f(LimbMiller& S, const LmLane& c, int32_t v) {
    const int l = c.k.l, o = 2 * c.kc + c.e;
    limb_put(S.f[0] + LIMB_ROW * o, l, v);
    limb_put(S.f[1] + LIMB_ROW * o, l, 2 * v);
    __syncwarp();
    const int32_t p = S.f[0][LIMB_ROW * (o ^ 1) + l];
    lm_put_windows<6>(S.fw, c.kc, c.e, l, c.e ? p : v, c.e ? v : p);
}

// f slots: g = f^2
FPG_DEV void lm_f_sqr(LimbMiller& S, const LmLane& c) {
    int64_t lo, hi;
    const int32_t* base = S.f[0];
    if (c.four) {                                  // warp-uniform
        const int32_t *row[8], *win[8];
#pragma unroll
        for (int t = 0; t < 8; t++) {
            row[t] = base + c.sr[t >> 1] + (t & 1) * LIMB_ROW;
            win[t] = S.fw + c.sw[t];
        }
        limb_dot<8>(c.k, lo, hi, row, win);
    } else {
        const int32_t *row[6], *win[6];
#pragma unroll
        for (int t = 0; t < 6; t++) {
            row[t] = base + c.sr[t >> 1] + (t & 1) * LIMB_ROW;
            win[t] = S.fw + c.sw[t];
        }
        limb_dot<6>(c.k, lo, hi, row, win);
    }
    limb_put(S.g + LIMB_ROW * (2 * c.kc + c.e), c.k.l, lm_finish(S, c, lo, hi));
}
// f slots: f = src * line
FPG_DEV void lm_f_line(LimbMiller& S, const LmLane& c, const int32_t* src) {
    const int32_t *row[6], *win[6];
#pragma unroll
    for (int t = 0; t < 6; t++) {
        row[t] = src + c.gr[t >> 1] + (t & 1) * LIMB_ROW;
        win[t] = S.lw + c.gw[t];
    }
    int64_t lo, hi;
    limb_dot<6>(c.k, lo, hi, row, win);
    const int32_t v = lm_finish(S, c, lo, hi);
    lm_put_f(S, c, v);
}
// point slots: XX, YY, bz = 4 xi ZZ, YZ, XY of T
FPG_DEV void lm_point_squares(LimbMiller& S, const LmLane& c) {
    const int w = c.kc;
    const int32_t(*a[1])[LIMB_ROW] = {w == 0 || w == 4 ? S.T[0].r : w == 2 ? S.zx : S.T[1].r};
    const LmFq2* b[1] = {w == 0 ? &S.T[0] : w == 1 || w == 4 ? &S.T[1] : &S.T[2]};
    int64_t lo, hi;
    lm_dot<1>(c, lo, hi, a, b);
    if (w == 2) {
        lo *= 4;
        hi *= 4;
    }
    lm_put_rows(S.v[w], c.e, c.k.l, lm_finish(S, c, lo, hi));
}
// point slots: 2T and the line from them
FPG_DEV void lm_point_dbl(LimbMiller& S, const LmLane& c) {
    const int w = c.kc, e = c.e, l = c.k.l;
    const int64_t yy = S.v[1][e][l], bz = S.v[2][e][l];
    if (w == 0) {                                  // X' = XY (2 (YY - 9 bz))
        lm_put(S.a[0], e, l, limb_carry(2 * (yy - 9 * bz), l));
        __syncwarp();
        lm_put_T(S, c, 0, lm_mul(S, c, S.v[4], S.a[0]));
    } else if (w == 1) {                           // Y' = (YY + 9 bz)^2 + (-108 bz) bz
        lm_put(S.a[1], e, l, limb_carry(yy + 9 * bz, l));
        lm_put_rows(S.a[2].r, e, l, limb_carry(-108 * bz, l));
        limb_put_window(S.a[2].w + (e ? LIMB_WIN + 16 : 0), l, (int32_t)bz);
        __syncwarp();
        lm_put_T(S, c, 1, lm_mul2(S, c, S.a[1].r, S.a[1], S.a[2].r, S.a[2]));
    } else if (w == 2) {                           // Z' = YZ (8 YY)
        lm_put(S.a[3], e, l, limb_carry(8 * yy, l));
        __syncwarp();
        lm_put_T(S, c, 2, lm_mul(S, c, S.v[3], S.a[3]));
    } else if (w == 3) {                           // l0, l2
        lm_put_line(S, c, 0, limb_carry(yy - 3 * bz, l));
        lm_put_line(S, c, 1, lm_scale(S, c, S.v[0][e], S.cst[0]));
    } else {                                       // l3
        lm_put_line(S, c, 2, lm_scale(S, c, S.v[3][e], S.cst[1]));
    }
}

// the addition step's rounds on the point slots (0: theta, lambda; 1: C, D and the line; 2: E, F, G;
// 3: the new point).  S.a: theta, lambda, C, D; S.v: E, F, G; S.b: H, G - H, E, -E
FPG_DEV void lm_point_add(LimbMiller& S, const LmLane& c, int round) {
    const int w = c.kc, e = c.e, l = c.k.l;
    if (round == 0) {
        if (w < 2) {                               // theta = Y - yQ Z, lambda = X - xQ Z
            const int32_t p = lm_mul(S, c, S.T[2].r, S.q[1 - w]);
            const int32_t v = limb_carry((int64_t)S.T[1 - w].r[e][l] - p, l);
            lm_put(S.a[w], e, l, v);
            if (w == 1) {
                limb_put(S.ln[e], l, -v);
                if (e) limb_put(S.ln[2], l, v);
            }
        }
    } else if (round == 1) {
        if (w < 2) lm_put(S.a[2 + w], e, l, lm_mul(S, c, S.a[w].r, S.a[w]));
        else if (w == 2) lm_put_line(S, c, 0, lm_mul2(S, c, S.a[0].r, S.q[0], S.ln, S.q[1]));
        else if (w == 3) lm_put_line(S, c, 1, lm_scale(S, c, S.a[0].r[e], S.cst[2]));
        else lm_put_line(S, c, 2, lm_scale(S, c, S.a[1].r[e], S.cst[3]));
    } else if (round == 2) {
        if (w < 3) {                               // E = D lambda, F = Z C, G = X D
            const int32_t(*a)[LIMB_ROW] = w == 0 ? S.a[3].r : w == 1 ? S.T[2].r : S.T[0].r;
            lm_put_rows(S.v[w], e, l, lm_mul(S, c, a, w == 0 ? S.a[1] : w == 1 ? S.a[2] : S.a[3]));
        }
    } else if (w < 3) {
        const int64_t E = S.v[0][e][l], F = S.v[1][e][l], G = S.v[2][e][l];
        if (w == 0) {                              // X' = lambda H, H = E + F - 2 G
            lm_put(S.b[0], e, l, limb_carry(E + F - 2 * G, l));
            __syncwarp();
            lm_put_T(S, c, 0, lm_mul(S, c, S.a[1].r, S.b[0]));
        } else if (w == 1) {                       // Y' = theta (G - H) - Y E
            lm_put(S.b[1], e, l, limb_carry(3 * G - E - F, l));
            lm_put(S.b[3], e, l, (int32_t)-E);
            __syncwarp();
            const int32_t v = lm_mul2(S, c, S.a[0].r, S.b[1], S.T[1].r, S.b[3]);
            __syncwarp();
            lm_put_T(S, c, 1, v);
        } else {                                   // Z' = Z E
            lm_put(S.b[2], e, l, (int32_t)E);
            __syncwarp();
            const int32_t v = lm_mul(S, c, S.T[2].r, S.b[2]);
            __syncwarp();
            lm_put_T(S, c, 2, v);
        }
    }
}

// conj(f_{|x|,Q}(P)), 1 when P or Q is the identity: component 2 kc + e as a residue times 2^384 on the
// first lane of f slot (kc, e)
FPG_DEV fq lm_miller(LimbMiller& S, const LmLane& c, g1a P, g2a Q) {
    const int l = c.k.l, e = c.e;
    const bool inf = g1a_is_inf(P) || g2a_is_inf(Q);
    if (inf) {
        P = g1_generator();
        Q = g2_generator();
    }
    const int32_t one = LIMB_FROB2[0][l];
    // inputs times 2^396 2^-390 on the slots 0 .. 5 (xP, yP, xQ, yQ); S.v holds the words' limbs
    int32_t* row = &S.v[0][0][0];
    const fq& in = c.slot == 0 ? P.x : c.slot == 1 ? P.y : c.slot == 2 ? Q.x.c0 : c.slot == 3 ? Q.x.c1 : c.slot == 4 ? Q.y.c0
                                                                                                            : Q.y.c1;
    if (c.slot < 6) limb_put(row + LIMB_ROW * c.slot, l, limb_of_words(in.v, l));
    if (c.slot == 6) limb_put_window(S.cst[0], l, LIMB_CONV[0][l]);
    __syncthreads();
    int32_t v = lm_scale(S, c, row + LIMB_ROW * (c.slot < 6 ? c.slot : 0), S.cst[0]);
    const int32_t m3 = limb_carry(-3 * (int64_t)v, l);     // (of xP, on slot 0)
    __syncthreads();
    if (c.slot == 0) {
        limb_put_window(S.cst[0], l, m3);
        limb_put_window(S.cst[2], l, -v);
    } else if (c.slot == 1) {
        limb_put_window(S.cst[1], l, 2 * v);
        limb_put_window(S.cst[3], l, v);
    } else if (c.slot < 6) {
        const int i = (c.slot - 2) >> 1;
        lm_put(S.q[i], e, l, v);
        lm_put(S.T[i], e, l, v);
    } else if (c.slot < 8) {                       // slots 6, 7: Z = 1
        lm_put_T(S, c, 2, e ? 0 : one);
    }
    __syncthreads();
    if (c.point) lm_point_squares(S, c);
    else lm_put_f(S, c, c.kc == 0 && e == 0 ? one : 0);
    __syncthreads();
    for (int i = 62; i >= 0; i--) {
        if (c.point) lm_point_dbl(S, c);
        else lm_f_sqr(S, c);
        __syncthreads();
        const bool add = (BLS_X_ABS >> i) & 1;
        if (!c.point) lm_f_line(S, c, S.g);
        else if (!add) lm_point_squares(S, c);
        else lm_point_add(S, c, 0);
        __syncthreads();
        if (add) {
            if (c.point) lm_point_add(S, c, 1);
            __syncthreads();
            if (c.point) lm_point_add(S, c, 2);
            else {                                 // f * line reads f's rows of other slots: from a copy
                const int o = LIMB_ROW * (2 * c.kc + e) + l;
                S.g[o] = S.f[0][o];
            }
            __syncthreads();
            if (c.point) lm_point_add(S, c, 3);
            else lm_f_line(S, c, S.g);
            __syncthreads();
            if (c.point && i) lm_point_squares(S, c);
            __syncthreads();
        }
    }
    fq r;
    fq_zero(r);
    // the conjugation (x < 0) by the factor's sign, so that the value stays above -p
    if (c.slot < 2) limb_put_window(S.cst[c.slot], l, e ? -LIMB_CONV[1][l] : LIMB_CONV[1][l]);
    __syncthreads();
    if (!c.point) {
        const int o = 2 * c.kc + e;
        limb_put(S.g + LIMB_ROW * o, l, lm_scale(S, c, S.f[0] + LIMB_ROW * o, S.cst[c.kc & 1]));
        __syncwarp();
        if (l == 0) {
            r = limb_canon(S.g + LIMB_ROW * o);
            if (inf) {
                fq_zero(r);
                if (o == 0) fq_one(r);
            }
        }
    }
    return r;
}
