// Fq12 operations and the final exponentiation with one limb per lane (limb.cuh): a block of 192
// threads, twelve slots of 16 lanes, slot o holding Fq component o = 2 k + e of a value (flat as
// Fq2[w]/(w^6 - xi), coefficient k of w^k, part e).  Every output component is one sum of products with
// one reduction:
//   product:              12 products (two per coefficient pair; pairs that wrap past w^6 times xi)
//   cyclotomic squaring:  2 or 3 products and +-2 times the component itself
//   Frobenius p / p^2:    2 / 1 products by constants
// The chain of a final exponentiation is ~315 cyclotomic squarings and ~55 products: what counts is one
// operation's latency.  On the 128-thread block engine (warp12.cuh), with each of a squaring's 21 Fq
// products split over four warps and then recombined by field additions, a squaring took 4.0 k cycles and
// the final exponentiation 0.74 ms; here 0.335 ms (one GB300 at 2070 MHz, beside the round's other
// kernels).  It is bound by the issue of the two sub-partitions that hold two of the six warps.
#pragma once
#include "limb.cuh"
#include "tower.cuh"

constexpr int L12_THREADS = 192;
constexpr int L12_VALUE = 12 * LIMB_ROW;                 // words of an Fq12 value
constexpr int L12_WIN0 = 0, L12_WIN1 = 12 * LIMB_WIN + 16;   // windows: read together, so 16 banks apart
constexpr int L12_PRIV = 3 * LIMB_WIN + 3 * LIMB_ROW;    // a slot's windows and rows (odd multiple of 16 words)

struct L12 {
    alignas(16) int32_t v[9][L12_VALUE];                 // values
    alignas(16) int32_t win[12 * L12_PRIV];              // windows of a product, or the slots' own areas
    alignas(16) int32_t u[12][LIMB_ROW];
    fq x[2];                                             // the Fq2 inversion's operand and result
};
static_assert(12 * L12_PRIV >= L12_WIN1 + 24 * LIMB_WIN, "product windows fit");

// a thread's place and its constants of the two frequent operations
struct L12Lane {
    LimbLane k;
    int o, kc, e;                    // component 2 kc + e
    int wofs[12];                    // product: windows of the terms (i, part)
    // cyclotomic squaring: term t is (z[p] + beta z[q]) (gamma z[r] + delta z[s]), then + own * z[o]
    int p[3], q[3], r[3], s[3], beta[3], gamma[3], delta[3], own;
    bool heavy;                      // three terms (the coefficients w^0, w^2, w^4), else two
};

// Coefficient of warp w's two slots.  Warps 0, 4 and 1, 5 share a sub-partition: the two-term ones go
// there first.
FPG_DEV int l12_coef(int w) { return w == 0 ? 1 : w == 1 ? 3 : w == 2 ? 0 : w == 3 ? 2 : w == 4 ? 5 : 4; }

FPG_DEV L12Lane l12_lane() {
    L12Lane c;
    c.k = limb_lane();
    const int kc = l12_coef((int)(threadIdx.x >> 5)), e = (int)(threadIdx.x >> 4) & 1;
    c.kc = kc;
    c.e = e;
    c.o = 2 * kc + e;
    // windows of b: for each coefficient j  b0, b0 - b1 (first group), b1, -b1, b0 + b1, -(b0 + b1)
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const bool tw = i > kc;
        const int j = tw ? kc - i + 6 : kc - i;
        const int b0 = L12_WIN0 + (2 * j) * LIMB_WIN, d = b0 + LIMB_WIN, b1 = L12_WIN1 + (4 * j) * LIMB_WIN,
                  nb1 = b1 + LIMB_WIN, s = b1 + 2 * LIMB_WIN, ns = b1 + 3 * LIMB_WIN;
        c.wofs[2 * i] = e == 0 ? (tw ? d : b0) : (tw ? s : b1);              // times a_i's part 0
        c.wofs[2 * i + 1] = e == 0 ? (tw ? ns : nb1) : (tw ? d : b0);        // times a_i's part 1
    }
    // Granger-Scott: pair (a, b) = (z_n, z_{n+3}); A = a^2 + xi b^2, B = 2 a b;
    // out_0 = 3 A_0 - 2 z_0, out_3 = 3 B_0 + 2 z_3, out_1 = 3 xi B_2 + 2 z_1, out_4 = 3 A_2 - 2 z_4,
    // out_2 = 3 A_1 - 2 z_2, out_5 = 3 B_1 + 2 z_5
    const int n = (kc == 0 || kc == 3) ? 0 : (kc == 2 || kc == 5) ? 1 : 2;
    c.heavy = (kc & 1) == 0;
    c.own = c.heavy ? -2 : 2;
    const int a0 = 2 * n, a1 = 2 * n + 1, b0 = 2 * n + 6, b1 = 2 * n + 7;
#pragma unroll
    for (int t = 0; t < 3; t++) {
        c.p[t] = c.q[t] = c.r[t] = c.s[t] = a0;
        c.beta[t] = c.gamma[t] = c.delta[t] = 0;
    }
    auto term = [&](int t, int p, int beta, int q, int gamma, int r, int delta, int s) {
        c.p[t] = p; c.beta[t] = beta; c.q[t] = q;
        c.gamma[t] = gamma; c.r[t] = r; c.delta[t] = delta; c.s[t] = s;
    };
    if (c.heavy && e == 0) {             // 3 ((a0 + a1)(a0 - a1) + b0 (b0 - 2 b1) - b1^2)
        term(0, a0, 1, a1, 3, a0, -3, a1);
        term(1, b0, -2, b1, 3, b0, 0, b0);
        term(2, b1, 0, b1, -3, b1, 0, b1);
    } else if (c.heavy) {                // 3 (2 a0 a1 + (b0 - b1)(b0 + b1) + 2 b0 b1)
        term(0, a1, 0, a1, 6, a0, 0, a0);
        term(1, b0, -1, b1, 3, b0, 3, b1);
        term(2, b1, 0, b1, 6, b0, 0, b0);
    } else if (kc != 1) {                // 6 (a0 b0 - a1 b1), 6 (a0 b1 + a1 b0)
        term(0, e ? b1 : b0, 0, a0, 6, a0, 0, a0);
        term(1, e ? b0 : b1, 0, a0, e ? 6 : -6, a1, 0, a0);
    } else {                             // times xi: 6 (a0 (b0 - b1) - a1 (b0 + b1)), 6 (a0 (b0 + b1) + a1 (b0 - b1))
        term(0, b0, e ? 1 : -1, b1, 6, a0, 0, a0);
        term(1, b0, e ? -1 : 1, b1, e ? 6 : -6, a1, 0, a0);
    }
    return c;
}

FPG_DEV void l12_put(const L12Lane& c, int32_t* out, int32_t limb) { limb_put(out + LIMB_ROW * c.o, c.k.l, limb); }

template <int NT>
FPG_DEV int64_t l12_cyc_terms(L12& W, const L12Lane& c, const int32_t* z) {
    const int l = c.k.l;
    int32_t* priv = W.win + L12_PRIV * (int)(threadIdx.x >> 4);
    int32_t* rows = priv + 3 * LIMB_WIN;
    const int32_t *win[NT], *row[NT];
#pragma unroll
    for (int t = 0; t < NT; t++) {
        const int32_t x = z[LIMB_ROW * c.p[t] + l] + c.beta[t] * z[LIMB_ROW * c.q[t] + l];
        const int32_t y = c.gamma[t] * z[LIMB_ROW * c.r[t] + l] + c.delta[t] * z[LIMB_ROW * c.s[t] + l];
        limb_put_window(priv + LIMB_WIN * t, l, x);
        rows[LIMB_ROW * t + l] = y;
        win[t] = priv + LIMB_WIN * t;
        row[t] = rows + LIMB_ROW * t;
    }
    __syncwarp();
    int64_t lo, hi;
    limb_dot<NT>(c.k, lo, hi, row, win);
    return limb_reduce(c.k, lo, hi, W.u[threadIdx.x >> 4]) + (int64_t)c.own * limb_near_zero(c.k, z + LIMB_ROW * c.o);
}
// out = z^2 for z in the cyclotomic subgroup; out != z
FPG_DEV void l12_cyc_sqr(L12& W, const L12Lane& c, int32_t* out, const int32_t* z) {
    const int64_t col = c.heavy ? l12_cyc_terms<3>(W, c, z) : l12_cyc_terms<2>(W, c, z);   // warp-uniform
    l12_put(c, out, limb_carry(col, c.k.l));
    __syncthreads();
}

// out = a b, or a conj(b) (b's odd coefficients negated); out != a, b
FPG_DEV void l12_mul(L12& W, const L12Lane& c, int32_t* out, const int32_t* a, const int32_t* b, bool conj_b) {
    const int l = c.k.l, j = c.kc;
    const int32_t sg = conj_b && (j & 1) ? -1 : 1;
    const int32_t b0 = sg * b[LIMB_ROW * (2 * j) + l], b1 = sg * b[LIMB_ROW * (2 * j + 1) + l];
    int32_t* w0 = W.win + L12_WIN0 + (2 * j) * LIMB_WIN;
    int32_t* w1 = W.win + L12_WIN1 + (4 * j) * LIMB_WIN;
    if (c.e == 0) {
        limb_put_window(w0, l, b0);
        limb_put_window(w0 + LIMB_WIN, l, b0 - b1);
        limb_put_window(w1 + 3 * LIMB_WIN, l, -b0 - b1);
    } else {
        limb_put_window(w1, l, b1);
        limb_put_window(w1 + LIMB_WIN, l, -b1);
        limb_put_window(w1 + 2 * LIMB_WIN, l, b0 + b1);
    }
    __syncthreads();
    const int32_t *win[12], *row[12];
#pragma unroll
    for (int t = 0; t < 12; t++) {
        win[t] = W.win + c.wofs[t];
        row[t] = a + LIMB_ROW * t;
    }
    int64_t lo, hi;
    limb_dot<12>(c.k, lo, hi, row, win);
    l12_put(c, out, limb_carry(limb_reduce(c.k, lo, hi, W.u[threadIdx.x >> 4]), l));
    __syncthreads();
}

// out component = sum of NT products of rows y, y + 16, .. by constant values
template <int NT>
FPG_DEV int32_t l12_const_dot(L12& W, const L12Lane& c, const int32_t* y, const int32_t (&x)[NT]) {
    const int l = c.k.l;
    int32_t* priv = W.win + L12_PRIV * (int)(threadIdx.x >> 4);
    const int32_t *win[NT], *row[NT];
#pragma unroll
    for (int t = 0; t < NT; t++) {
        limb_put_window(priv + LIMB_WIN * t, l, x[t]);
        win[t] = priv + LIMB_WIN * t;
        row[t] = y + LIMB_ROW * t;
    }
    __syncwarp();
    int64_t lo, hi;
    limb_dot<NT>(c.k, lo, hi, row, win);
    return limb_carry(limb_reduce(c.k, lo, hi, W.u[threadIdx.x >> 4]), l);
}
// out = a^p: coefficient k is conj(a_k) g_k; out != a
FPG_DEV void l12_frob(L12& W, const L12Lane& c, int32_t* out, const int32_t* a) {
    const int32_t g0 = LIMB_FROB1[2 * c.kc][c.k.l], g1 = LIMB_FROB1[2 * c.kc + 1][c.k.l];
    const int32_t x[2] = {c.e ? g1 : g0, c.e ? -g0 : g1};
    l12_put(c, out, l12_const_dot<2>(W, c, a + LIMB_ROW * (2 * c.kc), x));
    __syncthreads();
}
// out = a^(p^2): coefficient k is a_k g_k, g_k in Fq; out != a
FPG_DEV void l12_frob2(L12& W, const L12Lane& c, int32_t* out, const int32_t* a) {
    const int32_t x[1] = {LIMB_FROB2[c.kc][c.k.l]};
    l12_put(c, out, l12_const_dot<1>(W, c, a + LIMB_ROW * c.o, x));
    __syncthreads();
}
// out = conj(a) = a^(p^6); out != a
FPG_DEV void l12_conj(const L12Lane& c, int32_t* out, const int32_t* a) {
    const int32_t v = a[LIMB_ROW * c.o + c.k.l];
    l12_put(c, out, c.kc & 1 ? -v : v);
    __syncthreads();
}

// component o of a value from a residue times 2^384, and back (the canonical words)
FPG_DEV void l12_load(L12& W, const L12Lane& c, int32_t* out, int32_t* tmp, const fq& a) {
    const int32_t x[1] = {LIMB_CONV[0][c.k.l]};
    l12_put(c, tmp, limb_of_words(a.v, c.k.l));
    __syncwarp();
    l12_put(c, out, l12_const_dot<1>(W, c, tmp + LIMB_ROW * c.o, x));
    __syncthreads();
}
// the component's words are returned on the slot's first lane
FPG_DEV fq l12_store(L12& W, const L12Lane& c, const int32_t* a, int32_t* tmp) {
    const int32_t x[1] = {LIMB_CONV[1][c.k.l]};
    l12_put(c, tmp, l12_const_dot<1>(W, c, a + LIMB_ROW * c.o, x));
    __syncwarp();
    fq r;
    fq_zero(r);
    if (c.k.l == 0) r = limb_canon(tmp + LIMB_ROW * c.o);
    __syncthreads();
    return r;
}

// out = a^-1 for a in Fq2 (coefficient 0; the others are ignored), zero elsewhere: on the canonical
// words, on the quad of lanes 0 .. 3 of the block (fq2_inv_quad); out != a, tmp
FPG_NOINL void l12_inv_fq2(L12& W, int32_t* out, const int32_t* a, int32_t* tmp) {
    const L12Lane c = l12_lane();
    const fq x = l12_store(W, c, a, tmp);
    if (c.kc == 0 && c.k.l == 0) W.x[c.e] = x;
    __syncthreads();
    if (threadIdx.x < 4) {
        const fq2 v{W.x[0], W.x[1]};
        const fq2 r = fq2_inv_quad(v);
        if (threadIdx.x == 0) {
            W.x[0] = r.c0;
            W.x[1] = r.c1;
        }
    }
    __syncthreads();
    fq y;
    fq_zero(y);
    if (c.kc == 0) y = W.x[c.e];
    l12_load(W, c, out, tmp, y);
}

// f^((p^12 - 1)/r) for f in W.v[0], into W.v[L12_FE_RESULT]: the list of operations L12_FE (its derivation and
// the check that its exponent is (p^12 - 1)/r stand where it is generated).  One loop with every operation inlined
// once, so that the lane's constants stay in registers; they are formed anew after the inversion, whose
// call would put them on the stack.
FPG_DEV void l12_final_exp(L12& W) {
    for (int part = 0; part < 2; part++) {
        const L12Lane c = l12_lane();
        const int end = part ? L12_FE_LEN : L12_FE_SPLIT;
        for (int i = part ? L12_FE_SPLIT : 0; i < end; i++) {
            const int op = L12_FE[i][0];
            int32_t* d = W.v[L12_FE[i][1]];
            const int32_t* a = W.v[L12_FE[i][2]];
            const int32_t* b = W.v[L12_FE[i][3]];
            if (op == 0) l12_cyc_sqr(W, c, d, a);
            else if (op <= 2) l12_mul(W, c, d, a, b, op == 2);
            else if (op == 3) l12_conj(c, d, a);
            else if (op == 4) l12_frob(W, c, d, a);
            else l12_frob2(W, c, d, a);
        }
        if (!part) l12_inv_fq2(W, W.v[4], W.v[3], W.v[2]);
    }
}
