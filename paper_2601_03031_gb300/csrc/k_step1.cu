// Step 1 of OpenAll: FC.BOpen (Sec. 3, Eq. b and Eq. folding) for every block S_k at once, with
// b = sum_{a in S_k} r_a u_a held densely per block, and the faster-verification proof of v_l.
// Per-block arrays are laid out block-major: X[k * R + i].
#include <algorithm>

#include "group_ec.cuh"
#include "limb_ec.cuh"
#include "k_common.cuh"

namespace fpk {

__global__ void k_step1_init(const g1a* rows, const g2a* g2pow, uint32_t K, uint32_t R, g1a* A, g2a* v, fr* bvec) {
    uint64_t t = gtid();
    if (t >= (uint64_t)K * R) return;
    uint32_t i = (uint32_t)(t % R);
    A[t] = rows[i];
    v[t] = g2pow[2 * i];
    fr_zero(bvec[t]);
}

// SHA256(C || u32be(k) || u32be(b) || u32be(|S_k|) || C_a for a in S_k), for the K blocks
// k = k0 .. k0 + K - 1 (stored at local index k - k0)
// SHA256 of block k's statement C || u32be(k) || u32be(b) || u32be(|S_k|) || D_k, D_k the root of the
// tree over the block's row commitments C_a (leaves SHA256("FP-sleaf" || C_a), nodes
// SHA256("FP-snode" || left || right) pairing each level left to right, an odd last node carried up).
// One block per k: warps 0..7 hash the leaves and the levels (ping-pong between two halves of the
// scratch, nk digests each), warp 8 meanwhile absorbs C and the header into the final hash's state.
constexpr int STMT_TPB = 288;
__global__ void __launch_bounds__(STMT_TPB) k_stmt_hash(const uint8_t* C_ser, const uint8_t* rows_ser, uint32_t k0,
                                                        uint32_t R, uint32_t b, uint8_t* scratch, uint8_t* hstmt) {
    __shared__ sha256_ctx pre;
    __shared__ uint8_t* root;
    const uint32_t kl = blockIdx.x, k = k0 + kl, lo = k * b, hi = min(lo + b, R), nk = hi - lo;
    const uint32_t bb = min(b, R), tid = threadIdx.x, nt = STMT_TPB - 32;
    if (tid >= nt) {                      // warp 8: C and the header, beside the tree
        if (tid == nt) {
            sha256_init(pre);
            sha256_update(pre, C_ser, 576);
            uint8_t hdr[12];
            put_be32(hdr, k); put_be32(hdr + 4, b); put_be32(hdr + 8, nk);
            sha256_update(pre, hdr, 12);
        }
    } else {                              // warps 0..7: leaves, then the levels (barrier 1 of 256)
        uint8_t* src = scratch + (size_t)kl * 2 * bb * 32;
        uint8_t* dst = src + (size_t)bb * 32;
        for (uint32_t t = tid; t < nk; t += nt) {
            sha256_ctx c;
            sha256_init(c);
            sha256_update(c, (const uint8_t*)"FP-sleaf", 8);
            sha256_update(c, rows_ser + (size_t)(lo + t) * 96, 96);
            sha256_final(c, src + (size_t)t * 32);
        }
        for (uint32_t n = nk; n > 1; n = (n + 1) / 2) {
            asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
            for (uint32_t i = tid; i < (n + 1) / 2; i += nt) {
                if (2 * i + 1 < n) {
                    sha256_ctx c;
                    sha256_init(c);
                    sha256_update(c, (const uint8_t*)"FP-snode", 8);
                    sha256_update(c, src + (size_t)(2 * i) * 32, 64);
                    sha256_final(c, dst + (size_t)i * 32);
                } else {
                    for (int q = 0; q < 32; q++) dst[(size_t)i * 32 + q] = src[(size_t)(2 * i) * 32 + q];
                }
            }
            uint8_t* t = src;
            src = dst;
            dst = t;
        }
        if (tid == 0) root = src;
    }
    __syncthreads();
    if (tid == 0) {
        sha256_update(pre, root, 32);
        sha256_final(pre, hstmt + (size_t)kl * 32);
    }
}

// r_a = HFr("FP-r", SHA256(statement_k) || u32be(a)) placed at b[a] of block k (local index k - k0)
__global__ void k_block_r(const uint8_t* hstmt, uint32_t k0, uint32_t K, uint32_t R, uint32_t b, fr* bvec) {
    uint64_t t = gtid();
    if (t >= (uint64_t)K * b) return;
    const uint32_t kl = (uint32_t)(t / b), a = (k0 + kl) * b + (uint32_t)(t % b);
    if (a >= R) return;
    uint8_t buf[36];
    for (int q = 0; q < 32; q++) buf[q] = hstmt[(size_t)kl * 32 + q];
    put_be32(buf + 32, a);
    bvec[(size_t)kl * R + a] = hash_to_fr("FP-r", 4, buf, 36, nullptr, 0, nullptr, 0);
}

// Both folds of round j in one launch: blocks [0, nb_g2) fold v, the remaining blocks fold A and b.
__global__ void __launch_bounds__(64) k_fold(g1a* A, g2a* v, fr* bvec, const fr* x_mont, const fr* xinv_mont,
                                             uint32_t K, uint32_t R, uint32_t h, uint32_t nb_g2) {
    const bool g2 = blockIdx.x < nb_g2;
    uint64_t t = (uint64_t)(g2 ? blockIdx.x : blockIdx.x - nb_g2) * blockDim.x + threadIdx.x;
    if (t >= (uint64_t)K * h) return;
    uint64_t k = t / h;
    uint32_t i = (uint32_t)(t % h);
    uint64_t lo = k * R + i, hi = k * R + h + i;
    uint32_t kw[8];
    if (g2) {
        fr_canon_words(kw, xinv_mont[k]);
        v[lo] = g2_affine(g2_madd(g2_mul(v[hi], kw), v[lo]));
    } else {
        fr_canon_words(kw, x_mont[k]);
        A[lo] = g1_affine(g1_madd(g1_mul(A[hi], kw), A[lo]));
        bvec[lo] = fr_add(bvec[lo], fr_mul(bvec[hi], xinv_mont[k]));
    }
}

// the G1 parts of round j's record (the GT parts are written by the final exponentiation); a quad of
// four threads per point shares the inversion (jac_to_affine_quad), whole quads leave together
__global__ void __launch_bounds__(64) k_round_g1_out(const g1j* sp, uint32_t K, int j, uint8_t* blocks,
                                                     size_t bopen_len) {
    const uint64_t t = gtid() >> 2;
    if (t >= (uint64_t)K * 2) return;
    g1a a;
    jac_to_affine_quad(a.x, a.y, sp[t]);
    if ((threadIdx.x & 3) == 0) {
        uint8_t* rec = blocks + (t >> 1) * bopen_len + (size_t)(j - 1) * ROUND_BYTES + (t & 1) * (GT_SER + G1_SER);
        g1a_to_be(rec + GT_SER, a);
    }
}

// Both folds of round j with one limb per lane (limb_ec.cuh): blocks [0, n) fold a point of v each, the
// remaining blocks two points of A (96 threads each) and their entries of b, n = K h points t = (k, i).
// Latency-bound up to about one block per SM: 0.155 ms for 1 to 64 points and 0.19 for 128 from tables of the
// bases' shifts formed beside the round's pairings (k_fold_pre, 0.13 ms), 0.25 and 0.31 without them; 0.79 ms
// for 512 points, 2.8 for 2048, 5.5 for 4096 (one GB300).  A warp per G2 point and 8 lanes per G1 point took
// 1.21 ms for 512 points and 6.1 for 4096.  One thread per point (k_fold) takes 4.2 ms for any number up to 8192
// and 5.7 for 16384, so the two meet at about 3200 points: the default limit is right for 2048 points (2.8) and
// 8192 (10.7), and 1.2 ms dear at 4096 (5.4), which a fold_warp_max of 3000 saves.  Full comb tables of the bases (0.16 ms for 64 points after the challenge)
// took 0.96 ms of chains and tables per round beside the pairings.
union FoldSmemW {
    LimbEc2 g2;
    LimbEc g1[2];
};
// PRE: from the tables of the points' shifts (fold_pre_bytes, by k_fold_pre)
template <bool PRE>
__global__ void __launch_bounds__(LEC2_THREADS) k_fold_w(g1a* A, g2a* v, fr* bvec, const fr* x_mont,
                                                         const fr* xinv_mont, uint32_t K, uint32_t R, uint32_t h,
                                                         const int32_t* pre) {
    __shared__ FoldSmemW sm;
    const uint64_t n = (uint64_t)K * h;
    uint32_t kw[8];
    if (blockIdx.x < n) {
        const uint64_t t = blockIdx.x, k = t / h;
        const uint64_t lo = k * R + (uint32_t)(t % h), hi = lo + h;
        fr_canon_words(kw, xinv_mont[k]);
        const Lec2Lane c = lec2_lane();
        if (PRE) lec2_g2_mul_pre(sm.g2, c, pre + n * LEC_PRE_INTS + t * LEC2_PRE_INTS, kw);
        else lec2_g2_mul(sm.g2, c, v[hi], kw);
        lec2_add_affine(sm.g2, c, v[lo]);
        const fq r = lec2_affine(sm.g2, c);
        if (c.k.l == 0 && c.slot < 4) reinterpret_cast<fq*>(&v[lo])[c.slot] = r;
        return;
    }
    const int half = (int)(threadIdx.x / LEC_THREADS);
    const uint64_t t = (blockIdx.x - n) * 2 + half;
    if (t >= n) return;                                       // three whole warps, with a barrier of their own
    const uint64_t k = t / h;
    const uint64_t lo = k * R + (uint32_t)(t % h), hi = lo + h;
    fr_canon_words(kw, x_mont[k]);
    const LecLane c = lec_lane();
    if (PRE) lec_g1_mul_pre(sm.g1[half], c, pre + t * LEC_PRE_INTS, kw);
    else lec_g1_mul(sm.g1[half], c, A[hi], kw);
    lec_add_affine(sm.g1[half], c, A[lo]);
    const fq r = lec_affine(sm.g1[half], c);
    if (c.k.l == 0 && c.slot < 2) reinterpret_cast<fq*>(&A[lo])[c.slot] = r;
    if (c.k.l == 0 && c.slot == 2) bvec[lo] = fr_add(bvec[lo], fr_mul(bvec[hi], xinv_mont[k]));
}
// The fold's bases A[h + i], v[h + i] are known a round before its challenge: their tables of shifts
// (lec_pre, lec2_pre) are formed beside the round's pairings, for rounds of few points
__global__ void __launch_bounds__(LEC2_THREADS) k_fold_pre(const g1a* A, const g2a* v, uint32_t K, uint32_t R,
                                                           uint32_t h, int32_t* pre) {
    __shared__ FoldSmemW sm;
    const uint64_t n = (uint64_t)K * h;
    if (blockIdx.x < n) {
        const uint64_t t = blockIdx.x;
        lec2_pre(sm.g2, lec2_lane(), v[t / h * R + h + (uint32_t)(t % h)], pre + n * LEC_PRE_INTS + t * LEC2_PRE_INTS);
        return;
    }
    const int half = (int)(threadIdx.x / LEC_THREADS);
    const uint64_t t = (blockIdx.x - n) * 2 + half;
    if (t >= n) return;
    lec_pre(sm.g1[half], lec_lane(), A[t / h * R + h + (uint32_t)(t % h)], pre + t * LEC_PRE_INTS);
}
size_t fold_pre_bytes(uint32_t n) { return (size_t)n * (LEC_PRE_INTS + LEC2_PRE_INTS) * sizeof(int32_t); }

// L_j.1 and R_j.1 terms at the support of b only, for the blocks
// k0 .. k0 + K - 1 (local index k - k0).  Block k's vector b is
// non-zero only at its statement indices S_k = [k b, k b + |S_k|) folded mod the current length 2h:
// term t < min(|S_k|, 2h) sits at p = (k b + t) mod 2h (all p < 2h when |S_k| > 2h); p < h is an
// L_j.1 term b[p] A[h + p], p >= h an R_j.1 term b[p] A[p - h].  Results go to the dense per-block
// layout out[k 2h + p] (Jacobian), whose other entries the caller has zeroed (Z = 0: identity).
// Few terms: a block each, one limb per lane (limb_ec.cuh), for the latency the challenge waits for.
__global__ void __launch_bounds__(LEC_THREADS) k_sparse_g(const g1a* A, const fr* bvec, uint32_t k0, uint32_t K,
                                                          uint32_t R, uint32_t h, uint32_t b, uint32_t cmax,
                                                          g1j* out) {
    __shared__ LimbEc S;
    const uint64_t k = blockIdx.x / cmax;
    const uint32_t t = (uint32_t)(blockIdx.x % cmax);
    const uint32_t sk = min(b, R - (k0 + (uint32_t)k) * b);
    if (t >= min(sk, 2 * h)) return;                          // block-uniform
    const uint32_t p = sk <= 2 * h ? (uint32_t)(((uint64_t)(k0 + k) * b + t) % (2 * h)) : t;
    uint32_t kw[8];
    fr_canon_words(kw, bvec[k * R + p]);
    const LecLane c = lec_lane();
    lec_g1_mul(S, c, A[k * R + (p < h ? h + p : p - h)], kw);
    const fq v = lec_jacobian(S, c);
    if (c.k.l == 0 && c.slot < 3) reinterpret_cast<fq*>(&out[k * 2 * h + p])[c.slot] = v;
}
// Many terms: 8 lanes each (group_ec.cuh), which issue less per term.  A launch beside the pairings of the same
// round (one GB300), blocks against groups: 512 terms 0.6 and 0.9 ms, 1024 0.55-0.65 and 1.0, 2048 1.1 and
// 0.9, 4096 2.0 and 1.1, 8192 3.8 and 2.1.  Whole openings of sub-arrays with the line at 1024 against blocks
// at every size: 8192 rows in one block 46.8 and 49.9 ms, in 16 blocks 174 and 184, 4096 in one 29.3 and 30.5,
// 2048 in one 20.8 and 21.1; with the line at 512 1024 rows in one block take 12.1 instead of 12.0.
constexpr uint64_t SPARSE_LIMB_MAX = 1024;
__global__ void __launch_bounds__(128) k_sparse_g8(const g1a* A, const fr* bvec, uint32_t k0, uint32_t K, uint32_t R,
                                                   uint32_t h, uint32_t b, uint32_t cmax, g1j* out) {
    __shared__ GEc<fq> sm[16];
    const int grp = threadIdx.x >> 3, lane = threadIdx.x & 7;
    const uint64_t u = (uint64_t)blockIdx.x * 16 + grp;
    uint64_t k = u / cmax;
    uint32_t t = (uint32_t)(u % cmax);
    bool valid = k < K;
    uint32_t sk = valid ? min(b, R - (k0 + (uint32_t)k) * b) : 1;
    valid = valid && t < min(sk, 2 * h);
    if (!valid) { k = 0; t = 0; sk = min(b, R - k0 * b); }    // idle groups repeat a term, store nothing
    const uint32_t p = sk <= 2 * h ? (uint32_t)(((uint64_t)(k0 + k) * b + t) % (2 * h)) : t;
    uint32_t kw[8];
    fr_canon_words(kw, bvec[k * R + p]);
    const GPt<fq> r = gec_g1_mul_proj_w2(sm[grp], lane, A[k * R + (p < h ? h + p : p - h)], kw);
    if (valid && lane == 0) out[k * 2 * h + p] = proj_to_jac(r);
}

// x_j = HFr("FP-x", x_{j-1} || L_j || R_j) and its inverse, one warp per block: the hash on the warp
// (hfr_wide_warp), the inverse on a quad (a zero challenge falls back to the serial re-hash): 0.052 ms (0.077
// with the hash's halves on two lanes)
constexpr uint32_t CHAL_MSG = (5 + 32 + ROUND_BYTES + 9 + 63) / 64 * 64;
__global__ void __launch_bounds__(64) k_challenge2(const uint8_t* blocks, size_t bopen_len, uint32_t K, int j,
                                                   uint8_t* xprev, fr* x_mont, fr* xinv_mont, fr* xinv_all,
                                                   int log_r) {
    __shared__ __align__(16) uint8_t msg[2][CHAL_MSG];
    __shared__ uint32_t wk[2][64 * 32];
    __shared__ uint8_t wide[2][64];
    const int w = threadIdx.x >> 5, L = threadIdx.x & 31;
    const uint64_t k = (uint64_t)blockIdx.x * 2 + w;
    if (k >= K) return;                                       // warp-uniform
    const uint8_t* rec = blocks + k * bopen_len + (size_t)(j - 1) * ROUND_BYTES;
    uint8_t* xp = xprev + k * 32;
    hfr_wide_warp(msg[w], wk[w], wide[w], "FP-x", j > 1 ? xp : nullptr, rec, ROUND_BYTES);
    if (L < 4) {                                              // the inverse on the quad of lanes 0 .. 3
        fr x = fr_from_be64(wide[w]);
        if (fr_is_zero(x)) x = hash_to_fr_nonzero("FP-x", 4, xp, j > 1 ? 32 : 0, rec, ROUND_BYTES, nullptr, 0);
        const fr xi = fr_inv_quad(x);
        if (L == 0) {
            x_mont[k] = x;
            xinv_mont[k] = xi;
            xinv_all[k * log_r + (j - 1)] = xi;
            fr_to_be(xp, x);
        }
    }
}

// W = sum_i q_i g2^{beta^i}: one term per (k, i < 2R), padding terms are zero
__global__ void __launch_bounds__(64) k_w_terms(const g2a* g2pow, const fr* q_canon, uint32_t K, uint32_t R, g2j* out) {
    uint64_t t = gtid();
    if (t >= (uint64_t)K * 2 * R) return;
    uint32_t i = (uint32_t)(t % (2 * R));
    fr sc = q_canon[t];
    g2j res;
    if (i >= 2 * R - 1 || fr_is_zero(sc)) jac_set_inf(res);
    else res = g2_mul(g2pow[i], sc.v);
    out[t] = res;
}

// W terms with one warp per term (few terms: latency); results as Jacobian (X Z, Y Z^2, Z)
__global__ void __launch_bounds__(128) k_w_terms_w(const g2a* g2pow, const fr* q_canon, uint32_t K, uint32_t R,
                                                   g2j* out) {
    __shared__ GEcW sm[4];
    const int w = threadIdx.x >> 5, L = threadIdx.x & 31;
    const uint64_t t = (uint64_t)blockIdx.x * 4 + w;
    if (t >= (uint64_t)K * 2 * R) return;                     // warp-uniform
    const uint32_t i = (uint32_t)(t % (2 * R));
    const fr sc = q_canon[t];
    if (i >= 2 * R - 1 || fr_is_zero(sc)) {
        if (L == 0) {
            g2j z;
            jac_set_inf(z);
            out[t] = z;
        }
        return;
    }
    const GPt<fq2> r = gecw_g2_mul_proj(sm[w], L, g2pow[i], sc.v);
    __syncwarp();
    if (L == 0) {
        g2j o;
        o.X = fq2_mul(r.X, r.Z);
        o.Y = fq2_mul(r.Y, fq2_sqr(r.Z));
        o.Z = r.Z;
        out[t] = o;
    }
}

// The fast-verification proof of v_l, one block per CTA: A_l and v_l go into the block's record,
// z = HFr("FP-z", x_l || v_l), and the quotient coefficients, stored canonical and zero-padded to 2R:
//   P(X) = prod_j (1 + x_j^-1 X^(2^(l - j + 1))): the coefficient of X^m (m even) is the product of
//   x_j^-1 over the bits l - j + 1 set in m, and 0 for odd m;
//   q = (P(X) - P(z)) / (X - z): q_(i-1) = sum_{m >= i} P_m z^(m - i), by chunks of C indices: each
//   thread runs its chunk's recurrence with a zero carry, one thread chains the chunk carries
//   (carry of the chunk below = local top + z^len carry), then each chunk adds z^(hi - i) carry.
constexpr int KZG_THREADS = 128, KZG_CHUNK_MAX = 128;   // chunk length C <= KZG_CHUNK_MAX, one chunk per thread
__global__ void __launch_bounds__(KZG_THREADS) k_kzg_p(const g1a* A, const g2a* v, const uint8_t* xprev,
                                                       const fr* xinv_all, uint32_t K, uint32_t R, int log_r,
                                                       uint8_t* blocks, size_t bopen_len, fr* pcoef, fr* q_canon,
                                                       uint32_t C) {
    __shared__ fr zpow[KZG_CHUNK_MAX + 1];
    __shared__ fr carry[KZG_THREADS];
    const uint32_t k = blockIdx.x;
    const int T = threadIdx.x;
    const uint32_t deg = 2 * R - 2;
    fr* P = pcoef + (size_t)k * (deg + 1);
    fr* q = q_canon + (size_t)k * (2 * R);
    if (T == 0) {
        uint8_t* tail = blocks + k * bopen_len + (size_t)log_r * ROUND_BYTES;
        g1a_to_be(tail, A[(size_t)k * R]);
        g2a_to_be(tail + G1_SER, v[(size_t)k * R]);
        const fr z = hash_to_fr("FP-z", 4, xprev + k * 32, 32, tail + G1_SER, G2_SER, nullptr, 0);
        fr_one(zpow[0]);
        for (uint32_t c = 1; c <= C; c++) zpow[c] = fr_mul(zpow[c - 1], z);
    }
    for (uint32_t m = T; m <= deg; m += KZG_THREADS) {
        fr c;
        fr_one(c);
        if (m & 1) {
            fr_zero(c);
        } else {
            for (int j = 1; j <= log_r; j++)
                if ((m >> (log_r - j + 1)) & 1) c = fr_mul(c, xinv_all[(size_t)k * log_r + (j - 1)]);
        }
        P[m] = c;
    }
    __syncthreads();
    // indices i = 1 .. deg produce q_(i-1); chunk c covers i in [1 + c C, min(1 + (c + 1) C, deg + 1))
    const uint32_t nchunks = (deg + C - 1) / C;
    for (uint32_t c = T; c < nchunks; c += KZG_THREADS) {
        const uint32_t lo = 1 + c * C, hi = min(lo + C, deg + 1);
        fr acc;
        fr_zero(acc);
        for (uint32_t i = hi - 1; i >= lo; i--) {
            acc = fr_add(P[i], fr_mul(zpow[1], acc));        // local q_(i-1) with zero carry from above
            q[i - 1] = acc;
        }
        carry[c] = acc;                                       // local q_(lo-1)
    }
    __syncthreads();
    if (T == 0) {
        // true q_(lo_c - 1) = local_c + z^(hi_c - lo_c) q_(hi_c - 1), q_deg = 0 above the top chunk;
        // carry[c] <- the true q_(hi_c - 1) that chunk c needs
        fr above;
        fr_zero(above);
        for (int c = (int)nchunks - 1; c >= 0; c--) {
            const uint32_t lo = 1 + c * C, hi = min(lo + C, deg + 1);
            const fr local = carry[c];
            carry[c] = above;
            above = fr_add(local, fr_mul(zpow[hi - lo], above));
        }
    }
    __syncthreads();
    for (uint32_t c = T; c < nchunks; c += KZG_THREADS) {
        const uint32_t lo = 1 + c * C, hi = min(lo + C, deg + 1);
        const fr cin = carry[c];
        for (uint32_t i = lo; i < hi; i++) q[i - 1] = fr_from_mont(fr_add(q[i - 1], fr_mul(zpow[hi - i], cin)));
    }
    if (T == 0) {
        fr_zero(q[deg]);
        fr_zero(q[deg + 1]);
    }
}

void step1_init(const void* rows, const void* g2pow, uint32_t K, uint32_t R, void* A, void* v, void* bvec,
                cudaStream_t s) {
    FP_KERNEL("k_step1_init", s, k_step1_init<<<grid_for((uint64_t)K * R), TPB, 0, s>>>((const g1a*)rows, (const g2a*)g2pow, K, R, (g1a*)A,
                                                          (g2a*)v, (fr*)bvec));
}
size_t stmt_hash_scratch_bytes(uint32_t K, uint32_t R, uint32_t b) { return (size_t)K * 2 * std::min(b, R) * 32; }
void step1_stmt_hash(const void* C_ser, const void* rows_ser, uint32_t k0, uint32_t K, uint32_t R, uint32_t b,
                     void* scratch, void* hstmt, cudaStream_t s) {
    FP_KERNEL("k_stmt_hash", s, k_stmt_hash<<<K, STMT_TPB, 0, s>>>((const uint8_t*)C_ser, (const uint8_t*)rows_ser, k0,
                                                                   R, b, (uint8_t*)scratch, (uint8_t*)hstmt));
}
void step1_block_r(const void* hstmt, uint32_t k0, uint32_t K, uint32_t R, uint32_t b, void* bvec, cudaStream_t s) {
    FP_KERNEL("k_block_r", s, k_block_r<<<grid_for((uint64_t)K * b, 64), 64, 0, s>>>((const uint8_t*)hstmt, k0, K, R, b,
                                                                                    (fr*)bvec));
}
void step1_sparse_terms(const void* A, const void* bvec, uint32_t k0, uint32_t K, uint32_t R, uint32_t h, uint32_t b,
                        void* out, cudaStream_t s) {
    const uint32_t cmax = std::min(b, 2 * h);
    cudaMemsetAsync(out, 0, (size_t)K * 2 * h * G1J_BYTES, s);
    const uint64_t n = (uint64_t)K * cmax;
    if (n > SPARSE_LIMB_MAX)
        FP_KERNEL("k_sparse_g", s, k_sparse_g8<<<grid_for(n, 16), 128, 0, s>>>((const g1a*)A, (const fr*)bvec, k0, K, R, h,
                                                                              b, cmax, (g1j*)out));
    else
        FP_KERNEL("k_sparse_g", s, k_sparse_g<<<(unsigned)n, LEC_THREADS, 0, s>>>((const g1a*)A, (const fr*)bvec, k0, K, R,
                                                                                 h, b, cmax, (g1j*)out));
}
void step1_gt_out(const void* ml, uint32_t K, int j, void* blocks, size_t bopen_len, cudaStream_t s) {
    final_exp_group(ml, 2 * K, nullptr, (uint8_t*)blocks + (size_t)(j - 1) * ROUND_BYTES, 2, bopen_len,
                    GT_SER + G1_SER, s);
}
void step1_g1_out(const void* sp, uint32_t K, int j, void* blocks, size_t bopen_len, cudaStream_t s) {
    FP_KERNEL("k_round_g1_out", s, k_round_g1_out<<<grid_for((uint64_t)K * 8, 64), 64, 0, s>>>((const g1j*)sp, K, j,
                                                                                          (uint8_t*)blocks,
                                                                                          bopen_len));
}
void step1_challenge(void* blocks, size_t bopen_len, uint32_t K, int j, void* xprev, void* x_mont, void* xinv_mont,
                     void* xinv_all, int log_r, cudaStream_t s) {
    FP_KERNEL("k_challenge2", s, k_challenge2<<<(K + 1) / 2, 64, 0, s>>>((const uint8_t*)blocks, bopen_len, K, j,
                                                                         (uint8_t*)xprev, (fr*)x_mont, (fr*)xinv_mont,
                                                                         (fr*)xinv_all, log_r));
}
void step1_kzg(const void* A, const void* v, const void* xprev, const void* xinv_all, uint32_t K, uint32_t R,
               int log_r, void* blocks, size_t bopen_len, void* pcoef, void* q_canon, cudaStream_t s) {
    // chunks of C >= 32 coefficients, at most one per thread: C <= KZG_CHUNK_MAX for 2R - 2 <= 2^14
    const uint32_t deg = 2 * R - 2;
    uint32_t C = (deg + KZG_THREADS - 1) / KZG_THREADS;
    if (C < 32) C = 32;
    FP_KERNEL("k_kzg_p", s, k_kzg_p<<<K, KZG_THREADS, 0, s>>>((const g1a*)A, (const g2a*)v, (const uint8_t*)xprev,
                                                             (const fr*)xinv_all, K, R, log_r, (uint8_t*)blocks,
                                                             bopen_len, (fr*)pcoef, (fr*)q_canon, C));
}
// Comb tables of fixed G2 bases (the W proofs' g2^{beta^i}, built once at setup): per base its 64
// position tables (gpt_g2_comb_table) at tab[(i 64 + pos) 16], from the chain 2^pos B_i (a warp per
// base, then a thread per table).
__global__ void __launch_bounds__(128) k_g2_chain(const g2a* pts, uint32_t n, GPt<fq2>* chain) {
    __shared__ GEcWs sm[4];
    const int w = threadIdx.x >> 5, L = threadIdx.x & 31;
    const uint64_t t = (uint64_t)blockIdx.x * 4 + w;
    if (t >= n) return;                                       // warp-uniform
    GPt<fq2> acc = gec_from_affine_or_inf(pts[t].x, pts[t].y);
    for (int i = 0; i < 64; i++) {
        if (i) acc = gecw_dbl(sm[w], L, acc);
        if (L == 0) chain[t * 64 + i] = acc;
    }
}
__global__ void __launch_bounds__(64) k_g2_comb_tab(uint64_t m, const GPt<fq2>* chain, GPt<fq2>* tab) {
    const uint64_t u = gtid();
    if (u < m) gpt_g2_comb_table(chain[u], tab + u * 16);
}
size_t g2_comb_bytes(uint32_t n) { return (size_t)n * 64 * 16 * sizeof(GPt<fq2>); }
size_t g2_comb_chain_bytes(uint32_t n) { return (size_t)n * 64 * sizeof(GPt<fq2>); }
void g2_comb_tables(const void* pts_g2a, uint32_t n, void* chain_scratch, void* tab, cudaStream_t s) {
    if (!n) return;
    FP_KERNEL("k_g2_chain", s, k_g2_chain<<<(n + 3) / 4, 128, 0, s>>>((const g2a*)pts_g2a, n, (GPt<fq2>*)chain_scratch));
    FP_KERNEL("k_g2_comb_tab", s, k_g2_comb_tab<<<grid_for((uint64_t)n * 64, 64), 64, 0, s>>>(
                                      (uint64_t)n * 64, (const GPt<fq2>*)chain_scratch, (GPt<fq2>*)tab));
}

// W = sum_i q_i g2^{beta^i} from the comb tables, one limb per lane (limb_ec.cuh): a block per term (k, i < 2R)
// adds the entries of its 64 positions in a row, the next entry's limbs loaded while an addition runs; then
// blocks of up to 16 terms each, the last with the conversion to affine.  A point is kept as the limbs of
// its homogeneous coordinates (residues' limbs as they are: a common factor leaves the point the same).
// The term 2R - 1 and zero factors are the identity.
// 2R = 512 terms: 8-lane groups, their trees and the conversion took 0.25 + 0.21 + 0.055 ms in five launches.
struct WPart { int32_t c[6][LIMB_ROW]; };
FPG_DEV void w_put(LimbEc2& S, const Lec2Lane& c, int32_t v, bool first) {   // slot s < 6's coordinate part
    if (c.slot < 6) {
        if (first) lec2_put_acc(S, c.slot >> 1, c.e, c.k.l, v);
        else limb_put_window(lec2_win(S.two[c.slot >> 1], c.e), c.k.l, v);
    }
    __syncthreads();
}
__global__ void __launch_bounds__(LEC2_THREADS) k_w_comb(const GPt<fq2>* tab, const fr* q_canon, uint32_t R, WPart* out) {
    __shared__ LimbEc2 S;
    __shared__ unsigned char dg[64];
    const Lec2Lane c = lec2_lane();
    const int l = c.k.l, s = c.slot;
    const uint64_t t = blockIdx.x;
    const uint32_t i = (uint32_t)(t % (2 * R));
    if (threadIdx.x < 64) {
        uint32_t d[4][2];
        gls_digits(d, q_canon[t].v);
        dg[threadIdx.x] = i < 2 * R - 1 ? (unsigned char)gls_position(d, (int)threadIdx.x) : 0;
    }
    lec2_set_identity(S, c);                                  // (and the digits are visible)
    const GPt<fq2>* tb = tab + (size_t)(i < 2 * R - 1 ? i : 0) * 64 * 16;
    auto limb = [&](int pos) -> int32_t {
        return limb_of_words(reinterpret_cast<const fq*>(&tb[pos * 16 + dg[pos]])[s < 6 ? s : 0].v, l);
    };
    int pos = 0;
    while (pos < 64 && !dg[pos]) pos++;
    int32_t next = pos < 64 ? limb(pos) : 0;
    for (bool first = true; pos < 64; first = false) {
        w_put(S, c, next, first);
        do pos++;
        while (pos < 64 && !dg[pos]);
        if (pos < 64) next = limb(pos);
        if (!first) lec2_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
    }
    if (s < 6) out[t].c[s][l] = l < LIMB_N ? S.acc[s >> 1][c.e][l] : 0;
}
// out[b] = sum of in[gs b .. gs b + gs); with ser the affine sum's serialisation at ser + b stride instead
__global__ void __launch_bounds__(LEC2_THREADS) k_w_sum(const WPart* in, uint32_t gs, WPart* out, uint8_t* ser,
                                                        size_t stride) {
    __shared__ LimbEc2 S;
    const Lec2Lane c = lec2_lane();
    const int l = c.k.l, s = c.slot, co = s < 6 ? s : 0;
    const WPart* p = in + blockIdx.x * (uint64_t)gs;
    int32_t next = p[0].c[co][l];
    for (uint32_t u = 0; u < gs; u++) {
        w_put(S, c, next, u == 0);
        if (u + 1 < gs) next = p[u + 1].c[co][l];
        if (u) lec2_step<false>(S, c, S.two[0], S.two[1], S.two[2]);
    }
    if (ser) {
        const fq v = lec2_affine(S, c);
        if (l == 0 && s < 4) fq_to_be(ser + blockIdx.x * stride + 48 * s, v);
    } else if (s < 6) {
        out[blockIdx.x].c[s][l] = S.acc[s >> 1][c.e][l];
    }
}
size_t w_comb_bytes(uint32_t K, uint32_t R) { return (size_t)K * 2 * R * sizeof(WPart); }
void step1_w_comb(const void* tab, const void* q_canon, uint32_t K, uint32_t R, void* buf, void* buf2, void* ser,
                  size_t stride, cudaStream_t s) {
    uint64_t n = (uint64_t)K * 2 * R;
    WPart *a = (WPart*)buf, *b = (WPart*)buf2;
    FP_KERNEL("k_w_comb", s, k_w_comb<<<(unsigned)n, LEC2_THREADS, 0, s>>>((const GPt<fq2>*)tab, (const fr*)q_canon, R, a));
    while (n > K) {
        const uint32_t gs = (uint32_t)std::min<uint64_t>(16, n / K);
        n /= gs;
        FP_KERNEL("k_w_sum", s, k_w_sum<<<(unsigned)n, LEC2_THREADS, 0, s>>>(a, gs, b, n == K ? (uint8_t*)ser : nullptr, stride));
        std::swap(a, b);
    }
}

void step1_w_terms(const void* g2pow, const void* q_canon, uint32_t K, uint32_t R, void* out, cudaStream_t s) {
    const uint64_t n = (uint64_t)K * 2 * R;
    if (n <= engine_limits().wterm_warp_max) {      // few terms: a warp per term for latency
        FP_KERNEL("k_w_terms_w", s, k_w_terms_w<<<(unsigned)((n + 3) / 4), 128, 0, s>>>((const g2a*)g2pow,
                                                                                       (const fr*)q_canon, K, R,
                                                                                       (g2j*)out));
        return;
    }
    FP_KERNEL("k_w_terms", s, k_w_terms<<<grid_for(n, 64), 64, 0, s>>>((const g2a*)g2pow, (const fr*)q_canon, K, R,
                                                                      (g2j*)out));
}

}  // namespace fpk

namespace fpk {
uint64_t step1_miller_g(const void* A, const void* v, uint32_t K, uint32_t R, uint32_t h, void* ml_out,
                        cudaStream_t s) {
    uint64_t n = (uint64_t)K * 2 * h;
    const EngineLimits lim = engine_limits();
    if (n > lim.miller_warp_max && n > lim.miller_block_max) {   // many pairs: threads, less work in all
        const uint32_t group = step1_miller_group(n, h, lim);
        step1_miller(A, v, K, R, h, group, ml_out, s);
        return n / group;
    }
    round_miller(A, v, K, R, h, ml_out, s);        // few pairs: one block each, for latency
    return n;
}
void step1_fold_pre(const void* A, const void* v, uint32_t K, uint32_t R, uint32_t h, void* pre, cudaStream_t s) {
    const uint32_t n = K * h;
    FP_KERNEL("k_fold_pre", s, k_fold_pre<<<n + (n + 1) / 2, LEC2_THREADS, 0, s>>>((const g1a*)A, (const g2a*)v, K, R, h,
                                                                                  (int32_t*)pre));
}
void step1_fold(void* A, void* v, void* bvec, const void* x_mont, const void* xinv_mont, uint32_t K, uint32_t R,
                uint32_t h, const void* pre, cudaStream_t s) {
    const uint64_t n = (uint64_t)K * h;
    if (pre || n <= engine_limits().fold_warp_max) {   // few points: a block per G2 point, half a block per G1
        const unsigned nb = (unsigned)(n + (n + 1) / 2);
        if (pre)
            FP_KERNEL("k_fold_w", s, k_fold_w<true><<<nb, LEC2_THREADS, 0, s>>>((g1a*)A, (g2a*)v, (fr*)bvec,
                                         (const fr*)x_mont, (const fr*)xinv_mont, K, R, h, (const int32_t*)pre));
        else
            FP_KERNEL("k_fold_w", s, k_fold_w<false><<<nb, LEC2_THREADS, 0, s>>>((g1a*)A, (g2a*)v, (fr*)bvec,
                                         (const fr*)x_mont, (const fr*)xinv_mont, K, R, h, nullptr));
        return;
    }
    uint32_t nb = grid_for((uint64_t)K * h, 64);
    FP_KERNEL("k_fold", s, k_fold<<<2 * nb, 64, 0, s>>>((g1a*)A, (g2a*)v, (fr*)bvec, (const fr*)x_mont,
                                                        (const fr*)xinv_mont, K, R, h, nb));
}
}  // namespace fpk
