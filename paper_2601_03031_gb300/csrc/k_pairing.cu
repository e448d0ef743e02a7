// Batched Miller loops and final exponentiations.
#include "k_common.cuh"
#include "limb_miller.cuh"
#include "warp12.cuh"

namespace fpk {

// FC.Commit (Eq. genC): pair j is (C_j, v_j = g2^{beta^{2j}})
__global__ void __launch_bounds__(64) k_commit_miller(const g1a* rows, const g2a* g2pow, uint32_t R, fq12* out) {
    uint64_t j = gtid();
    if (j >= R) return;
    out[j] = miller_loop(rows[j], g2pow[2 * j]);
}

// Round j of FC.BOpen (Eq. folding) for every block at once, h = R / 2^j:
// pair t = (k, side, i): side 0 -> (A_R)[i] with (v_L)[i]  (L_j.T), side 1 -> (A_L)[i] with (v_R)[i]  (R_j.T)
__global__ void __launch_bounds__(64) k_step1_miller(const g1a* A, const g2a* v, uint32_t K, uint32_t R, uint32_t h,
                                                     fq12* out) {
    uint64_t t = gtid();
    if (t >= (uint64_t)K * 2 * h) return;
    uint64_t k = t / (2 * h);
    uint32_t r = (uint32_t)(t % (2 * h)), side = r / h, i = r % h;
    const g1a* Ak = A + k * R;
    const g2a* vk = v + k * R;
    out[t] = side == 0 ? miller_loop(Ak[h + i], vk[i]) : miller_loop(Ak[i], vk[h + i]);
}

// G consecutive pairs of the same (k, side) product in one multi-pair Miller loop; output t covers
// pairs (k, side, i) with i in [G t', G t' + G), t = (k 2 + side) (h / G) + t'
template <int G>
__global__ void __launch_bounds__(64) k_step1_miller_multi(const g1a* A, const g2a* v, uint32_t K, uint32_t R,
                                                           uint32_t h, fq12* out) {
    const uint64_t t = gtid();
    const uint32_t per = h / G;
    if (t >= (uint64_t)K * 2 * per) return;
    const uint64_t k = t / (2 * per);
    const uint32_t r = (uint32_t)(t % (2 * per)), side = r / per, i0 = (r % per) * G;
    const g1a* Ak = A + k * R;
    const g2a* vk = v + k * R;
    g1a P[G];
    g2a Q[G];
    for (int g = 0; g < G; g++) {
        P[g] = side == 0 ? Ak[h + i0 + g] : Ak[i0 + g];
        Q[g] = side == 0 ? vk[i0 + g] : vk[h + i0 + g];
    }
    out[t] = miller_loop_multi<G>(P, Q);
}

// one warp per final exponentiation (warp12.cuh): value t's result goes to out[t] and/or its
// serialisation to ser + (t / per) stride_a + (t % per) stride_b
__global__ void __launch_bounds__(128) k_final_exp_w(const fq12* in, uint32_t n, fq12* out, uint8_t* ser,
                                                     uint32_t per, size_t stride_a, size_t stride_b) {
    __shared__ W12 sm[4];
    const int w = threadIdx.x >> 5, L = threadIdx.x & 31;
    const uint64_t t = (uint64_t)blockIdx.x * 4 + w;
    if (t >= n) return;                                   // warp-uniform
    W12& W = sm[w];
    w_from_tower<1>(W.s[0], in[t]);
    w_final_exp<1>(W);
    if (L < 12) {
        const int tp = w_tower_pos(L >> 1), e = L & 1;
        const fq v = W.s[2][L];
        if (out) reinterpret_cast<fq*>(&out[t])[2 * tp + e] = v;
        if (ser) fq_to_be(ser + (t / per) * stride_a + (t % per) * stride_b + 96 * tp + 48 * e, v);
    }
}

// one block of twelve 16-lane slots per final exponentiation, one limb per lane (limb12.cuh): few of
// them, so the latency of one counts
__global__ void __launch_bounds__(L12_THREADS) k_final_exp_c(const fq12* in, uint32_t n, fq12* out, uint8_t* ser,
                                                             uint32_t per, size_t stride_a, size_t stride_b) {
    __shared__ L12 W;
    const uint64_t t = blockIdx.x;
    {
        const L12Lane c = l12_lane();
        l12_load(W, c, W.v[0], W.v[1], reinterpret_cast<const fq*>(&in[t])[2 * w_tower_pos(c.kc) + c.e]);
    }
    l12_final_exp(W);
    const L12Lane c = l12_lane();
    const int tp = w_tower_pos(c.kc);
    const fq v = l12_store(W, c, W.v[L12_FE_RESULT], W.v[0]);
    if (c.k.l == 0) {
        if (out) reinterpret_cast<fq*>(&out[t])[2 * tp + c.e] = v;
        if (ser) fq_to_be(ser + (t / per) * stride_a + (t % per) * stride_b + 96 * tp + 48 * c.e, v);
    }
}

// one thread per final exponentiation (many of them: the least work in total)
__global__ void k_final_exp_t(const fq12* in, uint32_t n, fq12* out, uint8_t* ser, uint32_t per, size_t stride_a,
                              size_t stride_b) {
    const uint64_t t = gtid();
    if (t >= n) return;
    const fq12 r = final_exp(in[t]);
    if (out) out[t] = r;
    if (ser) {
        const fq* c = reinterpret_cast<const fq*>(&r);
        for (int q = 0; q < 12; q++) fq_to_be(ser + (t / per) * stride_a + (t % per) * stride_b + 48 * q, c[q]);
    }
}

constexpr uint32_t FE_LIMB_MAX = 6 * 152;
void final_exp_group(const void* in, uint32_t n, void* out, void* ser, uint32_t per, size_t stride_a,
                     size_t stride_b, cudaStream_t s) {
    if (!n) return;
    const EngineLimits lim = engine_limits();
    if (n > lim.fe_warp_max && n > lim.fe_block_max) {
        FP_KERNEL("k_final_exp_t", s, k_final_exp_t<<<grid_for(n, 64), 64, 0, s>>>((const fq12*)in, n, (fq12*)out,
                                                                                  (uint8_t*)ser, per, stride_a,
                                                                                  stride_b));
        return;
    }
    // limb lanes also beyond the block limit (if there is one) up to six blocks per SM: 512 take 0.8 ms, 1024
    // 1.56 ms; a warp each takes 1.48 ms for 257 to 1024
    if (n <= lim.fe_block_max || (lim.fe_block_max && n <= FE_LIMB_MAX)) {
        FP_KERNEL("k_final_exp_c", s, k_final_exp_c<<<n, L12_THREADS, 0, s>>>((const fq12*)in, n, (fq12*)out,
                                                                             (uint8_t*)ser, per, stride_a, stride_b));
        return;
    }
    FP_KERNEL("k_final_exp_w", s, k_final_exp_w<<<(n + 3) / 4, 128, 0, s>>>((const fq12*)in, n, (fq12*)out,
                                                                           (uint8_t*)ser, per, stride_a, stride_b));
}

// out[q out_stride] = (base ? *base : 1) prod_{u < per} in[q stride + u], one block per q, one limb per lane:
// a factor costs its conversion and a product, 1.8 us, where a launch of pairwise products takes 8
__global__ void __launch_bounds__(L12_THREADS) k_fq12_prod(const fq12* base, const fq12* in, uint32_t stride,
                                                           uint32_t per, fq12* out, uint32_t out_stride) {
    __shared__ L12 W;
    const L12Lane c = l12_lane();
    const uint64_t q = blockIdx.x;
    const int pos = 2 * w_tower_pos(c.kc) + c.e;
    const fq12* src = in + q * stride;
    const uint32_t n = per + (base ? 1 : 0);
    int32_t *acc = W.v[0], *nxt = W.v[1];
    for (uint32_t u = 0; u < n; u++) {
        const fq12* f = base ? (u ? src + (u - 1) : base) : src + u;
        l12_load(W, c, u ? W.v[2] : acc, W.v[3], reinterpret_cast<const fq*>(f)[pos]);
        if (u) {
            l12_mul(W, c, nxt, acc, W.v[2], false);
            int32_t* t = acc;
            acc = nxt;
            nxt = t;
        }
    }
    const fq v = l12_store(W, c, acc, W.v[3]);
    if (c.k.l == 0) reinterpret_cast<fq*>(&out[q * out_stride])[pos] = v;
}
void fq12_products(const void* base, const void* in, uint32_t stride, uint32_t per, void* out, uint32_t out_stride,
                   uint64_t n, cudaStream_t s) {
    if (!n) return;
    FP_KERNEL("k_fq12_prod", s, k_fq12_prod<<<(unsigned)n, L12_THREADS, 0, s>>>((const fq12*)base, (const fq12*)in, stride,
                                                                               per, (fq12*)out, out_stride));
}

// pairwise Fq12 products out[i] = in[2i] in[2i+1]: one 128-thread block per product when there are
// few (latency), one thread per product otherwise
__global__ void k_fq12_pair(const fq12* in, fq12* out, uint64_t n) {
    uint64_t i = gtid();
    if (i < n) out[i] = fq12_mul(in[2 * i], in[2 * i + 1]);
}
__global__ void __launch_bounds__(128) k_fq12_pair_c(const fq12* in, fq12* out) {
    __shared__ W12 W;
    const int L = threadIdx.x;
    const uint64_t i = blockIdx.x;
    if (L < 12) {
        const int pos = 2 * w_tower_pos(L >> 1) + (L & 1);
        W.s[0][L] = reinterpret_cast<const fq*>(&in[2 * i])[pos];
        W.s[1][L] = reinterpret_cast<const fq*>(&in[2 * i + 1])[pos];
    }
    __syncthreads();
    w_mul<4>(W, W.s[2], W.s[0], W.s[1]);
    if (L < 12) reinterpret_cast<fq*>(&out[i])[2 * w_tower_pos(L >> 1) + (L & 1)] = W.s[2][L];
}
void fq12_pair_reduce(const void* in, void* out, uint64_t n, cudaStream_t s) {
    if (!n) return;
    if (n <= engine_limits().pair_block_max) {
        FP_KERNEL("k_fq12_pair_c", s, k_fq12_pair_c<<<(unsigned)n, 128, 0, s>>>((const fq12*)in, (fq12*)out));
        return;
    }
    FP_KERNEL("k_fq12_pair", s, k_fq12_pair<<<grid_for(n, 64), 64, 0, s>>>((const fq12*)in, (fq12*)out, n));
}

// Miller loops with few pairs, one block per pair, one limb per lane (limb_miller.cuh).  Pair t of Step 1
// round h: t = (k, side, i) with side 0: (A_k[h + i], v_k[i]) and side 1: (A_k[i], v_k[h + i]); Commit:
// (C_j, v_j = g2pow[2 j]).
// One launch (one GB300): 0.205 ms for up to 152 pairs (latency: 152 rounds of ~2.8 k cycles), 0.34 for
// 256, 1.25 for 1024, 4.5 for 4096, 8.8 for 8192.  With one Fq product per lane a 128-thread block per pair
// took 0.42 ms for few pairs and 1.4 for 1024, a warp per pair 11.1 ms for 8192; one thread per pair takes
// 19.8 ms for 16384 and 14.2 for 32768 (fewer run slower: their spills then miss).
FPG_DEV void miller_block(const g1a& P, const g2a& Q, fq12* out) {
    __shared__ LimbMiller S;
    const LmLane c = lm_lane();
    const fq v = lm_miller(S, c, P, Q);
    if (!c.point && c.k.l == 0) reinterpret_cast<fq*>(out)[2 * w_tower_pos(c.kc) + c.e] = v;
}
__global__ void __launch_bounds__(LM_THREADS, 2) k_round_miller_c(const g1a* A, const g2a* v, uint32_t K, uint32_t R,
                                                               uint32_t h, fq12* out) {
    const uint64_t t = blockIdx.x;
    const uint64_t k = t / (2 * h);
    const uint32_t r = (uint32_t)(t % (2 * h)), side = r / h, i = r % h;
    const g1a* Ak = A + k * R;
    const g2a* vk = v + k * R;
    miller_block(side == 0 ? Ak[h + i] : Ak[i], side == 0 ? vk[i] : vk[h + i], &out[t]);
}
__global__ void __launch_bounds__(LM_THREADS, 2) k_commit_miller_c(const g1a* rows, const g2a* g2pow, fq12* out) {
    const uint64_t j = blockIdx.x;
    miller_block(rows[j], g2pow[2 * j], &out[j]);
}
void round_miller(const void* A, const void* v, uint32_t K, uint32_t R, uint32_t h, void* out, cudaStream_t s) {
    const uint64_t n = (uint64_t)K * 2 * h;
    FP_KERNEL("k_round_miller_c", s, k_round_miller_c<<<(unsigned)n, LM_THREADS, 0, s>>>((const g1a*)A, (const g2a*)v, K,
                                                                                        R, h, (fq12*)out));
}

void commit_miller(const void* rows, const void* g2pow, uint32_t R, void* out, cudaStream_t s) {
    const EngineLimits lim = engine_limits();
    if (R > lim.commit_warp_max && R > lim.commit_block_max) {   // many pairs: one thread each, less work
        FP_KERNEL("k_commit_miller", s, k_commit_miller<<<grid_for(R, 64), 64, 0, s>>>((const g1a*)rows,
                                                                                       (const g2a*)g2pow, R,
                                                                                       (fq12*)out));
        return;
    }
    FP_KERNEL("k_commit_miller_c", s, k_commit_miller_c<<<R, LM_THREADS, 0, s>>>((const g1a*)rows, (const g2a*)g2pow,
                                                                                (fq12*)out));
}
// Pairs per thread of a launch of n pairs.  These kernels hold 255 registers a thread, so the GPU takes
// 152 x 256 threads at once and a launch costs whole waves: measured per wave 12.6 ms with one pair per
// thread, 21.4 with two sharing the squarings, 38.3 with four.  From miller_group_min on four (fewer
// products; 2^18 pairs 77 ms against 88).  Down to a quarter of it the fewest ms by waves: 2^17 pairs
// one wave of four, 38.3 ms against 42.5 (two waves of two) and 47.7 (four of one); 2^16 pairs one wave of
// two, 21.4 against 25.2 and 27.9; 87552 pairs 36 ms each way.  2^15 pairs and fewer fit one wave as
// they are (12.7 ms; pairs of them 15.4).  Eight per thread gained 6 ms at 2^18 pairs, lost 5 at 2^20 and
// doubled the local memory.
constexpr uint64_t MILLER_WAVE = 152 * 256;
uint32_t step1_miller_group(uint64_t n, uint32_t h, const EngineLimits& lim) {
    if (h >= 4 && n >= lim.miller_group_min) return 4;
    uint32_t best = 1;
    if (n < lim.miller_group_min / 4) return best;
    const uint32_t wave_ms10[3] = {126, 214, 383};
    uint64_t best_ms = ~0ull;
    for (uint32_t i = 0; i < 3 && (1u << i) <= h; i++) {
        const uint64_t ms = ((n >> i) + MILLER_WAVE - 1) / MILLER_WAVE * wave_ms10[i];
        if (ms < best_ms) { best_ms = ms; best = 1u << i; }
    }
    return best;
}
template <int G>
static void launch_miller_multi(const void* A, const void* v, uint32_t K, uint32_t R, uint32_t h, void* out,
                                cudaStream_t s) {
    const uint64_t n = (uint64_t)K * 2 * (h / G);
    FP_KERNEL("k_step1_miller_multi", s,
              k_step1_miller_multi<G><<<grid_for(n, 64), 64, 0, s>>>((const g1a*)A, (const g2a*)v, K, R, h,
                                                                    (fq12*)out));
}
void step1_miller(const void* A, const void* v, uint32_t K, uint32_t R, uint32_t h, uint32_t group, void* out,
                  cudaStream_t s) {
    if (group == 4) return launch_miller_multi<4>(A, v, K, R, h, out, s);   // pairs sharing the squarings
    if (group == 2) return launch_miller_multi<2>(A, v, K, R, h, out, s);
    uint64_t n = (uint64_t)K * 2 * h;
    FP_KERNEL("k_step1_miller", s, k_step1_miller<<<grid_for(n, 64), 64, 0, s>>>((const g1a*)A, (const g2a*)v, K, R, h, (fq12*)out));
}
}  // namespace fpk
