// SHA-256 (FIPS 180-4) for one thread, streaming, plus the hash-to-Fr used for every
// Fiat-Shamir challenge: HFr(tag, data) = SHA256(tag || 0x00 || data) || SHA256(tag || 0x01 || data)
// read as a 512-bit big-endian integer and reduced mod r.
#pragma once
#include "fp.cuh"

struct sha256_ctx {
    uint32_t h[8];
    alignas(16) uint8_t buf[64];
    uint32_t nbuf;
    uint64_t total;
};

FPG_DEV uint32_t sha_rotr(uint32_t x, int n) { return (x >> n) | (x << (32 - n)); }

FPG_NOINL void sha256_compress(uint32_t* h, const uint8_t* blk) {
    uint32_t w[16];
    if (((uintptr_t)blk & 3) == 0) {                  // word loads, byte-swapped to big-endian
        const uint32_t* b4 = reinterpret_cast<const uint32_t*>(blk);
#pragma unroll
        for (int t = 0; t < 16; t++) w[t] = __byte_perm(b4[t], 0, 0x0123);
    } else {
#pragma unroll
        for (int t = 0; t < 16; t++)
            w[t] = ((uint32_t)blk[4 * t] << 24) | ((uint32_t)blk[4 * t + 1] << 16) | ((uint32_t)blk[4 * t + 2] << 8) |
                   blk[4 * t + 3];
    }
    uint32_t a = h[0], b = h[1], c = h[2], d = h[3], e = h[4], f = h[5], g = h[6], hh = h[7];
#pragma unroll
    for (int t = 0; t < 64; t++) {
        uint32_t wt;
        if (t < 16) {
            wt = w[t];
        } else {
            uint32_t w15 = w[(t - 15) & 15], w2 = w[(t - 2) & 15];
            uint32_t s0 = sha_rotr(w15, 7) ^ sha_rotr(w15, 18) ^ (w15 >> 3);
            uint32_t s1 = sha_rotr(w2, 17) ^ sha_rotr(w2, 19) ^ (w2 >> 10);
            wt = w[t & 15] = w[t & 15] + s0 + w[(t - 7) & 15] + s1;
        }
        uint32_t S1 = sha_rotr(e, 6) ^ sha_rotr(e, 11) ^ sha_rotr(e, 25);
        uint32_t ch = (e & f) ^ (~e & g);
        uint32_t t1 = hh + S1 + ch + SHA256_K[t] + wt;
        uint32_t S0 = sha_rotr(a, 2) ^ sha_rotr(a, 13) ^ sha_rotr(a, 22);
        uint32_t mj = (a & b) ^ (a & c) ^ (b & c);
        uint32_t t2 = S0 + mj;
        hh = g; g = f; f = e; e = d + t1; d = c; c = b; b = a; a = t1 + t2;
    }
    h[0] += a; h[1] += b; h[2] += c; h[3] += d; h[4] += e; h[5] += f; h[6] += g; h[7] += hh;
}

FPG_DEV void sha256_init(sha256_ctx& c) {
#pragma unroll
    for (int i = 0; i < 8; i++) c.h[i] = SHA256_H0[i];
    c.nbuf = 0;
    c.total = 0;
}
// whole 64-byte blocks of the input are compressed in place; only partial blocks are buffered.
// When the buffered length and the input address are multiples of 4 (long inputs after a header
// of whole words: statements, tree nodes), the input moves into the buffer a word at a time.
FPG_DEV void sha256_update(sha256_ctx& c, const uint8_t* data, uint32_t n) {
    c.total += n;
    if (((c.nbuf | (uint32_t)(uintptr_t)data) & 3) == 0) {
        const uint32_t* d32 = reinterpret_cast<const uint32_t*>(data);
        uint32_t* b32 = reinterpret_cast<uint32_t*>(c.buf);
        while (n >= 4) {
            if (c.nbuf == 0 && n >= 64) {
                sha256_compress(c.h, reinterpret_cast<const uint8_t*>(d32));
                d32 += 16;
                n -= 64;
                continue;
            }
            const uint32_t o = c.nbuf >> 2, take = min(16u - o, n >> 2);
            for (uint32_t i = 0; i < take; i++) b32[o + i] = d32[i];
            d32 += take;
            n -= 4 * take;
            c.nbuf += 4 * take;
            if (c.nbuf == 64) {
                sha256_compress(c.h, c.buf);
                c.nbuf = 0;
            }
        }
        data = reinterpret_cast<const uint8_t*>(d32);
    }
    while (n) {
        if (c.nbuf == 0 && n >= 64) {
            sha256_compress(c.h, data);
            data += 64;
            n -= 64;
            continue;
        }
        const uint32_t take = min(64u - c.nbuf, n);
        for (uint32_t i = 0; i < take; i++) c.buf[c.nbuf + i] = data[i];
        c.nbuf += take;
        data += take;
        n -= take;
        if (c.nbuf == 64) {
            sha256_compress(c.h, c.buf);
            c.nbuf = 0;
        }
    }
}
FPG_DEV void sha256_byte(sha256_ctx& c, uint8_t b) { sha256_update(c, &b, 1); }
FPG_DEV void sha256_final(sha256_ctx& c, uint8_t* out) {
    uint64_t bits = c.total * 8;
    c.buf[c.nbuf++] = 0x80;
    if (c.nbuf > 56) {
        while (c.nbuf < 64) c.buf[c.nbuf++] = 0;
        sha256_compress(c.h, c.buf);
        c.nbuf = 0;
    }
    while (c.nbuf < 56) c.buf[c.nbuf++] = 0;
    for (int i = 0; i < 8; i++) c.buf[56 + i] = (uint8_t)(bits >> (56 - 8 * i));
    sha256_compress(c.h, c.buf);
    for (int i = 0; i < 8; i++) {
        out[4 * i] = (uint8_t)(c.h[i] >> 24); out[4 * i + 1] = (uint8_t)(c.h[i] >> 16);
        out[4 * i + 2] = (uint8_t)(c.h[i] >> 8); out[4 * i + 3] = (uint8_t)c.h[i];
    }
}
FPG_DEV void sha256(uint8_t* out, const uint8_t* data, uint32_t n) {
    sha256_ctx c; sha256_init(c); sha256_update(c, data, n); sha256_final(c, out);
}

// HFr over the concatenation of up to three byte ranges (pieces may be empty) followed by
// `nsuffix` bytes 0x01 (the re-hash rule for a challenge that must be invertible)
FPG_NOINL fr hash_to_fr(const char* tag, uint32_t taglen, const uint8_t* d0, uint32_t n0,
                        const uint8_t* d1, uint32_t n1, const uint8_t* d2, uint32_t n2,
                        uint32_t nsuffix = 0) {
    uint8_t wide[64];
    for (int half = 0; half < 2; half++) {
        sha256_ctx c;
        sha256_init(c);
        sha256_update(c, (const uint8_t*)tag, taglen);
        sha256_byte(c, (uint8_t)half);
        if (n0) sha256_update(c, d0, n0);
        if (n1) sha256_update(c, d1, n1);
        if (n2) sha256_update(c, d2, n2);
        for (uint32_t k = 0; k < nsuffix; k++) sha256_byte(c, 0x01);
        sha256_final(c, wide + 32 * half);
    }
    return fr_from_be64(wide);
}

#ifndef FPG_PRIMITIVES_EXTERNAL
// The two SHA-256 halves of HFr(tag, prev || data) on one warp, into the 64 bytes at `wide` (shared): tag of 4
// bytes, prev of 32 or null, data of n bytes, n and its address multiples of 4, 5 + 32 + n + 9 <= 31 x 64.
// The hash itself is a serial chain of compressions, but the message is known: the warp lays it out in
// `msg` (shared, whole blocks), every lane expands the schedule of one block (column `lane` of wk[64][32],
// round constants added; lane 31 the second half's first block, the only one that differs), and two lanes
// then run the rounds alone.  22 blocks: 20 us instead of 45 when each of the two lanes also gathered its
// message byte by byte and expanded it.
FPG_DEV void hfr_wide_warp(uint8_t* msg, uint32_t* wk, uint8_t* wide, const char* tag, const uint8_t* prev,
                           const uint8_t* data, uint32_t n) {
    const uint32_t L = threadIdx.x & 31, o = prev ? 37 : 5, total = o + n, nb = (total + 9 + 63) / 64;
    if (L < 5) msg[L] = L < 4 ? (uint8_t)tag[L] : 0;
    if (prev) msg[5 + L] = prev[L];
    const uint32_t* d32 = reinterpret_cast<const uint32_t*>(data);
    for (uint32_t i = L; i < n / 4; i += 32) {
        const uint32_t w = d32[i];
#pragma unroll
        for (int k = 0; k < 4; k++) msg[o + 4 * i + k] = (uint8_t)(w >> (8 * k));
    }
    const uint64_t bits = (uint64_t)total * 8;
    for (uint32_t i = total + L; i < nb * 64; i += 32) {
        const uint32_t back = nb * 64 - 1 - i;             // bytes after this one
        msg[i] = i == total ? 0x80 : back < 8 ? (uint8_t)(bits >> (8 * back)) : 0;
    }
    __syncwarp();
    if (L < nb || L == 31) {
        const uint32_t* m32 = reinterpret_cast<const uint32_t*>(msg + (L == 31 ? 0 : 64 * L));
        uint32_t w[16];
#pragma unroll
        for (int t = 0; t < 16; t++) w[t] = __byte_perm(m32[t], 0, 0x0123);
        if (L == 31) w[1] |= 0x01000000u;
#pragma unroll
        for (int t = 0; t < 64; t++) {
            if (t >= 16) {
                const uint32_t w15 = w[(t - 15) & 15], w2 = w[(t - 2) & 15];
                w[t & 15] += (sha_rotr(w15, 7) ^ sha_rotr(w15, 18) ^ (w15 >> 3)) + w[(t - 7) & 15] +
                             (sha_rotr(w2, 17) ^ sha_rotr(w2, 19) ^ (w2 >> 10));
            }
            wk[32 * t + L] = w[t & 15] + SHA256_K[t];
        }
    }
    __syncwarp();
    if (L < 2) {
        uint32_t h[8];
#pragma unroll
        for (int i = 0; i < 8; i++) h[i] = SHA256_H0[i];
        for (uint32_t q = 0; q < nb; q++) {
            const uint32_t* c = wk + (L == 1 && q == 0 ? 31 : q);
            uint32_t a = h[0], b = h[1], cc = h[2], d = h[3], e = h[4], f = h[5], g = h[6], hh = h[7];
#pragma unroll 16
            for (int t = 0; t < 64; t++) {
                const uint32_t t1 = hh + (sha_rotr(e, 6) ^ sha_rotr(e, 11) ^ sha_rotr(e, 25)) + ((e & f) ^ (~e & g)) +
                                    c[32 * t];
                const uint32_t t2 = (sha_rotr(a, 2) ^ sha_rotr(a, 13) ^ sha_rotr(a, 22)) + ((a & b) ^ (a & cc) ^ (b & cc));
                hh = g; g = f; f = e; e = d + t1; d = cc; cc = b; b = a; a = t1 + t2;
            }
            h[0] += a; h[1] += b; h[2] += cc; h[3] += d; h[4] += e; h[5] += f; h[6] += g; h[7] += hh;
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
#pragma unroll
            for (int k = 0; k < 4; k++) wide[32 * L + 4 * i + k] = (uint8_t)(h[i] >> (24 - 8 * k));
        }
    }
    __syncwarp();
}
#endif

// HFr that never returns 0: re-hash with one more 0x01 byte appended while the value is 0
FPG_NOINL fr hash_to_fr_nonzero(const char* tag, uint32_t taglen, const uint8_t* d0, uint32_t n0,
                                const uint8_t* d1, uint32_t n1, const uint8_t* d2, uint32_t n2) {
    fr v = hash_to_fr(tag, taglen, d0, n0, d1, n1, d2, n2, 0);
    for (uint32_t k = 1; fr_is_zero(v) && k < 64; k++) v = hash_to_fr(tag, taglen, d0, n0, d1, n1, d2, n2, k);
    return v;
}
