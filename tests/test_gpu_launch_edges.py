"""Launch rules that depend on the number of pairs, fold points or buckets, at the sizes where they change:
the bytes equal those of the thread-per-item kernels (held to the oracle by the engine tests) or, for
the MSM, the oracle's."""
import pytest

pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2601_03031_gb300 import _lib as F  # noqa: E402
from paper_2601_03031_gb300 import inputs as I  # noqa: E402

BIG = 0xFFFFFFFF


@pytest.mark.parametrize("log_r,b,plain", [
    # 2^17 then 2^16 Miller loops: four, then two per thread; against one per thread
    (9, 2, {"miller_group_min": BIG}),
    # 19 blocks: 152 fold points in the fifth round (the largest with tables of the shifts), 304 before it
    (8, 14, {"fold_warp_max": 0}),
    # 16 blocks of 16 rows: 128 fold points in the first round, 256 Miller outputs reduced by eights
    (4, 1, {"fold_warp_max": 0, "miller_block_max": 0, "miller_warp_max": 0, "pair_block_max": 0}),
])
def test_openall_equal_across_launch_rules(log_r, b, plain):
    pp = F.PP(log_r + 1, b, 5, log_r=log_r)
    m = I.vector(17, log_r + 1)
    out = []
    try:
        for lim in ({}, plain):
            F.set_engine_limits(None)
            if lim:
                F.set_engine_limits(lim)
            cm = F.Commitment(pp, m)
            pf = F.vc_open_segments(pp, cm, b)
            out.append((cm.get(), [pf.segment_proof(j) for j in range(0, pp.R, b)]))
    finally:
        F.set_engine_limits(None)
    assert out[0] == out[1]


@pytest.mark.parametrize("window", [11, 12])       # 12 x 1024 buckets: one limb per lane; 11 x 2048: threads
def test_msm_bucket_count_edge(window):
    n = 40
    pts = b"".join(O.g1_mul(O.g1_gen(), 3 * v + 1) for v in range(n))
    k = I.vector(23, 6)[:n]
    assert F.msm_g1(F.G1Bases(points=pts), k, 1, window) == O.g1_msm(pts, I.to_ints(k))


@pytest.mark.parametrize("log_r,b,some", [
    (11, 37, 8),        # 56 blocks, the last of 13 rows: 2072 terms in the early rounds on 8 lanes each
    (11, 3, 128),       # 683 blocks: more than 1024 terms also where three rows meet two or four values
    (11, 2048, 1),      # one block: 2048 terms in the first round alone
])
def test_sparse_terms_equal_on_groups_and_blocks(log_r, b, some):
    """A call over all blocks (more than 1024 terms in a round) against calls over a few of them (at most 1024), or,
    for one block, the verifier; four rows commit to zeros."""
    pp = F.PP(log_r + 1, b, 5, log_r=log_r)
    m = I.vector(17, log_r + 1)
    m[6:12] = 0
    m[-2:] = 0
    cm = F.Commitment(pp, m)
    C, R, K = cm.get()[0], pp.R, -(-pp.R // b)
    pf = F.vc_open_segments(pp, cm, b)
    for k in ([0] if K == 1 else [0, K // 2, K - some]):
        if K > 1:
            few = F.vc_open_segments(pp, cm, b, k, some)
            for j in range(k * b, min((k + some) * b, R), b):
                assert pf.segment_proof(j) == few.segment_proof(j), j
        assert F.vc_verify_segment(pp, C, b, k * b, m[2 * k * b:2 * k * b + 2], pf.segment_proof(k * b))


def test_msm_batches_equal_on_groups_and_blocks():
    """1025 sums in one call (8 lanes each at the end) against the same sums in two calls (half a block each)."""
    n, nb = 3, 1025
    bases = F.G1Bases(points=b"".join(O.g1_mul(O.g1_gen(), 5 * v + 2) for v in range(n)))
    k = I.fr_uniform(29, n * nb)
    k[3 * 700:3 * 701] = 0                             # one sum is the identity
    whole = F.msm_g1(bases, k, nb)
    assert whole == F.msm_g1(bases, k[:3 * 600], 600) + F.msm_g1(bases, k[3 * 600:], 425)
    assert whole[:96] == O.g1_msm(b"".join(O.g1_mul(O.g1_gen(), 5 * v + 2) for v in range(n)), I.to_ints(k[:3]))


@pytest.mark.parametrize("log_c", [11, 12])        # 2047 terms: half a block each; 4095: 8 lanes each
def test_evaluation_proof_verifies_on_either_side_of_the_term_limit(log_c):
    """Its PST proofs are the only points that satisfy the oracle's check (pairing by pairing over every level)."""
    pp = F.PP(1 + log_c, 1, 9, log_r=1)
    m = I.vector(31, 1 + log_c)
    m[:1 << (log_c - 1)] = 0                       # and zero factors
    cm = F.Commitment(pp, m)
    C = cm.get()[0]
    for r in (I.to_ints(I.fr_uniform(37, 1 + log_c)), [1] + [0] * log_c):
        proof = F.vc_eval_prove(pp, cm, r)
        assert O.eval_verify(O.PP(1 + log_c, 9, log_r=1), C, r, proof)
        assert F.vc_eval_verify(pp, C, r, proof)
        bad = bytearray(proof)
        bad[-1] ^= 1
        assert not F.vc_eval_verify(pp, C, r, bytes(bad))


@pytest.mark.parametrize("log_r,log_c,b", [
    (9, 1, 3),         # 171 blocks of up to 22 terms, the last of two rows: block terms on 8 lanes each
    (12, 1, 64),       # 4096 rows
    (1, 12, 2),        # 4096 columns
    (1, 14, 2),        # 16384 columns: products of a thread each
    (5, 6, 32),        # everything on half a block each, but the 2048 single checks of `each`
])
def test_verify_all_equal_on_groups_and_blocks(log_r, log_c, b):
    """Acceptance of every proof, by shared and by single checks, against the claimed values that are wrong, and the
    single verifier (half a block per multiplication) at some positions."""
    pp = F.PP(log_r + log_c, b, 7, log_r=log_r)
    m = I.vector(41, log_r + log_c)
    m[: 1 << log_c] = 0                                # row 0 commits to the identity
    cm = F.Commitment(pp, m)
    C = cm.get()[0]
    pf = F.vc_prove_all(pp, cm, b)
    claim, wrong = m.copy(), [1, pp.N // 2 + 1, pp.N - 1]
    for i in wrong:
        claim[i, 0] ^= 1
    for each in (False, True):
        ok, n_ok = F.vc_verify_all(pf, C, claim, each=each)
        assert n_ok == pp.N - 3 and [i for i in range(pp.N) if not ok[i]] == wrong
    for i in [0] + wrong:
        v = I.to_ints(claim[i:i + 1])[0]
        assert F.vc_verify(pp, C, b, i, v, pf.proof(i)) == (i not in wrong)
    ok, n_ok = F.vc_verify_all(pf, F.Commitment(pp, claim).get()[0], m)
    assert n_ok == 0 and not any(ok)
