"""The work that users of this library have it do, as timed cases: proving all positions of a committed
vector (one vector or a batch), opening sub-arrays, the standalone G1 multi-scalar multiplication,
evaluation proofs, and verification.  Every output is bytes or a truth value of exact integer
arithmetic, so there is no rounding anywhere and outputs are compared for equality.

A case is a dict of plain values; "kind" names the call:
  open      vc_commit + vc_prove_all, the commitment and the whole shared proof state in host memory
            (log_n, b, dist: the value distribution)
  batch     commitments of many vectors of mixed sizes on one resident setup and one
            vc_prove_all_batch over them (jobs, log_min, log_max, mix: the seed of the sizes, graph)
  segments  vc_open_segments: Step 1 only, for R = 2^log_r segments of 2^log_c values in blocks of b
  msm       fp_msm_g1 on device-resident scalars (n terms, nbatch sums over the same n bases)
  eval      vc_eval_prove at a random point, and vc_eval_verify of the proof
  one       vc_prove_one of a random position, and vc_verify of the proof with the committed value and
            with another
  verify_all  vc_verify_all of every proof of a handle (wrong: how many claimed values at random
            positions are not the committed ones)
"""
import math

import numpy as np
import torch

from paper_2601_03031_gb300 import _lib as F
from paper_2601_03031_gb300 import inputs as I


def listed():
    return [
        # a short vector with no batching: the smallest all-proofs pass a user asks for (latency and
        # launches; every row is a block of its own)
        {"name": "open_n10_b1", "kind": "open", "log_n": 10, "b": 1, "dist": "uniform"},
        # an odd logarithm (64 rows of 128), small integers as values, a ragged last block (64 = 37 + 27)
        {"name": "open_n13_b37_u32", "kind": "open", "log_n": 13, "b": 37, "dist": "u32"},
        # the paper's headline setting, b = log^2 N: one block, latency-bound rounds
        {"name": "open_n16_b256", "kind": "open", "log_n": 16, "b": 256, "dist": "uniform"},
        # many blocks with short proofs: 512 blocks at once, throughput-bound pairings and folds
        {"name": "open_n18_b1", "kind": "open", "log_n": 18, "b": 1, "dist": "uniform"},
        # a long vector in one block: Step 2's trees and folds over a million values beside the rounds
        {"name": "open_n20_b1024", "kind": "open", "log_n": 20, "b": 1024, "dist": "uniform"},
        # the served mix: independent vectors of different sizes proved by one call
        {"name": "batch_16_jobs", "kind": "batch", "jobs": 16, "log_min": 8, "log_max": 16, "mix": 7, "graph": True},
        # sub-array openings of a sharded array: 1024 short segments, 8 blocks
        {"name": "segments_r10_b128", "kind": "segments", "log_r": 10, "log_c": 4, "b": 128},
        # a small commitment-sized multi-scalar multiplication, ragged
        {"name": "msm_3000", "kind": "msm", "n": 3000, "nbatch": 1},
        # a large one, not a power of two
        {"name": "msm_1m", "kind": "msm", "n": 1000003, "nbatch": 1},
        # a zkSNARK's use of the commitment: one evaluation proof and its verification
        {"name": "eval_n16", "kind": "eval", "log_n": 16},
        # a client asking for its own position's proof and checking it
        {"name": "one_n16_b16", "kind": "one", "log_n": 16, "b": 16},
        # an auditor checking every proof of a handle, a few claimed values being wrong
        {"name": "verify_all_n16_b16", "kind": "verify_all", "log_n": 16, "b": 16, "wrong": 5},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["open", "open", "open", "batch", "segments", "msm", "msm", "eval", "one", "verify_all"])
    if kind == "open":
        log_n = rng.randint(8, 20)
        R = 1 << (log_n // 2)
        b = _log_int(rng, 1 if log_n <= 17 else 4 << (2 * (log_n - 18)), R)
        return {"kind": kind, "log_n": log_n, "b": b, "dist": rng.choice(["uniform", "u32"])}
    if kind == "batch":
        return {"kind": kind, "jobs": _log_int(rng, 2, 24), "log_min": 8, "log_max": rng.randint(9, 16),
                "mix": rng.randrange(1 << 30), "graph": rng.random() < 0.5}
    if kind == "segments":
        log_r = rng.randint(4, 11)
        return {"kind": kind, "log_r": log_r, "log_c": rng.randint(1, 9),
                "b": _log_int(rng, max(1, (1 << log_r) // 32), 1 << log_r)}
    if kind == "msm":
        n = _log_int(rng, 100, 1 << 21)
        return {"kind": kind, "n": n, "nbatch": 1 if n > 100000 else _log_int(rng, 1, 32)}
    if kind == "eval":
        return {"kind": kind, "log_n": rng.randint(6, 20)}
    log_n = rng.randint(6, 17)
    b = _log_int(rng, 1, 1 << (log_n // 2))
    if kind == "one":
        return {"kind": kind, "log_n": log_n, "b": b}
    return {"kind": kind, "log_n": log_n, "b": b, "wrong": _log_int(rng, 1, 20)}


def _device(m):
    return torch.from_numpy(m.view(np.int64).copy()).cuda()


def _pinned(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8).pin_memory()


def _u8(b):
    return np.frombuffer(b, dtype=np.uint8)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "msm":
        n, nb = case["n"], case["nbatch"]
        return {"kind": kind, "bases": F.G1Bases(scalars=_device(I.fr_uniform(2 * seed + 1, n))), "nbatch": nb,
                "k": _device(I.fr_uniform(2 * seed, n * nb)),
                "out": torch.empty(96 * nb, dtype=torch.uint8, device="cuda")}
    if kind == "batch":
        jobs = I.batched_jobs(case["mix"], case["jobs"], case["log_min"], case["log_max"])
        pp = F.PP(case["log_max"], seed=seed)
        views = {k: pp.view(k) for k in sorted({j["log_n"] for j in jobs})}
        st = {"kind": kind, "graph": case["graph"], "jobs": [], "pp": pp}
        for q, j in enumerate(jobs):
            v = views[j["log_n"]]
            st["jobs"].append((v, _device(I.vector(seed * 1000 + q, j["log_n"])), j["b"],
                               _pinned(_state_bytes(v.R, v.M, j["b"]))))
        return st
    log_r = case.get("log_r")
    log_n = case["log_n"] if log_r is None else log_r + case["log_c"]
    b = case.get("b", 1)
    pp = F.PP(log_n, b, seed, log_r=log_r)
    m = I.vector(seed + 1, log_n, case.get("dist", "uniform"))
    st = {"kind": kind, "pp": pp, "b": b, "m": _device(m)}
    if kind == "open":
        st["host"] = _pinned(_state_bytes(pp.R, pp.M, b))
        return st
    st["cm"] = F.vc_commit(pp, st["m"])
    st["C"] = st["cm"].get(rows=False)[0]
    if kind == "eval":
        st["r"] = I.to_ints(I.fr_uniform(seed + 2, log_n))
    elif kind == "one":
        st["i"] = int(I.splitmix64(seed, 0, 1)[0]) % pp.N
        st["m_i"] = I.to_ints(m[st["i"]: st["i"] + 1])[0]
    elif kind == "verify_all":
        st["pf"] = F.vc_prove_all(pp, st["cm"], b)
        at = np.unique(I.splitmix64(seed, 0, case["wrong"]) % np.uint64(pp.N)).astype(np.int64)
        m[at] = I.u32_embedded(seed + 3, len(at))
        st["m"] = _device(m)
    return st


def run(state):
    kind = state["kind"]
    if kind == "msm":
        return F.msm_g1(state["bases"], state["k"], state["nbatch"], out=state["out"])
    if kind == "batch":
        cms = [F.Commitment(v, m, sync=False) for v, m, _, _ in state["jobs"]]
        pfs = F.vc_prove_all_batch([(cm, job[2]) for cm, job in zip(cms, state["jobs"])], use_graph=state["graph"])
        got = []
        for cm, pf, job in zip(cms, pfs, state["jobs"]):
            pf.state_into(job[3])
            got.append((_u8(cm.get(rows=False)[0]), job[3]))
        return got
    pp, b = state["pp"], state["b"]
    if kind == "open":
        cm = F.vc_commit(pp, state["m"])
        pf = F.vc_prove_all(pp, cm, b)
        C, rows = cm.get()
        pf.state_into(state["host"])
        return {"C": _u8(C), "rows": _u8(rows), "state": state["host"]}
    if kind == "segments":
        # the proof of a block's first segment holds the block's row commitments and its opening,
        # which every segment of the block shares
        pf = F.vc_open_segments(pp, state["cm"], b)
        return {"blocks": _u8(b"".join(pf.segment_proof(j) for j in range(0, pp.R, b)))}
    if kind == "eval":
        proof = F.vc_eval_prove(pp, state["cm"], state["r"])
        return {"proof": _u8(proof), "ok": F.vc_eval_verify(pp, state["C"], state["r"], proof)}
    if kind == "one":
        i, m_i = state["i"], state["m_i"]
        proof = F.vc_prove_one(pp, state["cm"], b, i)
        return {"proof": _u8(proof), "ok": F.vc_verify(pp, state["C"], b, i, m_i, proof),
                "other": F.vc_verify(pp, state["C"], b, i, m_i ^ 1, proof)}
    ok, n_ok = F.vc_verify_all(state["pf"], state["C"], state["m"])
    return {"ok": ok, "n_ok": n_ok}


def exact(case, seed):
    """No output is a rounded number: every one is bytes or a truth value."""
    return None


# One Fq product: 12 x 12 limb products of the factors and as many of the Montgomery reduction, each a
# 32 x 32 -> 64 bit multiply-add (two operations).
_FQ = 2 * 288
# Fq products of one unit by efficient textbook formulas
_MILLER, _FINAL_EXP, _G1_MUL, _G2_MUL = 7135, 10120, 2000, 3300
_MSM_TERM, _COMB_G1, _COMB_G2 = 2 * 13 * 10, 352, 2268      # 13 windows of two GLV halves; comb terms


def _state_bytes(R, M, b):
    K, lr = -(-R // b), R.bit_length() - 1
    return (K * (1344 * lr + 480) + R * (2 * M - 1) * 32 + (2 * R - 1) * 32 + R * 32 + (2 * R - 1) * 96
            + (2 * R - 1) * M * 32 + (M - 1) * 96)


def _commit_muls(R, M):
    return R * M * _COMB_G1 + R * _MILLER + _FINAL_EXP


def _step1_muls(R, b):
    K, lr = -(-R // b), R.bit_length() - 1
    sparse = sum(min(b, 2 * (R >> j)) for j in range(1, lr + 1))
    return K * ((R - 1) * (2 * _MILLER + _G1_MUL + _G2_MUL) + 2 * lr * _FINAL_EXP + sparse * _G1_MUL
                + (2 * R - 2) * _COMB_G2)


def _step2_muls(R, M):
    lc = M.bit_length() - 1
    return (R + lc * (M // 2)) * _G1_MUL


def work(case):
    kind = case["kind"]
    if kind == "msm":
        n, nb = case["n"], case["nbatch"]
        return {"bytes": 96 * n + 32 * n * nb + 96 * nb, "flops": _FQ * _MSM_TERM * n * nb}
    if kind == "batch":
        nbytes = muls = 0
        for j in I.batched_jobs(case["mix"], case["jobs"], case["log_min"], case["log_max"]):
            R, M = 1 << (j["log_n"] // 2), 1 << (j["log_n"] - j["log_n"] // 2)
            nbytes += 32 * R * M + 576 + _state_bytes(R, M, j["b"])
            muls += _commit_muls(R, M) + _step1_muls(R, j["b"]) + _step2_muls(R, M)
        return {"bytes": nbytes, "flops": _FQ * muls}
    if kind == "segments":
        R, b = 1 << case["log_r"], case["b"]
        K, out = -(-R // b), 1344 * case["log_r"] + 480
        return {"bytes": 96 * R + 192 * (2 * R - 1) + 96 * R + K * out, "flops": _FQ * _step1_muls(R, b)}
    log_n = case["log_n"]
    R, M = 1 << (log_n // 2), 1 << (log_n - log_n // 2)
    N, lr, lc = R * M, log_n // 2, log_n - log_n // 2
    pi = 1344 * lr + 480
    check = (2 * lr + 4) * _MILLER + 4 * _FINAL_EXP
    if kind == "open":
        b = case["b"]
        return {"bytes": 32 * N + 576 + 96 * R + _state_bytes(R, M, b),
                "flops": _FQ * (_commit_muls(R, M) + _step1_muls(R, b) + _step2_muls(R, M))}
    if kind == "eval":
        muls = _step1_muls(R, R) + M * _G1_MUL + R * _G1_MUL + 2 * check
        return {"bytes": 32 * N + 96 * R + 192 * (2 * R - 1) + 96 * (2 * M - 1) + 2 * (128 + pi + 96 * lc),
                "flops": _FQ * muls}
    b = case["b"]
    K = -(-R // b)
    if kind == "one":
        nbytes = 576 + 32 + 96 * b + pi + 32 * log_n + lr * 128 + 96 * lc
        prove = -(-_step1_muls(R, b) // K) + _step2_muls(R, M)
        return {"bytes": 32 * N + 96 * R + 192 * (2 * R - 1) + 96 * (2 * M - 1) + 3 * nbytes,
                "flops": _FQ * (prove + 2 * (check + (lc + 1) * _MILLER + _FINAL_EXP + b * _G1_MUL))}
    return {"bytes": 32 * N + 96 * R + _state_bytes(R, M, b) + N,
            "flops": _FQ * (K * check + R * _G1_MUL + M * ((lc + 1) * _MILLER + _FINAL_EXP))}
