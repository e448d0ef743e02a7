"""The library's host path on the CPU, its object files linked against a CUDA runtime that runs nothing
(tests/emu/fake_cudart.cpp): the order of work over streams and what a failing event call leaves behind."""
import ctypes
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
vp, u32, u64, sz = ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint64, ctypes.c_size_t


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2601_03031_gb300 import build as B
    gxx = shutil.which("g++")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    if not gxx or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("g++ or the CUDA headers not available")
    B.build()
    objs = [os.path.join(B.BUILD_DIR, os.path.basename(s) + ".o") for s in B.sources()]
    if any(not os.path.exists(o) for o in objs):
        B.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-I{inc}", "-o", out,
                           os.path.join(ROOT, "tests", "emu", "fake_cudart.cpp"), *objs])
    L = ctypes.CDLL(out)
    for f in ("fake_event_calls", "fake_bad_frees", "fake_late_launches"):
        getattr(L, f).restype = ctypes.c_long
    L.fake_log.restype = ctypes.c_char_p
    for f in ("vc_proof_len", "vc_segment_proof_len", "vc_eval_proof_len"):
        getattr(L, f).restype = sz
    return L


@pytest.fixture(scope="module")
def pp(lib):
    lib.fake_reset(ctypes.c_long(-1))
    h = vp()
    assert lib.vc_setup(u32(8), u32(3), u64(1), None, ctypes.byref(h)) == 0
    return h


@pytest.fixture(scope="module")
def cm(lib, pp):
    h = vp()
    assert lib.vc_commit(pp, ctypes.create_string_buffer(32 << 8), 0, None, ctypes.byref(h)) == 0
    return h


C = ctypes.create_string_buffer(576)
B = 3


def verify_one(lib, pp, cm):
    n = lib.vc_proof_len(pp, u32(B), u64(5))
    return lib.vc_verify(pp, C, u32(B), u64(5), (u64 * 4)(), ctypes.create_string_buffer(n), sz(n), None)


def verify_segment(lib, pp, cm):
    n = lib.vc_segment_proof_len(pp, u32(B), u32(4))
    return lib.vc_verify_segment(pp, C, u32(B), u32(4), (u64 * 64)(), ctypes.create_string_buffer(n), sz(n), None)


def verify_eval(lib, pp, cm):
    n = lib.vc_eval_proof_len(pp)
    return lib.vc_eval_verify(pp, C, ctypes.create_string_buffer(1024), ctypes.create_string_buffer(n), sz(n), None)


def verify_all(lib, pp, cm):
    return lib.vc_verify_all(pp, C, ctypes.create_string_buffer(32 << 8), 0, verify_all.pf, 0, None, None, None)


def run(lib, pp, cm, call, fail_at):
    """Status of the call whose fail_at-th event call fails (-1: none), how many event calls it made, buffers it
    freed under running work, and launches after the failure."""
    if call is verify_all:
        lib.fake_reset(ctypes.c_long(-1))
        verify_all.pf = vp()
        assert lib.vc_prove_all(pp, cm, u32(B), None, ctypes.byref(verify_all.pf)) == 0
    lib.fake_reset(ctypes.c_long(fail_at))
    st = call(lib, pp, cm)
    return st, lib.fake_event_calls(), lib.fake_bad_frees(), lib.fake_late_launches()


@pytest.mark.parametrize("call", [verify_one, verify_segment, verify_eval, verify_all])
def test_failed_joins_of_the_verifier(lib, pp, cm, call):
    """Whichever event call of a verification fails, the call says so (FP_EDEVICE), launches nothing after it
    and gives no buffer back that a side stream may still use."""
    st, calls, bad, _ = run(lib, pp, cm, call, -1)
    assert (st, bad) == (0, 0) and calls > 0
    for n in range(calls):
        st, _, bad, late = run(lib, pp, cm, call, n)
        assert (st, bad, late) == (3, 0, 0), n
        st, _, bad, _ = run(lib, pp, cm, call, -1)          # and the failure is not reported again
        assert (st, bad) == (0, 0), n


def prove_all(lib, pp, cm):
    pf = vp()
    st = lib.vc_prove_all(pp, cm, u32(B), None, ctypes.byref(pf))
    if st == 0:
        lib.fp_proofs_free(pf)
    return st


def prove_one(lib, pp, cm):
    n = lib.vc_proof_len(pp, u32(B), u64(5))
    return lib.vc_prove_one(pp, cm, u32(B), u64(5), None, ctypes.create_string_buffer(n), sz(n), ctypes.byref(sz()))


def eval_prove(lib, pp, cm):
    n = lib.vc_eval_proof_len(pp)
    return lib.vc_eval_prove(pp, cm, ctypes.create_string_buffer(1024), None, ctypes.create_string_buffer(n), sz(n),
                             ctypes.byref(sz()))


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("call", [prove_all, prove_one, eval_prove])
def test_failed_events_of_the_prover(lib, pp, cm, call, schedule):
    """The same for the proving calls, which work on up to seven internal streams, under both schedules."""
    lib.fp_set_schedule(schedule)
    try:
        st, calls, bad, _ = run(lib, pp, cm, call, -1)
        assert (st, bad) == (0, 0) and calls > 0
        for n in range(calls):
            st, _, bad, late = run(lib, pp, cm, call, n)
            assert (st, bad, late) == (3, 0, 0), n
            st, _, bad, _ = run(lib, pp, cm, call, -1)
            assert (st, bad) == (0, 0), n
    finally:
        lib.fp_set_schedule(0)


LIMITS = ["miller_block_max", "miller_warp_max", "miller_group_min", "commit_block_max", "commit_warp_max", "fe_block_max",
          "fe_warp_max", "pair_block_max", "fold_warp_max", "wterm_warp_max", "msm_chunks", "msm_segment_threads"]


def kernel(mangled):
    m = re.match(r"_ZN3fpk(\d+)", mangled)
    return mangled[m.end():m.end() + int(m.group(1))] if m else mangled


def launches(lib, fn, **limits):
    """[(kernel, grid, block)] of fn() under the given engine limits."""
    lim = (u32 * len(LIMITS))()
    lib.fp_engine_limits_default(lim)
    for k, v in limits.items():
        lim[LIMITS.index(k)] = v
    lib.fp_set_engine_limits(lim)
    try:
        lib.fake_reset(ctypes.c_long(-1))
        assert fn() == 0
        return [(kernel(w[0]), int(w[1]), int(w[2])) for w in (x.split() for x in lib.fake_log().decode().splitlines())]
    finally:
        lib.fp_set_engine_limits(None)


@pytest.mark.parametrize("pair_block_max", [0, 2, 1 << 16])
def test_fq12_products_keep_to_their_limit(lib, pp, cm, pair_block_max):
    """pair_block_max: rounds with more pairwise products than that run them one per thread."""
    log = launches(lib, lambda: prove_all(lib, pp, cm), pair_block_max=pair_block_max)
    threads = [g for n, g, _ in log if n == "k_fq12_pair"]
    blocks = [g for n, g, _ in log if n == "k_fq12_prod"]
    # R = 16, six blocks of up to 3 rows: 96, 48, 24 and 12 Miller values in the rounds, reduced to 12: halved 3, 2, 1
    # and 0 times, or by eights, fours and twos
    want = {0: (6, 0), 2: (6, 0), 1 << 16: (0, 3)}[pair_block_max]
    assert (len(threads), len(blocks)) == want, (threads, blocks)


@pytest.mark.parametrize("limits", [{}, {"miller_block_max": 0, "commit_block_max": 0}, {"fe_block_max": 1},
                                    {"fe_block_max": 0}, {"fe_block_max": 0, "fe_warp_max": 0},
                                    {"miller_block_max": 0, "miller_warp_max": 0, "miller_group_min": 64,
                                     "commit_block_max": 0, "commit_warp_max": 0}])
def test_pairing_launches_are_profiled_by_the_kernel_that_runs(lib, pp, limits):
    def work():
        h, pf = vp(), vp()
        st = lib.vc_commit(pp, ctypes.create_string_buffer(32 << 8), 0, None, ctypes.byref(h))
        st = st or lib.vc_prove_all(pp, h, u32(1), None, ctypes.byref(pf))
        if st == 0:
            lib.fp_proofs_free(pf)
            lib.fp_commit_free(h)
        return st

    def counts(names):
        return {n: sum(1 for x in names if x == n) for n in names if "miller" in n or "final_exp" in n}

    lib.fp_profile_report.restype = sz
    buf = ctypes.create_string_buffer(1 << 16)
    lib.fp_profile_enable(1)
    try:
        log = launches(lib, work, **limits)
    finally:
        lib.fp_profile_enable(0)
        lib.fp_profile_report(buf, sz(len(buf)))
    labels = {w[0]: int(w[1]) for w in (x.split() for x in buf.value.decode().splitlines())
              if "miller" in w[0] or "final_exp" in w[0]}
    assert labels == counts([n for n, _, _ in log])


@pytest.mark.parametrize("log_r,b,groups", [(10, 1024, 0), (11, 2048, 1), (11, 37, 7)])
def test_many_sparse_terms_take_the_groups(lib, log_r, b, groups):
    """L_j.1 / R_j.1 terms of a round: a block each up to 1024, above that 8 lanes each (16 terms per block)."""
    p, h = vp(), vp()
    assert lib.vc_setup_split(u32(log_r), u32(1), u32(b), u64(1), None, ctypes.byref(p)) == 0
    assert lib.vc_commit(p, ctypes.create_string_buffer(64 << log_r), 0, None, ctypes.byref(h)) == 0

    def work():
        pf = vp()
        st = lib.vc_open_segments(p, h, u32(b), u32(0), u32(0), None, ctypes.byref(pf))
        if st == 0:
            lib.fp_proofs_free(pf)
        return st

    R = 1 << log_r
    K = -(-R // b)
    terms = [K * min(b, R >> j) for j in range(log_r)]
    got = [(g, t) for n, g, t in launches(lib, work) if n.startswith("k_sparse_g")]
    assert got == [(n, 96) if n <= 1024 else (-(-n // 16), 128) for n in terms]
    assert sum(n > 1024 for n in terms) == groups
    lib.fp_commit_free(h)
    lib.fp_pp_free(p)


@pytest.mark.parametrize("nbatch", [1024, 1025])
def test_many_msm_batches_take_the_groups(lib, nbatch):
    """Horner over the windows of a sum: half a block each up to 1024 sums, above that 8 lanes each."""
    lib.fake_reset(ctypes.c_long(-1))
    bases = vp()
    assert lib.fp_g1_bases_from_scalars(vp(4096), u64(2), 1, None, ctypes.byref(bases)) == 0
    log = launches(lib, lambda: lib.fp_msm_g1(bases, vp(4096), u64(2), u32(nbatch), 1, 0, None, vp(8192)))
    got = [(n, g, t) for n, g, t in log if n.startswith("k_msm_final")]
    assert got == ([("k_msm_final_l", 512, 192)] if nbatch == 1024 else [("k_msm_final", 129, 64)])
    lib.fp_g1_bases_free(bases)


@pytest.mark.parametrize("log_c", [11, 12])
def test_many_evaluation_proof_terms_take_the_groups(lib, log_c):
    """The PST terms of an evaluation proof: half a block each up to 2048, above that 8 lanes each."""
    p, h = vp(), vp()
    assert lib.vc_setup_split(u32(1), u32(log_c), u32(1), u64(1), None, ctypes.byref(p)) == 0
    assert lib.vc_commit(p, ctypes.create_string_buffer(64 << log_c), 0, None, ctypes.byref(h)) == 0
    log = launches(lib, lambda: eval_prove(lib, p, h))
    assert [x for x in log if x[0].startswith("k_eval_pst_terms")] == \
        [("k_eval_pst_terms", 1024, 192) if log_c == 11 else ("k_eval_pst_terms8", 256, 128)]
    lib.fp_commit_free(h)
    lib.fp_pp_free(p)


@pytest.mark.parametrize("log_r,log_c,b,groups", [(5, 6, 32, set()), (11, 1, 2048, set()), (9, 1, 3, {"k_vb_muls8"}), (8, 1, 2, {"k_vb_muls8"}),
                                                  (12, 1, 1024, {"k_vb_muls8", "k_va_rows8"}), (1, 12, 2, {"k_va_colE8"}),
                                                  (1, 13, 2, {"k_va_colE8"}), (1, 14, 2, {"k_va_colE8", "k_vp_prod"})])
def test_many_multiplications_of_the_verifier_take_the_groups(lib, log_r, log_c, b, groups):
    """Rows and columns: half a block each up to 2048 per launch, block terms up to 2304, above that 8 lanes each; a
    column's product of pairings on a block up to 8192 of them, above that on a thread."""
    p, h, pf = vp(), vp(), vp()
    N = 1 << (log_r + log_c)
    assert lib.vc_setup_split(u32(log_r), u32(log_c), u32(b), u64(1), None, ctypes.byref(p)) == 0
    assert lib.vc_commit(p, ctypes.create_string_buffer(32 * N), 0, None, ctypes.byref(h)) == 0
    assert lib.vc_prove_all(p, h, u32(b), None, ctypes.byref(pf)) == 0
    log = launches(lib, lambda: lib.vc_verify_all(p, C, ctypes.create_string_buffer(32 * N), 0, pf, 0, None, None, None))
    K, tpb = -(-(1 << log_r) // b), 1
    used = b + 2 * log_r + 1
    while tpb < used:
        tpb *= 2
    at = {n: g for n, g, _ in log}
    assert {n for n in at if n in ("k_vb_muls8", "k_va_rows8", "k_va_colE8", "k_vp_prod")} == groups
    assert at["k_vb_muls"] == K + (0 if "k_vb_muls8" in groups else (K * tpb + K + 1) // 2)
    if "k_vb_muls8" in groups:
        assert at["k_vb_muls8"] == -(-(K * used + K) // 16)
    assert at.get("k_va_rows8") == ((1 << log_r) // 16 if "k_va_rows8" in groups else None)
    assert at.get("k_va_colE8") == ((1 << log_c) // 16 if "k_va_colE8" in groups else None)
    lib.fp_proofs_free(pf)
    lib.fp_commit_free(h)
    lib.fp_pp_free(p)
