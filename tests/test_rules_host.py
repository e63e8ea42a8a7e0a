"""The host rules that choose a sweep's form (jd_rules.h), compiled here for this host."""
import ctypes
import os
import subprocess

import pytest

from paper_2505_04328_gb300 import _build

NONE, NORMAL, UNIFORM, KS = range(4)
COST, CKPT, STORE, PAIR, CKPT_PAIR, REPLAY = range(6)

SRC = r"""
#include "jd_rules.h"
using namespace jd;
static long long paths = 1 << 20;   // of the descriptors below
static jd_problem_desc desc(int d, int law, double rate) {
  jd_problem_desc q{};
  q.d = d;
  q.T = 2.0;
  q.Nt = 64;
  q.lambda = rate * 32.0;
  q.jump_law = (jd_jump_law)law;
  q.M = paths;
  return q;
}
static FormKey key(int d, int f64, int law, double rate) {
  return form_key(d <= 2 ? d : d <= 4 ? 4 : 8, f64 != 0, desc(d, law, rate));
}
extern "C" {
void set_paths(long long M) { paths = M; }
double rate_of(int law, double lambda, double T, int Nt) { return jump_rate((jd_jump_law)law, lambda, T, Nt); }
int chunk_len(int d, int law, double rate, int most) { return fwd_chunk_len(key(d, 0, law, rate).rate, most); }
int chunks(int d, int f64, int law, double rate, int kind) {
  return fwd_chunks(key(d, f64, law, rate), (SweepKind)kind);
}
long long pre_max(int d, int f64, int law, double rate, int kind) {
  return pre_max_paths(key(d, f64, law, rate), (SweepKind)kind);
}
long long pre_top(int d, int f64) { return pre_top_paths(d, f64 != 0); }
int one_slot(int f64, int ring, double rate) { return fb_one_slot(f64 != 0, ring, rate); }
int log_capacity(int f64, int law, double rate, int Nt) {
  jd_problem_desc q{};
  q.T = 1.0;
  q.Nt = Nt;
  q.lambda = rate * Nt;
  q.jump_law = (jd_jump_law)law;
  q.prec = f64 ? JD_FP64 : JD_FP32;
  return fb_log_capacity(q);
}
int log_fits(long long bytes, long long free_bytes) { return fb_log_fits((size_t)bytes, (size_t)free_bytes); }
int ks_short(double rate) { return ks_one_jump(rate); }
int keeps(int d, int f64, int law, double rate) { return theta_keeps(key(d, f64, law, rate)); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, lib = os.path.join(d, "rules.cpp"), os.path.join(d, "rules.so")
    with open(src, "w") as f:
        f.write(SRC)
    r = subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-Wno-unused-function", "-shared", "-fPIC",
                        "-I", _build.CSRC, "-I", _build.INCLUDE, src, "-o", lib], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    so = ctypes.CDLL(lib)
    so.rate_of.restype = ctypes.c_double
    so.pre_max.restype = so.pre_top.restype = ctypes.c_longlong

    class Rules:
        @staticmethod
        def rate(law, lam, T, Nt):
            return so.rate_of(law, ctypes.c_double(lam), ctypes.c_double(T), Nt)

        @staticmethod
        def chunk_len(d, law, rate, most=16):
            return so.chunk_len(d, law, ctypes.c_double(rate), most)

        @staticmethod
        def chunks(d, f64, law, rate, kind, M=1 << 20):
            so.set_paths(ctypes.c_longlong(M))
            return bool(so.chunks(d, int(f64), law, ctypes.c_double(rate), kind))

        @staticmethod
        def pre_max(d, f64, law, rate, kind):
            return so.pre_max(d, int(f64), law, ctypes.c_double(rate), kind)

        @staticmethod
        def pre_top(d, f64):
            return so.pre_top(d, int(f64))

        @staticmethod
        def one_slot(f64, ring, rate):
            return bool(so.one_slot(int(f64), ring, ctypes.c_double(rate)))

        @staticmethod
        def log_capacity(f64, law, rate, Nt):
            return so.log_capacity(int(f64), law, ctypes.c_double(rate), Nt)

        @staticmethod
        def log_fits(need, free):
            return bool(so.log_fits(ctypes.c_longlong(need), ctypes.c_longlong(free)))

        @staticmethod
        def ks_short(rate):
            return bool(so.ks_short(ctypes.c_double(rate)))

        @staticmethod
        def keeps(d, f64, law, rate):
            return bool(so.keeps(d, int(f64), law, ctypes.c_double(rate)))

    return Rules


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("d", [1, 2, 4, 8])
def test_a_problem_without_a_jump_law_has_no_rate(rules, d, f64):
    """Its intensity may be set: every form is then the one of rate 0 (FP32 d = 8 store sweep
    without jumps 0.473 -> 0.508 ms in the form for jumps)."""
    assert rules.rate(NONE, 5.0, 2.0, 100) == 0.0 and rules.rate(NORMAL, 5.0, 2.0, 100) == 0.1
    for rate in (0.002, 0.01, 0.05, 0.3):
        assert rules.chunk_len(d, NONE, rate) == 16
        for kind in (COST, STORE, REPLAY):
            assert rules.chunks(d, f64, NONE, rate, kind) == rules.chunks(d, f64, NORMAL, 0.0, kind)
        assert rules.keeps(d, f64, NONE, rate) == rules.keeps(d, f64, NORMAL, 0.0)
    if d > 2:
        assert not any(rules.chunks(d, f64, NONE, 0.01, kind) for kind in (COST, STORE, REPLAY))


@pytest.mark.parametrize("f64", [False, True])
def test_warp_wide_draws_need_a_one_jump_path(rules, f64):
    """Keilson-Storer steps of d > 2, and dimensions whose slot words are packed for fewer
    pairs than compiled (d = 5, 6 in the kernels of d = 8), have no one-jump path: the
    warp-wide form would cost and give nothing (KS d = 8, FP32, 0.02: store 1.52 -> 1.83 ms)."""
    rates = (0.002, 0.006, 0.012, 0.02, 0.05, 0.08)
    kinds = (COST, STORE, REPLAY)
    for d in (3, 4, 7, 8):
        assert not any(rules.chunks(d, f64, KS, r, k) for r in rates for k in kinds)
        assert any(rules.chunks(d, f64, NORMAL, r, k) for r in rates for k in kinds)
    for d in (5, 6):
        assert not any(rules.chunks(d, f64, law, r, k) for law in (NORMAL, UNIFORM, KS) for r in rates for k in kinds)


# (d, f64, law, kind, rate, in chunks): beside each line the launch step by step -> in chunks, ms
CHUNKS = [
    (2, False, UNIFORM, REPLAY, 0.07, True),    # 3.95 -> 3.78
    (2, False, UNIFORM, REPLAY, 0.1, False),    # 5.26 -> 5.68
    (2, False, KS, REPLAY, 0.2, False),         # 12.6 -> 14.5
    (1, False, NORMAL, REPLAY, 0.3, True),      # 14.8 -> 14.2
    (2, False, UNIFORM, STORE, 0.5, True),      # 3.23 -> 3.06
    (2, False, UNIFORM, STORE, 0.8, False),     # 3.87 -> 4.82
    (2, False, UNIFORM, PAIR, 0.8, False),      # 7.65 -> 9.41
    (2, True, UNIFORM, COST, 0.2, True),       # 3.22 -> 2.95
    (2, True, UNIFORM, COST, 0.4, False),      # 4.42 -> 4.71
    (1, True, NORMAL, STORE, 0.4, True),        # 4.64 -> 4.04
    (1, True, NORMAL, STORE, 0.8, False),       # 5.98 -> 6.81
    (2, True, KS, STORE, 0.0, False),           # 0.71 -> 0.79
    (2, True, KS, PAIR, 0.003, False),          # 1.17 -> 1.25
    (2, True, KS, STORE, 0.006, True),          # 1.04 -> 0.96
    (2, True, KS, COST, 0.4, True),             # 5.27 -> 5.12
    (2, True, KS, PAIR, 0.6, False),            # 10.8 -> 12.0
    (2, True, UNIFORM, STORE, 0.0, True),       # 0.81 -> 0.79
    (1, False, NORMAL, COST, 0.002, False),    # 0.945 -> 0.977
    (1, False, NORMAL, COST, 0.008, True),     # 1.20 -> 1.13
    (2, False, UNIFORM, COST, 0.0, True),      # 0.934 -> 0.894
    (2, False, UNIFORM, PAIR, 0.003, True),     # 1.417 -> 1.365 stored
]


@pytest.mark.parametrize("d,f64,law,kind,rate,want", CHUNKS)
def test_chunks_where_they_are_faster(rules, d, f64, law, kind, rate, want):
    assert rules.chunks(d, f64, law, rate, kind) == want


# (d, f64, law, rate, kept): the recompute adjoint with parameter gradients, regenerated -> kept, ms
KEPT = [
    (1, False, NORMAL, 0.0, False),    # 1.29 -> 1.33
    (2, False, NONE, 0.05, False),     # 1.55 -> 1.56
    (2, False, UNIFORM, 0.0002, True),  # 1.66 -> 1.58
    (4, False, NORMAL, 0.0002, False),  # 0.60 -> 0.64
    (4, False, NORMAL, 0.002, True),   # 1.36 -> 0.65
    (4, False, NORMAL, 0.1, False),    # 11.3 -> 11.6
    (2, False, UNIFORM, 0.1, True),    # 20.0 -> 17.6
    (2, False, KS, 0.12, False),       # 24.0 -> 25.3
    (2, False, UNIFORM, 0.2, False),   # 28.7 -> 36.1
    (2, True, UNIFORM, 0.14, True),    # 7.68 -> 7.34
    (1, True, NORMAL, 0.2, False),     # 8.80 -> 8.85
]


@pytest.mark.parametrize("d,f64,law,rate,want", KEPT)
def test_jump_draws_kept_where_that_is_faster(rules, d, f64, law, rate, want):
    assert rules.keeps(d, f64, law, rate) == want


def test_keilson_storer_short_path_ends_at_high_rates(rules):
    """FP32 store sweep, all steps by the general routine -> with the short path: 1.93 -> 1.16
    ms at 0.2, 3.24 -> 3.59 at 0.55."""
    assert rules.ks_short(0.2) and not rules.ks_short(0.55)


def test_four_components_draw_warp_wide_where_that_gains(rules):
    """FP32 d = 4: the store sweep gains at no rate for every size (M = 50,001 at 0.03: 0.271 ->
    0.281 ms), the cost and checkpoint sweeps around 0.02, the replay in a wide range."""
    for rate in (0.008, 0.012, 0.02, 0.03, 0.05):
        assert not rules.chunks(4, False, NORMAL, rate, STORE)
        assert rules.chunks(4, False, NORMAL, rate, REPLAY)
    assert rules.chunks(4, False, NORMAL, 0.02, COST)
    assert not rules.chunks(4, False, NORMAL, 0.03, COST) and not rules.chunks(4, False, NORMAL, 0.009, COST)


# (d, f64, kind, rate, M, pre-drawn): the sweep in the other form -> pre-drawn, us
PRE = [
    (1, False, STORE, 0.002, 2500, False),       # 52 -> 60
    (1, False, STORE, 0.002, 5500, False),       # 53 -> 67
    (1, False, COST, 0.002, 5500, True),         # 59 -> 50
    (1, False, PAIR, 0.0005, 3000, False),       # 48 -> 74
    (1, False, CKPT_PAIR, 0.007, 3000, True),    # 67 -> 60
    (1, False, CKPT, 0.0005, 3000, True),        # 57 -> 50
    (2, False, CKPT, 0.002, 4800, False),        # 55 -> 63
    (2, False, STORE, 0.002, 4800, False),       # 59 -> 67
    (2, False, COST, 0.02, 5500, True),
    (1, False, STORE, 0.02, 1000, True),
    (1, True, STORE, 0.002, 7500, True),         # 488 -> 378
    (1, True, PAIR, 0.002, 7500, False),         # 610 -> 735
    (2, True, PAIR, 0.002, 5500, False),         # 866 -> 1041
    (2, True, STORE, 0.002, 5500, True),         # 627 -> 547
    (2, True, PAIR, 0.2, 6000, True),            # 3189 -> 2890
    (1, True, PAIR, 0.03, 7200, True),           # 955 -> 904
]


@pytest.mark.parametrize("d,f64,kind,rate,M,want", PRE)
def test_pre_drawn_sweeps_where_they_are_faster(rules, d, f64, kind, rate, M, want):
    assert (M <= rules.pre_max(d, f64, NORMAL, rate, kind)) == want


@pytest.mark.parametrize("f64", [False, True])
def test_pre_pass_buffers_cover_every_rate(rules, f64):
    rates = (0.0, 0.001, 0.004, 0.005, 0.01, 0.03, 0.05, 0.3, 2.0)
    for d in (1, 2):
        for kind in (COST, CKPT, STORE, PAIR, CKPT_PAIR):
            limits = [rules.pre_max(d, f64, NORMAL, r, kind) for r in rates]
            assert f64 or limits == sorted(limits)
            assert max(limits) <= rules.pre_top(d, f64)
    assert rules.pre_max(4, f64, NORMAL, 0.1, COST) == rules.pre_top(4, f64) == 0


def test_forms_by_the_number_of_paths(rules):
    """FP32 d = 2 replay at high rates: in chunks while its blocks are resident (M = 80,000 1.37
    -> 1.21 ms at 0.2, 110,000 1.55 -> 2.11).  FP32 d = 4 warp-wide draws: from a full chip on
    (replay at 0.05, M = 8000 0.256 -> 0.285, 40,000 0.434 -> 0.398)."""
    for law in (UNIFORM, KS):
        assert rules.chunks(2, False, law, 0.2, REPLAY, M=13000) and rules.chunks(2, False, law, 0.2, REPLAY, M=80000)
        assert not rules.chunks(2, False, law, 0.2, REPLAY, M=110000)
    for kind, M in ((REPLAY, 8000), (COST, 8000), (CKPT, 20000)):
        assert not rules.chunks(4, False, NORMAL, 0.02, kind, M=M)
        assert rules.chunks(4, False, NORMAL, 0.02, kind, M=80000)


def test_feedback_straight_one_jump_code_where_it_is_faster(rules):
    """Independent paths (ring kind 0), FP32 4 x 4: 765 -> 720 us at 0.2, 880 -> 927 at 0.3; rings
    of 200 (kind 2): 686 -> 648 at 0.1, 762 -> 801 at 0.15; FP64 gains at no rate."""
    assert rules.one_slot(False, 0, 0.2) and not rules.one_slot(False, 0, 0.3)
    assert rules.one_slot(False, 1, 0.2)
    for ring in (2, 3):
        assert rules.one_slot(False, ring, 0.1) and not rules.one_slot(False, ring, 0.15)
    assert not any(rules.one_slot(True, ring, r) for ring in range(4) for r in (0.0, 0.02, 0.1, 1.0))


def test_feedback_log_capacity(rules):
    """The centering problem's 18 records as before; in FP32 no more than the steps before the
    first one with three jumps need (642 records at 0.5 and 1000 steps before); at least one."""
    for f64 in (False, True):
        assert rules.log_capacity(f64, KS, 0.0178, 100) == 18
        assert rules.log_capacity(f64, KS, 0.0, 100) == 0 and rules.log_capacity(f64, NONE, 0.1, 100) == 0
    assert rules.log_capacity(True, KS, 0.5, 1000) == 643
    assert 69 * 0.5 * 2 < rules.log_capacity(False, KS, 0.5, 1000) < 230
    # p3 = 0.9938: 1.0063 logged steps on average, four times that rounds up to 5, two records each
    assert rules.log_capacity(False, KS, 9.0, 45) == 10
    rates = (1e-7, 1e-4, 0.01, 0.0499, 0.0501, 0.2)
    caps = [rules.log_capacity(False, KS, r, 100) for r in rates]
    assert caps == sorted(caps) and caps == [rules.log_capacity(True, KS, r, 100) for r in rates]


def test_feedback_log_leaves_room_for_others(rules):
    """The default memory budget is half of what is free; a log of that size would leave a second
    problem with the same default half of the rest."""
    assert rules.log_fits(1 << 30, 4 << 30) and not rules.log_fits((1 << 30) + 1, 4 << 30)
    assert not rules.log_fits(1, 3) and rules.log_fits(70 << 30, 283 << 30)
