"""The host rules that cut the launchers' work (csrc/split_rules.cuh), on the CPU: compiled with the
host compiler and compared, over the whole range of sizes, with what a device would do with them."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 152

SRC = """
#include "split_rules.cuh"
using namespace estp;
extern "C" void lm(int64_t n_rb, int64_t n_unit, int64_t s_min, int64_t sms, int64_t* S, int* gran) {
    const LmSplit r = lm_split(n_rb, n_unit, s_min, sms);
    *S = r.S;
    *gran = r.gran;
}
extern "C" int64_t part_bytes(int B, int64_t sumT, int64_t longest, int n_heads, int n_groups, int sms) {
    return f32_part_bytes(f32_split(B, sumT, longest, n_heads, n_groups, sms), sumT, longest, n_heads, n_groups);
}
extern "C" int split(int B, int64_t sumT, int64_t longest, int n_heads, int n_groups, int sms) {
    const F32Split s = f32_split(B, sumT, longest, n_heads, n_groups, sms);
    return s.rows * 100 + s.qc * 10 + (s.per_head ? 1 : 0);
}
extern "C" int64_t begin(int64_t n_k, int bk, int rank, int ranks) { return rank_begin(n_k, bk, rank, ranks); }
extern "C" int ranks(int64_t tiles, int64_t n_k, int sms) { return wide_ranks(tiles, n_k, sms); }
extern "C" int64_t ranges(int64_t sumT, int64_t row_bytes, int B, int64_t full, int n_slices, int sms) {
    return pool_ranges(sumT, row_bytes, B, full, n_slices, sms);
}
extern "C" int pairs(int B, int64_t sumT, int n_groups, int sms) { return imp_pairs(B, sumT, n_groups, 256, sms); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SRC)
    lib = str(d / "rules.so")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Wextra", "-Werror", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2608_15592_gb300", "csrc"), str(d / "rules.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _up(a, b):
    return -(-a // b)


# ------------------------------------------------------------ entropy from hidden states
def _lm(rules, n_rb, n_unit, s_min):
    S, gran = ctypes.c_int64(), ctypes.c_int()
    i = ctypes.c_int64
    rules.lm(i(n_rb), i(n_unit), i(s_min), i(SMS), ctypes.byref(S), ctypes.byref(gran))
    return S.value, gran.value


def _lm_time(u):
    """An item of u units in units of a full tile's: a last tile that is not full is loaded unit by unit."""
    return u // 8 * 8 + (2 + 1.6 * (u % 8) if u % 8 else 0)


def _lm_cost(n_rb, n_unit, S, gran):
    """What the busiest SM has to do: items round-robin, split fastest, each with its tiles and its
    share of one more pass of W."""
    n = _up(n_unit, gran)
    cut = [sp * n // S * gran for sp in range(S + 1)]
    assert cut[0] == 0 and cut[-1] >= n_unit and all(b > a for a, b in zip(cut, cut[1:]))
    time = [_lm_time(b - a) for a, b in zip(cut, cut[1:])]
    load = [0] * SMS
    for item in range(n_rb * S):
        load[item % SMS] += time[item % S] + n_unit / 80
    return max(load)


@pytest.mark.parametrize("V", [5000, 8000, 11948, 32000, 50257, 128256, 152064])
def test_lm_split_leaves_no_sm_idle(rules, V):
    n_unit = _up(V, 32)
    rng = random.Random(V)
    for n_rb in {2, 3, 5, 10, 36, 46, 66, 71, 77, 116, 130, 143, 170, *(rng.randint(2, 470) for _ in range(30))}:
        for s_min in (1, 2, 4):  # D up to 1280, 2048, 4096
            S, gran = _lm(rules, n_rb, n_unit, s_min)
            assert s_min <= S <= _up(n_unit, gran)
            got = _lm_cost(n_rb, n_unit, S, gran)
            # every number of whole-tile splits the kernel could take, up to sixteen items an SM
            top = max(4 * s_min, _up(16 * SMS, n_rb))
            best = min(_lm_cost(n_rb, n_unit, s, 8) for s in range(s_min, min(top, _up(n_unit, 8)) + 1))
            # (the rule takes every item for the largest, a real SM has some smaller ones)
            assert got <= 1.06 * best + 8, (n_rb, s_min, S, gran, got, best)


def test_lm_split_of_one_row_block(rules):
    for V in (1, 31, 1000, 5000, 32000, 128256, 152064):
        n_unit = _up(V, 32)
        assert _lm(rules, 1, n_unit, 1) == (min(SMS, n_unit), 1), V


@pytest.mark.parametrize("n_rb,n_unit,s_min", [(1, 1, 1), (1, 2, 4), (3, 4, 13), (470, 1, 1), (5000, 4008, 4)])
def test_lm_split_small(rules, n_rb, n_unit, s_min):
    S, gran = _lm(rules, n_rb, n_unit, s_min)
    assert 1 <= S <= _up(n_unit, gran)
    _lm_cost(n_rb, n_unit, S, gran)


# ------------------------------------------------------------------- column sums (bf16)
def _items(n, qc):
    return sum(_up(m, qc) for m in range(1, n + 1))


@pytest.mark.parametrize("n_groups", [1, 2, 4, 8, 16])
def test_column_sum_items_of_one_pair_fit_the_sms(rules, n_groups):
    for B in (1, 2, 3, 4, 7, 8, 16, 40, 160):
        for T in (1, 100, 256, 257, 300, 700, 1000, 1500, 2300, 4000, 9000, 40000):
            nt = _up(T, 256)
            qc = rules.pairs(B, ctypes.c_int64(B * T), n_groups, SMS)
            items = B * n_groups * _items(nt, qc)
            if qc == 1:
                assert items <= SMS, (B, T)
            else:  # two pairs wherever one pair would not fit and longer items would leave SMs idle
                assert B * n_groups * _items(nt, 1) > SMS, (B, T)
                assert qc == 2 or items >= 16 * SMS, (B, T)


# ------------------------------------------------------------------- column sums (fp32)
@pytest.mark.parametrize("n_heads,n_groups", [(8, 8), (16, 4), (28, 4), (64, 8), (256, 1), (1, 1)])
def test_f32_partials_stay_bounded(rules, n_heads, n_groups):
    """No more than 64 MiB, or what chunks of 512 queries for each KV group take, however skewed the
    lengths and however loose the bound on them (at most the whole batch)."""
    i = ctypes.c_int64
    rules.part_bytes.restype = i
    for B in (1, 2, 8, 64, 256, 1000, 5000):
        for T in (1, 16, 100, 300, 1000, 4000):
            sumT = B * T
            for longest in {T, min(sumT, 8 * T), min(sumT, 131072)}:
                got = rules.part_bytes(B, i(sumT), i(longest), n_heads, n_groups, SMS)
                coarse = 4 * _up(_up(longest, 64), 8) * n_groups * sumT
                assert got <= max(coarse, 64 << 20), (B, T, longest, got, coarse)


def _f32_unlimited(B, sumT, n_heads, n_groups):
    rows, qc, per_head = 128, 8, False

    def enough():
        nt = _up(_up(sumT, B), rows)
        return B * (n_heads if per_head else n_groups) * _items(nt, qc) >= 8 * SMS

    per_head = per_head or not enough()
    while not enough() and qc > 1:
        qc //= 2
    if not enough():
        rows = 64
    return rows, qc, per_head


@pytest.mark.parametrize("n_heads,n_groups", [(8, 8), (16, 4), (28, 4), (1, 1)])
def test_f32_split_follows_the_items_within_the_bound(rules, n_heads, n_groups):
    i = ctypes.c_int64
    for B in (1, 2, 4, 32, 160):
        for T in (1, 16, 128, 300, 900, 1500, 4000):
            rows, qc, per_head = _f32_unlimited(B, B * T, n_heads, n_groups)
            if 4 * _up(_up(T, rows), qc) * (n_heads if per_head else n_groups) * B * T <= 64 << 20:
                got = rules.split(B, i(B * T), i(T), n_heads, n_groups, SMS)
                assert got == rows * 100 + qc * 10 + per_head, (B, T)


# ---------------------------------------------------------------------------- pooling
@pytest.mark.parametrize("row_bytes,ctas_per_sm,n_slices", [(2048, 8, 1), (4096, 4, 1), (7168, 2, 1), (8192, 2, 1),
                                                            (16384, 2, 2), (65536, 2, 8)])
def test_pool_ranges_balance_the_sms(rules, row_bytes, ctas_per_sm, n_slices):
    i = ctypes.c_int64
    rules.ranges.restype = i
    full = SMS * ctas_per_sm // n_slices
    for B in (1, 2, 8, 16, 64, 256):
        for T in (1, 2, 16, 58, 100, 300, 700, 2048, 8192):
            sumT = B * T
            G = rules.ranges(i(sumT), i(row_bytes), B, i(full), n_slices, SMS)
            assert 1 <= G <= min(full, sumT), (B, T)
            if sumT <= 16:
                assert G == min(full, sumT), (B, T, G)
            ctas = G * n_slices
            if sumT >= full and G < full:
                # no SM with two large CTAs among SMs with one, and no wave that is nearly full
                assert ctas <= SMS or ctas >= 2 * SMS or ctas_per_sm > 2, (B, T, G)
                assert ctas <= SMS or 6 * G < 5 * full, (B, T, G)
                # enough ranges in flight for the bytes, few enough slots to merge
                want = (sumT * row_bytes * B / 4000) ** 0.5
                assert 0.45 * want <= G <= want, (B, T, G)


# ----------------------------------------------------------------- wide products (MLP head)
@pytest.mark.parametrize("bk", [16, 32, 64])
def test_no_rank_of_a_wide_product_idles(rules, bk):
    i = ctypes.c_int64
    rules.begin.restype = i
    for n_k in [1, 15, 64, 127, 128, 255, 256, 1000, 1023, 1024, 1088, 1600, 2050, 4096, 5000, 8192, 12345]:
        for tiles in (1, 16, 38, 39, 76, 77, 152, 153, 1000):
            S = rules.ranks(i(tiles), i(n_k), SMS)
            assert S in (1, 2, 4, 8) and (S == 1 or (tiles * S <= 2 * SMS and n_k / S >= 128))
            cut = [rules.begin(i(n_k), bk, r, S) for r in range(S + 1)]
            assert cut[0] == 0 and cut[-1] == n_k and all(c % bk == 0 for c in cut[:-1])
            slices = [_up(b - a, bk) for a, b in zip(cut, cut[1:])]
            assert max(slices) - min(slices) <= 1 and min(slices) >= 1, (n_k, S, slices)
