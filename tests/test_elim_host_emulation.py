"""Host emulation of the eliminated walk's generated kernels: the source that
perm_elim_source gives is compiled as host C++ under AddressSanitizer and
UndefinedBehaviorSanitizer, and chunks of outer Gray indices are run as one
lane.  A chunk of 2^K outer steps with k low columns is the Gray range of
2^(K+k) indices of the order (low columns, outer columns, last column); its sum
is compared with the oracle's (exact: bit for bit; FP64: within the rounding
bound 64 n 2^-53 sum|terms|), and a sub-range's with the plan's own order."""
import os
import re
import subprocess
import tempfile

import numpy as np
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2501_15126_gb300", "csrc")
U = 2.0 ** -53

HARNESS = r'''
#include "shim.h"
#include "walk.cu"
#include <cstdio>
#include <cstdlib>
int main(int argc, char **argv) {
    const int K = std::atoi(argv[1]);
    unsigned long long q;
    while (std::scanf("%llu", &q) == 1) {
        unsigned long long w[6] = {0, 0, 0, 0, 0, 0};
        const auto acc = pk::walk_chunk_elim<pk::ElimPol, pk::A>(q, K);
        pk::A::acc_store(w, acc);
        std::printf("%llu", q);
        for (int i = 0; i < pk::A::ACC_WORDS; ++i) std::printf(" %016llx", w[i]);
        std::printf("\n");
    }
    return 0;
}
'''


def emulate(source, K, chunks):
    with tempfile.TemporaryDirectory() as d:
        open(os.path.join(d, "walk.cu"), "w").write(source)
        open(os.path.join(d, "main.cpp"), "w").write(HARNESS)
        exe = os.path.join(d, "walk")
        subprocess.check_call(["g++", "-std=c++17", "-O1", "-fsanitize=address,undefined", "-fno-sanitize-recover=all",
                               "-ftrivial-auto-var-init=pattern", "-I", os.path.join(HERE, "host_emulation"), "-I", CSRC,
                               "-I", d, os.path.join(d, "main.cpp"), "-o", exe])
        out = subprocess.run([exe, str(K)], input=" ".join(map(str, chunks)), capture_output=True, text=True,
                             check=True).stdout
    return {int(f[0]): [int(x, 16) for x in f[1:]] for f in (line.split() for line in out.splitlines())}


def compare(src, words, ao, lo, hi):
    n = ao.shape[0]
    m = re.search(r"typedef ArithExact<(\d+)> A;", src)
    if m:
        mask = (1 << min(128, 32 * int(m.group(1)))) - 1   # the oracle is exact modulo 2^128
        assert sum(w << (64 * i) for i, w in enumerate(words)) & mask == oracle.nw2_range(ao, lo, hi) & mask
        return
    s, sa = oracle.nw_range(ao, lo, hi)
    hi_w, lo_w, ab = np.array(words, dtype=np.uint64).view(np.float64)
    scale = int(re.search(r"int scale = (-?\d+);", src).group(1))
    assert abs(np.ldexp(hi_w + lo_w, scale) - float(s)) <= 64 * n * U * float(sa)
    if "kAbs = true" in src:
        assert abs(np.ldexp(ab, scale) - float(sa)) <= 1e-4 * float(sa)


def scaled_rows(n, p, seed):
    """Rows of magnitudes 2^-300..2^300: partial products leave FP64's range unless rows are scaled."""
    a = synth.single_er(n, p, seed, values="f64")
    return a * np.exp2(np.linspace(-300, 300, n).round())[:, None]


CASES = [
    ("er24_01", lambda: synth.single_er(24, 0.2, 1, values="01"), {}),
    ("er24_f64_abs", lambda: synth.single_er(24, 0.2, 1, values="f64"), {}),
    ("er36_f64", lambda: synth.single_er(36, 0.15, 2, values="f64", shuffle_cols=True), {}),
    ("er36_f64_abs", lambda: synth.single_er(36, 0.15, 2, values="f64"), {"flags": A.PERM_FLAG_ABS_SUM}),
    ("band48_01", lambda: synth.band_plus(48, 3, 2, seed=3, values="01"), {}),
    ("signed_ints", lambda: synth.single_er(26, 0.15, 9, values="01") * np.random.default_rng(9).integers(-40, 41, (26, 26)), {"exact_words": 3}),
    ("signed_reals", lambda: synth.single_er(25, 0.15, 8, values="f64") - 0.4 * synth.single_er(25, 0.15, 8, values="01"), {}),
    ("scaled_rows", lambda: scaled_rows(26, 0.15, 5), {}),
    ("n64_f64", lambda: synth.single_er(64, 0.08, 64, values="f64"), {"flags": A.PERM_FLAG_ABS_SUM}),
]


@pytest.mark.parametrize("name,make,kw", CASES, ids=[c[0] for c in CASES])
def test_chunks_of_the_outer_walk_equal_the_oracle(name, make, kw):
    a = make()
    src, k, order = A.elim_source(a, **kw)
    n = a.shape[0]
    h = n - 1 - k
    assert k >= 2 and sorted(order) == list(range(n))
    ao = np.ascontiguousarray(a[:, order[h:n - 1] + order[:h] + order[n - 1:]])
    for K in sorted({0, max(0, 13 - k)}):   # a single step, and ranges of at least 2^13 indices
        top = 1 << (h - K)
        chunks = sorted({0, 1, top // 3, top - 1})
        got = emulate(src, K, chunks)
        for q in chunks:
            compare(src, got[q], ao, (q << K) << k, ((q + 1) << K) << k)


@pytest.mark.parametrize("values", ["01", "f64"])
def test_a_sub_range_keeps_the_plans_partial_sum(values):
    """[q 2^a, (q+1) 2^a) in the plan's order: only the a low positions are reordered and summed out."""
    a_mat = synth.band_plus(30, 2, 1, seed=4, values=values)
    a = 20
    plan = np.ascontiguousarray(a_mat[:, list(A.inspect(a_mat).col_order)[:30]])
    for q in (0, 5, (1 << 9) - 1):
        kw = {"g_lo": q << a, "g_hi": (q + 1) << a, "flags": A.PERM_FLAG_ABS_SUM}
        if q == 0:
            kw["g_lo"] = 0
        src, k, _ = A.elim_source(a_mat, **kw)
        assert k >= 2
        compare(src, emulate(src, a - k, [q])[q], plan, q << a, (q + 1) << a)


def test_what_keeps_the_chained_walk():
    """Explicit orders, splits, chunks, schemes and deadlines, dense patterns and zero-span walks."""
    a = synth.single_er(24, 0.2, 1, values="f64")
    assert A.elim_source(a)[1] > 0
    for kw in ({"ordering": A.PERM_ORDER_PAPER}, {"reg_rows": 10}, {"shared_rows": 2}, {"chunk_log2": 9}, {"threads": 256},
               {"timeout_ms": 5}, {"flags": A.PERM_FLAG_PURE_REG}, {"flags": A.PERM_FLAG_PAIRED_CHAIN}, {"gr_ratio": 2.0}):
        assert A.elim_source(a, **kw)[1] == 0, kw
    assert A.elim_source(synth.ones(20))[1] == 0
    assert A.elim_source(synth.table2_like("bcspwr02"))[1] == 0
