"""Host emulation of the precompiled eliminated walk: vm_impl.cuh is compiled
as host C++ under AddressSanitizer and UndefinedBehaviorSanitizer and runs the
program images that the library builds for the GPU (perm_elim_image), one lane
at a time, with the image and the slot area in heap buffers of exactly their
sizes.  A chunk of 2^K outer steps is the Gray range of 2^(K+k) indices of the
order (low columns, outer columns, last column); its sum is compared with the
oracle's (exact: bit for bit; FP64: within 64 n 2^-53 sum|terms|;
double-double: within n 2^-60 sum|terms|, the oracle's own precision on x86)."""
import os
import subprocess
import tempfile

import numpy as np
import pytest

import oracle
from paper_2501_15126_gb300 import _abi as A
from paper_2501_15126_gb300 import synth
from tests.test_elim_host_emulation import scaled_rows

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2501_15126_gb300", "csrc")
U = 2.0 ** -53

HARNESS = r'''
#include "shim.h"
#include "vm_impl.cuh"
#include <cstdio>
#include <cstdlib>
int main(int argc, char **argv) {
    FILE *f = std::fopen(argv[1], "rb");
    std::fseek(f, 0, SEEK_END);
    const long bytes = std::ftell(f);
    std::fseek(f, 0, SEEK_SET);
    unsigned char *img = (unsigned char *)std::aligned_alloc(16, (size_t)bytes);
    if (std::fread(img, 1, (size_t)bytes, f) != (size_t)bytes) return 3;
    std::fclose(f);
    const pk::VmHeader *H = reinterpret_cast<const pk::VmHeader *>(img);
    const size_t area_bytes = 32 * ((size_t)PERM_TEST_LANE * H->nslots + (size_t)PERM_TEST_EXTRA * H->nextra);
    unsigned char *area = (unsigned char *)std::aligned_alloc(16, area_bytes);
    const int K = std::atoi(argv[2]);
    unsigned long long q;
    while (std::scanf("%llu", &q) == 1) {
        unsigned long long w[6] = {0, 0, 0, 0, 0, 0};
        const auto acc = pk::vm_chunk<PERM_TEST_VM>(img, area, (int)(q % 32), q, K);
        PERM_TEST_VM::A::acc_store(w, acc);
        std::printf("%llu", q);
        for (int i = 0; i < PERM_TEST_VM::A::ACC_WORDS; ++i) std::printf(" %016llx", w[i]);
        std::printf("\n");
    }
    std::free(img);
    std::free(area);
    return 0;
}
'''


def emulate(img, kind, K, chunks):
    vm, lane, extra = {0: ("pk::VmF64", 8, 4), 1: ("pk::VmDD", 16, 4)}.get(
        kind, ("pk::VmExact<%d>" % (kind // 2), 8, 8 * ((kind // 2 + 1) // 2)))
    with tempfile.TemporaryDirectory() as d:
        open(os.path.join(d, "image.bin"), "wb").write(img)
        open(os.path.join(d, "main.cpp"), "w").write(HARNESS)
        exe = os.path.join(d, "walk")
        subprocess.check_call(["g++", "-std=c++17", "-O1", "-fsanitize=address,undefined", "-fno-sanitize-recover=all",
                               "-ftrivial-auto-var-init=pattern", "-DPERM_TEST_VM=" + vm, "-DPERM_TEST_LANE=%d" % lane,
                               "-DPERM_TEST_EXTRA=%d" % extra, "-I", os.path.join(HERE, "host_emulation"), "-I", CSRC,
                               os.path.join(d, "main.cpp"), "-o", exe])
        out = subprocess.run([exe, os.path.join(d, "image.bin"), str(K)], input=" ".join(map(str, chunks)),
                             capture_output=True, text=True, check=True).stdout
    return {int(f[0]): [int(x, 16) for x in f[1:]] for f in (line.split() for line in out.splitlines())}


def compare(words, kind, scale, shift, ao, lo, hi):
    n = ao.shape[0]
    if kind >= 2:
        mask = (1 << min(128, 32 * (kind // 2))) - 1
        assert sum(w << (64 * i) for i, w in enumerate(words)) & mask == oracle.nw2_range(ao, lo, hi) & mask
        return
    s, sa = oracle.nw_range(ao, lo, hi)
    h, l, ab = np.array(words, dtype=np.uint64).view(np.float64)
    bound = (64 * n * U if kind == 0 else n * 2.0 ** -60) * float(sa)
    assert abs((np.ldexp(h, scale) - s.hi) + (np.ldexp(l, scale) - s.lo)) <= bound
    assert abs(np.ldexp(ab, shift) - float(sa)) <= 1e-4 * float(sa)


def signed_reals(n, p, seed):
    return synth.single_er(n, p, seed, values="f64") - 0.4 * synth.single_er(n, p, seed, values="01")


def signed_ints(n, p, seed, top):
    return synth.single_er(n, p, seed, values="01") * np.random.default_rng(seed).integers(-top, top + 1, (n, n)) \
        + np.eye(n, dtype=np.int64) * (2 * top + 1)


CASES = [
    ("n9_01", lambda: synth.single_er(9, 0.3, 1, values="01"), {}),
    ("n12_f64", lambda: synth.single_er(12, 0.4, 2, values="f64"), {}),
    ("n24_01", lambda: synth.single_er(24, 0.2, 1, values="01"), {}),
    ("n24_f64", lambda: synth.single_er(24, 0.2, 1, values="f64"), {}),
    ("n28_dense_f64", lambda: synth.single_er(28, 0.35, 3, values="f64"), {}),
    ("n23_dd", lambda: signed_reals(23, 0.2, 4), {"precision": A.PERM_PREC_DD}),
    ("n26_scaled_rows", lambda: scaled_rows(26, 0.15, 5), {}),
    ("n26_signed_f64", lambda: signed_reals(26, 0.2, 6), {}),
    ("n28_01_96", lambda: synth.single_er(28, 0.25, 7, values="01"), {}),
    ("n25_ints_128", lambda: signed_ints(25, 0.15, 8, 3), {"exact_words": 2}),
    ("n24_ints_192", lambda: signed_ints(24, 0.15, 9, 30), {"exact_words": 3}),
    ("n27_160", lambda: signed_ints(27, 0.12, 10, 2), {}),
    ("n48_band_01", lambda: synth.band_plus(48, 3, 2, seed=3, values="01"), {}),
    ("n40_f64", lambda: synth.single_er(40, 0.08, 11, values="f64"), {}),
]


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("name,make,kw", CASES, ids=[c[0] for c in CASES])
def test_program_images_equal_the_oracle(name, make, kw, shared):
    a = make()
    img, kind, k, order, scale, shift = A.elim_image(a, shared_launch=shared, **kw)
    n = a.shape[0]
    if not img:
        pytest.skip("the chained walk runs this size")
    h = n - 1 - k
    assert sorted(order) == list(range(n))
    ao = np.ascontiguousarray(a[:, order[h:n - 1] + order[:h] + order[n - 1:]])
    for K in sorted({0, min(h, max(1, 12 - k))}):
        top = 1 << (h - K)
        chunks = sorted({0, 1 % top, top // 3, top - 1})
        got = emulate(img, kind, K, chunks)
        for q in chunks:
            compare(got[q], kind, scale, shift, ao, (q << K) << k, ((q + 1) << K) << k)


@pytest.mark.parametrize("values", ["01", "f64"])
def test_a_sub_range_keeps_the_plans_partial_sum(values):
    m = synth.band_plus(40, 2, 1, seed=4, values=values)
    a = 21
    plan = np.ascontiguousarray(m[:, list(A.inspect(m).col_order)[:40]])
    for q in (0, 5, (1 << 18) - 1):
        img, kind, k, _, scale, shift = A.elim_image(m, g_lo=q << a, g_hi=(q + 1) << a)
        assert img and k >= 2
        compare(emulate(img, kind, a - k, [q])[q], kind, scale, shift, plan, q << a, (q + 1) << a)
