"""The decode-cache append inside the selection's launch: the numbering of its
16-byte copies, compiled for the host and compared with Python's integers."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_31598_gb300", "csrc")

PROGRAM = r"""
#include "append_plan.h"
#include <cstdio>
#include <cstdlib>
using namespace statekv;
template <class I> void put(long long i, int T, int Hkv, int D)
{
    const AppendAt a = append_at(static_cast<I>(i), static_cast<I>(append_copies(T, Hkv, D)), Hkv, D / 8);
    std::printf("%d %d %d\n", a.t, a.hkv, a.ch);
}
int main(int n, char** v)
{
    const int T = std::atoi(v[1]), Hkv = std::atoi(v[2]), D = std::atoi(v[3]);
    const bool narrow = append_narrow(T, Hkv, D);
    std::printf("%lld %d", append_copies(T, Hkv, D), narrow ? 1 : 0);
    for (int split = 1; split <= 8; split *= 2) std::printf(" %d", append_ctas(T, Hkv, D, split));
    std::printf("\n");
    for (int j = 4; j < n; ++j) {
        if (narrow) put<int>(std::atoll(v[j]), T, Hkv, D);
        else put<long long>(std::atoll(v[j]), T, Hkv, D);
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("append")
    src, exe = d / "append.cpp", d / "append"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("T,hkv,d", [
    (1, 1, 64), (196, 4, 128), (399, 28, 128),
    (4096, 8192, 128),    # 2^30 copies: the last shape with 32-bit indexes
    (4096, 8193, 128),
    (4096, 16384, 128),   # 2^31 copies of K and V
    (2048, 32768, 128), (4096, 65535, 64), (4096, 65535, 128),
])
def test_every_copy_has_its_place(program, T, hkv, d):
    ch = d // 8
    per = T * hkv * ch
    rng = random.Random(0)
    at = {0, per - 1, per, 2 * per - 1} | {rng.randrange(2 * per) for _ in range(40)}
    at |= {x for x in (2 ** 31 - 1, 2 ** 31, 2 ** 32) if x < 2 * per}
    at = sorted(at)
    out = subprocess.run([program, str(T), str(hkv), str(d)] + [str(x) for x in at], check=True,
                         capture_output=True, text=True).stdout.split("\n")
    copies, narrow, *ctas = map(int, out[0].split())
    assert copies == per
    # the kernel's loop goes past the last copy by at most 8 CTAs' batches of 8 x 640
    assert not narrow or 2 * per + 9 * 8 * 640 < 2 ** 31
    for i, line in zip(at, out[1:]):
        r = i % per
        assert tuple(map(int, line.split())) == (r // (hkv * ch), r // ch % hkv, r % ch), i


@pytest.mark.parametrize("T,hkv,d", [(16, 1, 64), (196, 4, 128), (399, 28, 128), (401, 1, 64), (4096, 65535, 128)])
def test_append_ctas_cover_the_copies_in_whole_clusters(program, T, hkv, d):
    """As many CTAs as batches of copies, eight at most; a cluster size rounds that up
    and never takes CTAs away."""
    out = subprocess.run([program, str(T), str(hkv), str(d)], check=True, capture_output=True, text=True).stdout
    want = min(8, -(-2 * T * hkv * (d // 8) // (8 * 640)))
    for split, n in zip((1, 2, 4, 8), map(int, out.split()[2:])):
        assert n % split == 0 and want <= n < want + split, (split, n)
