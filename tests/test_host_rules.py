"""Host rules of the library that need no GPU: headers without CUDA in them,
compiled here with the host compiler and compared with their plain statement.
"""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_04017_gb300", "csrc")


@pytest.fixture
def run_cpp(tmp_path):
    def run(source, *args):
        src, exe = tmp_path / "t.cpp", tmp_path / "t"
        src.write_text(source)
        subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
        out = subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True, text=True).stdout
        return [int(x) for x in out.split()]

    return run


def test_pieces_cover_a_batch(run_cpp):
    # around every multiple of a piece's unit in eighths, where the rounding
    # turns, and both ends of the range that is staged whole
    lo, hi = 1 << 20, 1 << 24
    sizes = sorted({n for k in range(2, 33) for d in range(-9, 10) if lo <= (n := (k << 19) + d) <= hi}
                   | {lo, hi, 7 * (3 << 16) + 1})
    pieces = run_cpp("""
#include <cstdio>
#include <cstdlib>
#include "cht_pieces.h"
int main(int n, char** v) {
    std::printf("%d\\n", cht::kPipePieces);
    for (int i = 1; i < n; ++i) std::printf("%llu\\n", (unsigned long long)cht::pipe_piece(std::strtoull(v[i], 0, 10)));
}
""", *sizes)
    most = pieces.pop(0)
    for n, p in zip(sizes, pieces):
        assert p % (1 << 16) == 0 and -(-n // p) <= most, (n, p)
        assert p - n / 8 < 1 << 16, (n, p)  # an eighth, rounded up


def test_read_only_loads_stay_in_ordinary_launches():
    # ld.global.nc needs data that nothing writes while the kernel lives.  A
    # kernel that begins with pdl_enter lives before the one ahead of it is
    # done, so neither it nor device functions (which any kernel may call) load
    # that way.
    header = re.compile(r"^(?:__global__|__device__|template)[^;{]*\{", re.M)
    users = 0
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        starts = [m.start() for m in header.finditer(text)]
        for b, e in zip(starts, starts[1:] + [len(text)]):
            body = text[b:e]
            if re.match(r"__device__ __forceinline__ void ld_\w+_nc\(", body):
                continue  # the load itself
            if re.search(r"\bld_\w+_nc\(|\.nc\.|__ldg\(", body):
                users += 1
                assert "__global__" in body.split("{")[0] and "pdl_enter" not in body, (f, body[:120])
    assert users > 0


def test_kept_numbers_are_a_device_s_own(run_cpp):
    # a kernel attribute set on one device is not set on another: what a launch
    # needs is asked (and done) on each device it comes to, once
    got = run_cpp("""
#include <cstdio>
#include <initializer_list>
#include "cht_per_device.h"
int main() {
    static cht::PerDevice kept;
    int fail = 7;
    for (int dev : {0, 1, 0, 1, 63, 63, 64, 64, 2, 2}) {
        int asked = 0, n = -1;
        const int e = kept.get(dev, &n, [&](int* out) {
            asked = 1;
            *out = dev + 10;
            if (dev == 2 && fail) { const int f = fail; fail = 0; return f; }
            return 0;
        });
        std::printf("%d %d %d\\n", e, n, asked);
    }
}
""")
    assert got == [0, 10, 1, 0, 11, 1, 0, 10, 0, 0, 11, 0, 0, 73, 1, 0, 73, 0, 0, 74, 1, 0, 74, 1, 7, 12, 1, 0, 12, 1]


def test_slots_spread_structured_keys(run_cpp):
    # looks of linear probing in 2048 slots for a window of 1024 distinct keys,
    # in hundredths: 150 for random slots (0.5 (1 + 1 / (1 - 0.5))), a few
    # hundredths more or less by chance
    got = run_cpp("""
#include <cstdio>
#include <vector>
#include "cht_hash.h"
typedef unsigned long long u64;
static int looks(const std::vector<u64>& keys) {
    static u64 slot[2048];
    for (u64& s : slot) s = 0;
    long n = 0;
    for (u64 k : keys) {
        unsigned s = cht::slot_hash(k, 2047);
        for (++n; slot[s]; ++n) s = (s + 1) & 2047;
        slot[s] = k;
    }
    return int(n * 100 / long(keys.size()));
}
int main() {
    std::vector<u64> k(1024);
    for (int sh = 0; sh < 54; ++sh)  // ids shifted left; strides of addresses and records
        for (u64 m : {1ull, 3ull, 7ull, 100ull, 4097ull}) {
            if (m > 1 && sh > 40) continue;
            for (u64 i = 0; i < 1024; ++i) k[i] = ((i + 1) * m) << sh;
            std::printf("%d\\n", looks(k));
        }
    for (int hi = 10; hi < 59; ++hi) {  // two ids of 32 values each in one word
        for (u64 i = 0; i < 1024; ++i) k[i] = (((i >> 5) + 1) << hi) | ((i & 31) + 1);
        std::printf("%d\\n", looks(k));
    }
    // keys of one home in 2^16, as a batch sorted by the hash brings them
    k.clear();
    for (u64 x = 1; k.size() < 1024; ++x)
        if (cht::fmix64(x) >> 52 == 77) k.push_back(x);
    std::printf("%d\\n", looks(k));
}
""")
    assert len(got) == 54 + 4 * 41 + 49 + 1 and max(got) < 200, max(got)


def test_grid_keeps_to_the_ctas_asked_for(run_cpp):
    # (operations in CTAs, CTAs per SM that fit, CTAs per SM asked for, modifies)
    sms = 152
    cases = [(need, fit, asked, mod) for need in (0, 1, 100, 151, 153, 608, 1216, 1520, 1521, 7295, 7296, 1 << 18, 1 << 27)
             for fit in (4, 8) for asked in (0, 1, 3, 4, 8, 20) for mod in (0, 1)]
    got = run_cpp("""
#include <cstdio>
#include <cstdlib>
#include "cht_grid.h"
int main(int n, char** v) {
    for (int i = 1; i + 3 < n; i += 4)
        std::printf("%llu\\n", (unsigned long long)cht::thread_grid(std::strtoull(v[i], 0, 10), 152, std::atoi(v[i + 1]),
                                                                   std::atoi(v[i + 2]), std::atoi(v[i + 3])));
}
""", *(x for c in cases for x in c))
    for (need, fit, asked, mod), grid in zip(cases, got, strict=True):
        assert 1 <= grid <= max(need, 1)
        if asked:
            assert grid == max(1, min(need, sms * min(asked, fit))), (need, fit, asked, mod, grid)
        elif need >= sms * fit:
            assert grid >= sms * fit  # never fewer than a wave


def test_arrays_that_share_memory(run_cpp):
    # every placement of two short arrays (and none)
    got = run_cpp("""
#include <cstdio>
#include "cht_pieces.h"
int main() {
    static char m[16];
    for (int a = 0; a < 6; ++a)
        for (int an = 1; an < 6; ++an)
            for (int b = 0; b < 6; ++b)
                for (int bn = 1; bn < 6; ++bn) {
                    bool both = false;
                    for (int x = 0; x < 16; ++x) both |= x >= a && x < a + an && x >= b && x < b + bn;
                    std::printf("%d\\n", cht::share_memory(m + a, an, m + b, bn) == both);
                }
    std::printf("%d\\n", !cht::share_memory(nullptr, 8, m, 8) && !cht::share_memory(m, 8, nullptr, 8));
}
""")
    assert len(got) == 901 and all(got)
