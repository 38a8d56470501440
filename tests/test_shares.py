"""How a launch's units are shared out over its CTAs, gone through on the CPU: the structs are compiled for the host.  CPU only."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "fq_shares.h"
using namespace fq;
#define CHECK(c, ...) do { if (!(c)) { std::printf("%s: ", #c); std::printf(__VA_ARGS__); std::printf("\n"); std::exit(1); } } while (0)

static void divisors() {
    std::mt19937 rng(1);
    std::vector<uint32_t> ds;
    for (uint32_t d = 1; d <= 4096; ++d) ds.push_back(d);
    for (int b = 12; b < 32; ++b)
        for (int e = -1; e <= 1; ++e) ds.push_back((1u << b) + e);
    for (int i = 0; i < 20000; ++i) ds.push_back((rng() >> (rng() % 32)) | 1u);
    ds.push_back(~0u), ds.push_back(~0u - 1);
    for (uint32_t d : ds) {
        const Divisor by = Divisor::of(d);
        const auto at = [&](uint32_t n) { CHECK(by(n) == n / d, "%u / %u", n, d); };
        const uint32_t top = ~0u / d * d;                      // the largest multiple
        for (uint32_t n : {0u, 1u, d - 1, d, d + 1, top - 1, top, ~0u - 1, ~0u}) at(n);
        for (int i = 0; i < 200; ++i) {
            const uint32_t n = rng(), m = n / d * d;
            at(n), at(m), at(m - 1);
        }
    }
}

static void plan(uint32_t NT, uint32_t KT, uint32_t sms, uint32_t slack) {
    const Split sp = split_units(NT, KT, sms, slack);
    const Shares sh = shares_of(sp, NT, KT);
    const uint32_t even = (NT * KT + std::min(sms, kMaxCtas) - 1) / std::min(sms, kMaxCtas);
    std::vector<uint32_t> first(NT, ~0u), last(NT, 0);
    uint32_t at = 0, longest = 0;
    CHECK(sp.grid >= 1 && sp.grid <= std::min(sms, kMaxCtas), "%u x %u: %u CTAs", NT, KT, sp.grid);
    for (uint32_t c = 0; c < sp.grid; ++c) {
        uint32_t begin, end;
        sh.range(c, KT, begin, end);
        CHECK(begin == at && end > begin, "%u x %u: CTA %u has [%u, %u) behind %u", NT, KT, c, begin, end, at);
        at = end;
        longest = std::max(longest, end - begin);
        int slots[2] = {0, 0};
        for (uint32_t tn = begin / KT; tn <= (end - 1) / KT; ++tn) {
            first[tn] = std::min(first[tn], c), last[tn] = std::max(last[tn], c);
            const bool whole = begin <= tn * KT && end >= (tn + 1) * KT;
            if (!whole) {
                const uint32_t s = sh.slot_of(c, tn, KT);
                CHECK(s < 2 && ++slots[s] == 1, "%u x %u: CTA %u, tile %u, slot %u", NT, KT, c, tn, s);
            }
        }
        CHECK(!sp.split || begin / KT == (end - 1) / KT, "%u x %u: CTA %u has parts of two tiles", NT, KT, c);
    }
    CHECK(at == NT * KT, "%u x %u: %u units dealt out", NT, KT, at);
    CHECK(longest == sp.units_per_cta && longest <= even + (sp.split ? slack : 0u), "%u x %u: %u units", NT, KT, longest);
    for (uint32_t tn = 0; tn < NT; ++tn) {
        uint32_t a, b;
        sh.owners(tn, KT, a, b);
        CHECK(a == first[tn] && b == last[tn], "%u x %u: tile %u of CTAs %u to %u, said to be of %u to %u", NT, KT, tn, first[tn], last[tn], a, b);
        CHECK(b - a < 255, "%u x %u: contributors of tile %u", NT, KT, tn);       // (arrivals are counted in bytes)
    }
}

// Plans that tests of the kernels name, on 148 SMs: CTAs to a tile (0: ranges) and units to a CTA
static void named() {
    const auto is = [](const Split& sp, uint32_t split, uint32_t units, int line) {
        CHECK(sp.split == split && sp.units_per_cta == units, "line %d: %u, %u", line, sp.split, sp.units_per_cta);
    };
    for (uint32_t nr : {16u, 32u, 64u, 128u})
        for (uint32_t g : {64u, 128u}) {
            const bool wide = nr == 64 && g == 128;
            const auto tc = [&](uint32_t K, uint32_t N) { return split_tc(N / 128, K / 128, 148, nr, g); };
            is(tc(8192, 1024), 18, 4, __LINE__);
            is(tc(2944, 1152), 16, 2, __LINE__);
            is(tc(4096, 4096), 4, 8, __LINE__);
            is(tc(3072, 5120), 3, 8, __LINE__);
            is(tc(1536, 9472), 2, 6, __LINE__);
            is(tc(5120, 5120), wide ? 3 : 0, wide ? 14 : 11, __LINE__);
            is(tc(14336, 4096), wide ? 4 : 0, wide ? 28 : 25, __LINE__);
            is(tc(2944, 11136), 0, 14, __LINE__);
        }
    const auto st = [](uint32_t K, uint32_t N, uint32_t rows, bool outliers) {
        const uint32_t BN = N % 256 ? 128 : 256;
        return split_streaming(BN, N / BN, K / 128, 148, rows, outliers);
    };
    for (uint32_t rows : {1u, 8u, 16u}) is(st(2048, 12800, rows, true), 2, 8, __LINE__);
    is(st(2304, 7296, 5, true), 2, 9, __LINE__);
    is(st(1664, 14336, 4, true), 2, 7, __LINE__);
    is(st(1664, 14336, 8, true), 0, 5, __LINE__);
    is(st(1664, 14336, 16, false), 2, 7, __LINE__);
    is(st(8192, 6400, 4, true), 5, 13, __LINE__);
    is(st(8192, 6400, 5, true), 0, 11, __LINE__);
    is(st(3840, 15360, 1, true), 2, 15, __LINE__);
    is(st(3840, 15360, 5, true), 0, 13, __LINE__);
    is(st(5120, 16384, 1, true), 0, 18, __LINE__);
    is(st(5120, 16384, 1, false), 2, 20, __LINE__);
    is(st(5120, 16384, 5, false), 0, 18, __LINE__);
    is(st(6272, 8832, 1, false), 2, 25, __LINE__);
    is(st(6272, 8832, 8, false), 0, 23, __LINE__);
    is(st(6528, 5504, 1, true), 3, 17, __LINE__);
    is(st(6528, 5504, 2, true), 0, 15, __LINE__);
}

int main() {
    divisors();
    named();
    for (uint32_t sms : {148u, 132u, 1u, 7u, 192u, 300u})
        for (uint32_t KT = 1; KT <= 224; KT += sms == 148 ? 1 : 13)
            for (uint32_t NT = 1; NT <= 448; NT += sms == 148 ? 1 : 11)
                for (uint32_t slack : {0u, 1u, 2u, 4u}) plan(NT, KT, sms, slack);
    for (uint32_t NT : {1023u, 1024u, 2048u})
        for (uint32_t KT : {1u, 2u, 73u, 1024u}) plan(NT, KT, 148, 1);
    std::printf("ok\n");
}
"""


@pytest.mark.skipif(subprocess.run(["which", "g++"], capture_output=True).returncode != 0, reason="no C++ compiler")
def test_ranges_owners_slots_and_division(tmp_path):
    """Every unit belongs to one CTA; the owners of a tile are those that have units of it; no CTA uses a slot twice; the
    divisions by multiplication are exact."""
    src, exe = tmp_path / "shares.cpp", tmp_path / "shares"
    src.write_text(_PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2608_15531_b200", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-o", str(exe), str(src)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True)
    assert p.returncode == 0 and p.stdout == "ok\n", p.stdout
