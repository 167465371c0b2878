"""Host rules for a list's device memory (csrc/memory.h), compiled and run without a GPU.

* a request for several blocks leaves none of them behind when one cannot be had, whichever it is, and
  can be made again;
* edge records leave a quarter of the free memory, and what the list's later calls take, to everything else; the
  free memory is asked for again once a 64th of it has been taken.
"""

from __future__ import annotations

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_06711_gb300", "csrc")

SOURCE = r"""
#include "memory.h"
#include <cstdio>
#include <cstdlib>
#include <set>
using namespace reann;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    for (int fail = 0; fail <= 6; ++fail)  // the fail-th block cannot be had (0: each can)
        for (int room = 0; room <= 2; ++room) {  // how often room can be made
            std::set<void*> held;
            int asked = 0, made = 0;
            double* a = (double*)1;
            float* b = (float*)1;
            int* c = (int*)1;
            auto take = [&](size_t n) -> void* {
                if (++asked == fail || (fail == 6 && n == 24)) return nullptr;
                return *held.insert(std::malloc(n)).first;
            };
            auto give = [&](void* p) {
                if (!held.erase(p)) std::abort();
                std::free(p);
            };
            const bool ok = take_all({{&a, 8}, {&b, 16}, {&c, 24}}, take, give, [&] { return made++ < room; });
            CHECK(ok == (fail == 0 || (fail >= 4 && fail != 6) || (fail != 6 && room > 0)));
            CHECK(held.size() == (ok ? 3u : 0u));
            CHECK(ok ? held.count(a) && held.count(b) && held.count(c) : !a && !b && !c);
            for (void* p : held) std::free(p);
        }
    for (int64_t rows : {1, 1000, 1024, 1025, 50000, 1048576})
        for (uint64_t row : {32ull, 4352ull})
            for (uint64_t later : {0ull, 100000000ull})
                for (double share : {0.0, 0.3, 0.9, 1.0, 1.3, 1.34, 2.0, 3.0, 100.0}) {
                    const uint64_t fr = (uint64_t)(share * (rows * row + later)), got_max = fr / 4 * 3;
                    const int64_t got = edge_rows_within(rows, row, later, fr);
                    CHECK(got >= 1 && got <= rows && (rows > kMinEdgeRows || got == rows));
                    CHECK(got * row + later <= got_max || got == std::min(rows, kMinEdgeRows));
                    if (got < rows) CHECK(std::min<int64_t>(rows, 2 * got) * row + later + row > got_max);
                }
    FreeMemory m;
    CHECK(m.ask(1));  // nothing known yet
    m.told(6400);
    CHECK(!m.ask(60) && m.ask(40));  // a 64th of 6,400 taken since
    m.told(64);
    CHECK(m.ask(1));
    m.told(0);
    CHECK(m.ask(0));
    std::puts("ok");
    return 0;
}
"""


def test_blocks_and_records(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0 and run.stdout.strip() == "ok", run.stdout


def test_later_blocks_are_taken_all_or_none():
    # the calls that take memory after the build go through it: a partial set must not be taken for a whole one
    text = open(os.path.join(CSRC, "reann_api.cu")).read()
    for block in ("vir_partial", "d_energy", "md_out"):
        assert f"nl->{block} = nl_alloc" not in text and f"&nl->{block}," in text, block
