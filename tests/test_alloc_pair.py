"""Buffers that are used together are allocated both or neither (csrc/alloc_pair.h), compiled for the host with an
allocator that fails when told to (CPU only).  The potential's copies rely on it: a call that found one of a pair
would launch a kernel with the other one null."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1708_03621_gb300", "csrc")

SOURCE = r"""
#include "alloc_pair.h"
#include <cstdio>
#include <cstdlib>
#include <set>
int main() {
    for (int fail = 0; fail < 3; ++fail) {       // the call that fails: none, the first, the second
        std::set<void*> live;
        int calls = 0;
        bool broken = fail > 0;
        auto alloc = [&](void** p, size_t n) {
            if (broken && ++calls == fail) return false;
            live.insert(*p = std::malloc(n));
            return true;
        };
        auto release = [&](void* p) { live.erase(p); std::free(p); };
        void *a = nullptr, *b = nullptr;
        const bool ok = jdft::alloc_pair(&a, 64, &b, 32, alloc, release);
        if (ok != (fail == 0) || (a != nullptr) != ok || (b != nullptr) != ok || live.size() != (ok ? 2u : 0u)) return 1;
        broken = false;                           // the next call finds room
        if (!jdft::alloc_pair(&a, 64, &b, 32, alloc, release) || !a || !b || live.size() != 2) return 2;
        void *a0 = a, *b0 = b;
        if (!jdft::alloc_pair(&a, 64, &b, 32, alloc, release) || a != a0 || b != b0 || live.size() != 2) return 3;
    }
    return 0;
}
"""


def test_both_or_neither(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_potential_copies_are_allocated_in_pairs():
    src = open(os.path.join(CSRC, "basis.cu")).read()
    body = src[src.index("jdft_status jdft_set_potential("):]
    body = body[:body.index("\n}\n")]
    assert not re.search(r"cudaMalloc\(\s*&b->V", body)
    for a, b in (("V", "V32"), ("Vn", "Vn32")):
        assert re.search(rf"alloc_pair\(\(void\*\*\)&b->{a}, n64, \(void\*\*\)&b->{b}, n32", body)
