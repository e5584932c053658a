"""The host side of the N-D contexts without a device: a small program linked against the library drives the planner."""
import os
import shutil
import subprocess

import pytest

from paper_2411_19870_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = "/usr/local/cuda/include"

PRELUDE = """
#include <chrono>
#include <cstdio>
#include "demo_internal.h"
static DemoNdEntry entry(const int (&s)[4], const long long (&n)[4], int k)
{
    DemoNdEntry e{};
    long long stride = 1, chunks = 1;
    e.M = 1;
    for (int a = 3; a >= 0; --a) {
        e.s[a] = s[a];
        e.c[a] = (int)(n[a] / s[a]);
        e.stride[a] = stride;
        stride *= n[a];
        chunks *= e.c[a];
        e.M *= s[a];
        e.inv[a] = s[a] > 1 ? (unsigned)(((1ULL << 32) + s[a] - 1) / s[a]) : 0u;
    }
    e.k_eff = k < e.M ? k : e.M;
    e.chunk_end = chunks;
    return e;
}
"""


def run(tmp_path, main):
    lib = build.build_library()
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INCLUDE):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "plan.cc", tmp_path / "plan"
    src.write_text(PRELUDE + "int main()\n{\n" + main + "\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CUDA_INCLUDE, "-I", os.path.join(os.path.dirname(lib), "csrc"), str(src), lib,
                    "-Wl,-rpath," + os.path.dirname(lib), "-o", str(exe)], check=True, capture_output=True, text=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split()


def test_tensors_of_one_chunk_shape_are_planned_once(tmp_path):
    """The layout search of a chunk shape runs once per context, and a later tensor of the shape gets the same layout."""
    out = run(tmp_path, """
    using clock = std::chrono::steady_clock;
    const int s[4] = {16, 12, 5, 7};
    const long long n[4] = {64, 24, 10, 14}, n2[4] = {16, 12, 50, 70};
    double first = 1e9, later = 1e9;
    bool same = true;
    for (int r = 0; r < 5; ++r) {
        DemoNdTables tables;
        DemoNdEntry a = entry(s, n, 32), b;
        auto t0 = clock::now();
        demo_nd_plan(&a, &tables);
        auto t1 = clock::now();
        for (int i = 0; i < 100; ++i) {
            b = entry(s, i % 2 ? n : n2, 32);
            demo_nd_plan(&b, &tables);
            for (int d = 0; d < 4; ++d) same = same && a.p[d] == b.p[d];
            same = same && a.tile == b.tile && a.tail == b.tail && a.threads == b.threads;
        }
        auto t2 = clock::now();
        const double x = std::chrono::duration<double>(t1 - t0).count(), y = std::chrono::duration<double>(t2 - t1).count();
        if (x < first) first = x;
        if (y < later) later = y;
    }
    std::printf("%d %g %g", (int)same, first, later);
    """)
    assert out[0] == "1"
    assert float(out[2]) < 20 * float(out[1])  # a hundred further tensors


def test_a_layout_does_not_depend_on_the_order_of_the_tensors(tmp_path):
    """Chunks of one shape whose rows are whole 16-byte pieces of one tensor and not of the other: planned alone, first and second, every tensor
    gets the same tile and the same rows."""
    out = run(tmp_path, """
    const int s[][4] = {{1, 1, 32, 6}, {1, 1, 16, 12}, {1, 4, 6, 10}, {1, 8, 12, 5}};
    const long long n[][4][4] = {{{1, 1, 4096, 6}, {1, 1, 64, 18}, {1, 1, 32, 6}, {1, 1, 64, 12}},
                                 {{1, 1, 64, 24}, {1, 1, 64, 12}, {1, 1, 16, 36}, {1, 1, 32, 12}},
                                 {{1, 8, 12, 20}, {1, 8, 6, 10}, {1, 4, 6, 30}, {1, 16, 18, 10}},
                                 {{1, 64, 12, 5}, {1, 8, 24, 5}, {1, 16, 12, 10}, {1, 8, 12, 5}}};
    auto same = [](const DemoNdEntry &a, const DemoNdEntry &b) {
        for (int d = 0; d < 4; ++d)
            if (a.p[d] != b.p[d]) return false;
        return a.tile == b.tile && a.row == b.row && a.quads == b.quads && a.row_table == b.row_table && a.threads == b.threads;
    };
    int differ = 0, kinds = 0;
    for (int k = 0; k < 4; ++k)
        for (int i = 0; i < 4; ++i) {
            DemoNdTables own;
            DemoNdEntry alone = entry(s[k], n[k][i], 32);
            demo_nd_plan(&alone, &own);
            kinds |= 1 << alone.quads;
            for (int j = 0; j < 4; ++j) {
                DemoNdTables tables;
                DemoNdEntry first = entry(s[k], n[k][j], 32), second = entry(s[k], n[k][i], 32);
                demo_nd_plan(&first, &tables);
                demo_nd_plan(&second, &tables);
                differ += !same(alone, second);
            }
        }
    std::printf("%d %d", differ, kinds);
    """)
    assert out == ["0", "5"]


def test_classes_stay_below_the_range_of_the_chunk_counters(tmp_path):
    """Three tensors of 2^31 - 1 chunks and a small one, all of one kind: no class of 2^31 chunks or more, every tensor in one class, its
    chunks consecutive."""
    out = run(tmp_path, """
    const int s[4] = {1, 1, 1, 2};
    const long long n[4] = {1, 1, 1, 2 * ((1LL << 31) - 1)}, few[4] = {1, 1, 1, 2000};
    DemoNdTables tables;
    std::vector<DemoNdEntry> entries;
    for (int t = 0; t < 4; ++t) {
        entries.push_back(entry(s, t == 2 ? few : n, 1));
        entries.back().tensor = t;
        demo_nd_plan(&entries.back(), &tables);
    }
    std::vector<DemoNdClass> classes;
    demo_nd_classify(entries, 148, &classes);
    bool in_order = true;
    int next = 0;
    for (const DemoNdClass &k : classes) {
        long long at = 0;
        in_order = in_order && k.first == next;
        for (int i = 0; i < k.n; ++i) {
            const DemoNdEntry &e = entries[k.first + i];
            in_order = in_order && e.chunk_begin == at && e.layout <= k.first + i;
            at = e.chunk_end;
        }
        in_order = in_order && at == k.n_chunks;
        next += k.n;
        std::printf("%lld ", k.n_chunks);
    }
    std::printf("%d %d", next, (int)in_order);
    """)
    chunks, (tensors, in_order) = [int(v) for v in out[:-2]], out[-2:]
    assert max(chunks) <= 2 ** 31 - 1 and sum(chunks) == 3 * (2 ** 31 - 1) + 1000
    assert tensors == "4" and in_order == "1"
