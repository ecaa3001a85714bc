"""The hub tables a graph keeps (csrc/hub_slots.h), compiled for the host: alternating keys,
runs without hub rows, and builds that fail half-way."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_14895_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "hub_slots.h"
using namespace fsgp;
static int builds = 0, live = 0;
static HubTable slots[2];
// fail_at: 1 before the table is allocated, 2 after
static int get(int min_deg, int chunk, int n_hubs, const HubTable **out, int fail_at = 0) {
    return hub_slot(slots, min_deg, chunk, n_hubs,
        [](HubTable &H) { if (H.d_chunk_base) { --live; std::free(H.d_chunk_base); } },
        [&](HubTable &H) {
            ++builds;
            if (fail_at == 1) return -5;
            H.d_chunk_base = (int64_t *)std::malloc(8); ++live;
            if (fail_at == 2) return -5;
            H.d_chunk_base[0] = min_deg * 100000 + chunk;
            H.n_chunks = 7;
            return 0;
        }, out);
}
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
static bool holds(const HubTable *t, int min_deg, int chunk, int n_hubs) {
    return t->d_chunk_base && t->d_chunk_base[0] == min_deg * 100000 + chunk && t->n_hubs == n_hubs && t->n_chunks == 7;
}
int main() {
    const HubTable *t = nullptr;
    // two keys alternate, with runs without hub rows in between: built once each
    for (int i = 0; i < 5; ++i) {
        CHECK(get(8192, 8192, 3, &t) == 0 && holds(t, 8192, 8192, 3));
        CHECK(get(65536, 8192, 0, &t) == 0 && !t->d_chunk_base && t->n_hubs == 0 && t->n_chunks == 0);
        CHECK(get(65536, 2048, 0, &t) == 0 && !t->d_chunk_base && t->n_hubs == 0);
        CHECK(get(8192, 2048, 3, &t) == 0 && holds(t, 8192, 2048, 3));
    }
    CHECK(builds == 2 && live == 2);
    // a third key takes the place of the one used longest ago
    CHECK(get(8192, 8192, 3, &t) == 0);
    CHECK(get(512, 100, 9, &t) == 0 && holds(t, 512, 100, 9) && builds == 3 && live == 2);
    CHECK(get(8192, 8192, 3, &t) == 0 && builds == 3);
    // a build that failed, before or after its allocation, leaves no table behind its key
    for (int at = 1; at <= 2; ++at) {
        CHECK(get(1024, 10 * at, 5, &t, at) == -5 && live == 1);
        CHECK(get(8192, 8192, 3, &t) == 0 && holds(t, 8192, 8192, 3));
        CHECK(get(1024, 10 * at, 5, &t) == 0 && holds(t, 1024, 10 * at, 5) && live == 2);
        CHECK(get(8192, 8192, 3, &t) == 0 && holds(t, 8192, 8192, 3));
    }
    return 0;
}
"""


def test_hub_tables(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "hub_slots_test.cpp"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
