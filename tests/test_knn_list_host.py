"""The ranked list of the kNN selection (csrc/sj_knn_list.cuh) run on the host,
lane by lane: for list sizes around the multiples of a warp and k on both sides
of the list's 256 entries, every output slot below min(m, k) is written by
exactly one lane, with the entry of that rank, and no other slot by any lane
(a second writer would race with the padding that follows a short list)."""
import os
import shutil
import subprocess

import pytest

from paper_2209_11287_gb300 import build

HARNESS = r"""
#include <cstdio>
#include <cstring>
#include <vector>
#include <algorithm>
#include "sj_knn_list.cuh"
using namespace sj;

template <int E>
int check(int m, int k) {
    std::vector<int4> list(32 * E);
    for (int j = 0; j < m; ++j) {  // distances in a scrambled order, some equal
        const double d = 0.25 * ((j * 37) % 61);
        long long b;
        memcpy(&b, &d, 8);
        list[j] = make_int4((int)b, (int)(b >> 32), (j * 91) % 257, 0);
    }
    auto less = [](const int4& a, const int4& b) {
        return a.y != b.y ? a.y < b.y : a.x != b.x ? (unsigned)a.x < (unsigned)b.x : a.z < b.z;
    };
    std::vector<int4> want(list.begin(), list.begin() + m);
    std::sort(want.begin(), want.end(), less);
    std::vector<int> writers(k, 0);
    int bad = 0;
    for (int lane = 0; lane < 32; ++lane) {
        std::vector<int32_t> idx(k, -7);
        std::vector<double> dist(k, -7.0);
        knn_write<E>(list.data(), m, k, 0, lane, idx.data(), dist.data());
        for (int r = 0; r < k; ++r)
            if (idx[r] != -7 || dist[r] != -7.0) {
                ++writers[r];
                if (r < m && (idx[r] != want[r].z || memcmp(&dist[r], &want[r].x, 8))) ++bad;
            }
    }
    for (int r = 0; r < k; ++r)
        if (writers[r] != (r < std::min(m, k) ? 1 : 0)) ++bad;
    if (bad) printf("list of %d entries (%d a lane), k = %d: %d bad slots\n", m, E, k, bad);
    return bad;
}

int main() {
    int bad = 0;
    for (int k : {1, 24, 192, 255, 256, 257, 300, 1024}) {
        for (int m : {1, 31, 32}) bad += check<1>(m, k);
        for (int m : {33, 63, 64}) bad += check<2>(m, k);
        for (int m : {65, 127, 128}) bad += check<4>(m, k);
        for (int m : {129, 200, 255, 256}) bad += check<8>(m, k);
    }
    return bad ? 1 : 0;
}
"""


def test_every_slot_has_one_writer(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "knn_list.cu"
    src.write_text(HARNESS)
    exe = str(tmp_path / "knn_list")
    subprocess.run([nvcc, "-std=c++17", "-O1", *build.ARCH, "-I", build.CSRC, "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
