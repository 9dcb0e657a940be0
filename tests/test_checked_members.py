"""The checked build's count of a family's members on one delta row, with a
delta entry that is no vertex: the entry has to be reported and left out.  A
GPU never gets such a row, so the device function's own text is compiled for
the host here (one thread of one)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2401_11029_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

HEAD = r'''
#define CFLR_CHECKED
#include <cstdio>
#include <vector>
#include "kernels.cuh"
using namespace cflr;
template <class T> static T atomicAdd(T *p, T v) { T o = *p; *p += v; return o; }
static unsigned atomicOr(unsigned *p, unsigned v) { unsigned o = *p; *p |= v; return o; }
static int __ffsll(long long x) { return __builtin_ffsll(x); }
'''
MAIN = r'''
int main() {
    // 3 members on slots 0..2, 8 vertices, row k of member i holds k + 10 i tiles
    const uint32_t n = 8, F = 3;
    std::vector<uint4> desc((size_t)F * 2 * n, make_uint4(0, 0, 0, 0));
    std::vector<uint32_t> occ(2 * n, 0);
    for (uint32_t i = 0; i < F; i++)
        for (uint32_t k = 1; k < n; k++) {
            desc[(size_t)2 * i * n + k].y = k + 10 * i;
            occ[k] |= 1u << i;
        }
    std::vector<uint4 *> dp;
    for (uint32_t i = 0; i < F; i++) dp.push_back(&desc[(size_t)2 * i * n]);
    std::vector<uint32_t *> op(F, occ.data());
    uint32_t occ_w[3] = {1, 1, 1}, local[3] = {0, 1, 2};
    SlotTab S{};
    S.desc = dp.data();
    S.occ = op.data();
    S.occ_w = occ_w;
    S.local = local;
    int bad = 0;
    for (int planted = 0; planted < 2; planted++) {
        // five entries (d < n: vertex 5 is one); the fourth may be no vertex
        uint32_t pool[5] = {1, 2, 7, planted ? 0xFFFFFF00u : 4u, 3};
        unsigned long long mf[3] = {0, 0, 0};
        uint32_t mc[3] = {0, 0, 0};
        unsigned err = 0;
        family_members(S, 0, F, 0, n, pool, 0, 5, 0, 1, mf, mc, &err);
        for (uint32_t i = 0; i < F; i++) {
            const unsigned long long rows = planted ? 4 : 5;
            const unsigned long long want = 1 + 2 + 7 + 3 + (planted ? 0 : 4) + 10 * i * rows;
            if (mf[i] != want || mc[i] != rows) {
                std::printf("planted %d member %u: %llu tiles of %u rows, not %llu of %llu\n",
                            planted, i, mf[i], mc[i], want, rows);
                bad = 1;
            }
        }
        if (err != (planted ? OVF_BOUNDS : 0u)) std::printf("planted %d: flags %u\n", planted, err), bad = 1;
    }
    return bad;
}
'''


def test_an_entry_that_is_no_vertex_is_left_out(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    with open(os.path.join(CSRC, "kernels.cu")) as f:
        text = f.read()
    text = text[text.index("constexpr int FM_BATCH"):text.index("__device__ __forceinline__ Work warp_sum")]
    src, exe = str(tmp_path / "members.cpp"), str(tmp_path / "members")
    with open(src, "w") as f:
        f.write(HEAD + text.replace("__device__ __forceinline__", "static") + MAIN)
    subprocess.run([cxx, "-O1", "-std=c++17", "-w", "-I", CSRC, "-I", CUDA, src, "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
