"""Layout of the solve kernel's workspaces, from the header that the kernels and
the host share: whatever the sizes, the parts lie apart, and those read 16
bytes at a time (the staged y above all) start on 16-byte boundaries in both
vector precisions."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "ndsolve.cuh"
using namespace thm;
template <class V> int check(const NdSizes& z) {
    const NdGlob g = nd_glob_layout(z);
    int bad = g.u1 < z.nu[0] || g.y < g.u1 + z.nu[1] || g.stride < g.y + z.ny;
    for (int cta = 0; cta < 3; ++cta)
        for (int64_t at : {(int64_t)0, g.u1, g.y}) bad |= (cta * g.stride + at) * (int64_t)sizeof(V) % 16 != 0;
    for (int k = 0; k < 8; ++k) {
        const NdLayout L = nd_layout<V>(z, k & 1, (k >> 1) & 1, k >> 2);
        for (size_t at : {L.lev, L.slt, L.vec, L.ysc, L.u0, L.u1, L.part}) bad |= at % 16 != 0;
        bad |= L.ysc < L.vec + z.nvec * sizeof(V) || L.total > L.part + ND_NT * sizeof(V);
    }
    return bad;
}
int main() {
    int bad = 0;
    for (int a = 0; a < 6; ++a)
        for (int b = 0; b < 6; ++b)
            for (int y = 0; y < 6; ++y) {
                NdSizes z;
                z.nlev = 9; z.nslt = 1366; z.nvec = 13500 + a; z.ny = 7252 + y; z.nu[0] = 6117 + a; z.nu[1] = 9620 + b;
                bad += check<float2>(z) + check<double2>(z);
            }
    printf("bad %d\n", bad);
    return bad != 0;
}
"""


def test_parts_are_apart_and_aligned(tmp_path):
    from paper_2105_11993_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, *build._flags(), str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
