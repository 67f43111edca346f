"""Shared memory of the trace kernels against the resident warps they are
compiled for, by the same constants (csrc/traverse.cuh)."""
import re
import subprocess

import pytest

from paper_2001_02620_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include "traverse.cuh"
using namespace qrt;
template <class Kind> void line(const char* name, int occ) {
    std::printf("%s %d %d %d\n", name, occ, Kind::STACK, Kind::kLaneBytes);
}
template <int OCC> void all() {
    line<QueryKind<true, 32, OCC>>("query any", OCC);
    line<QueryKind<false, 32, OCC>>("query closest", OCC);
    line<WaveKind<true, false, 32, OCC>>("wave any", OCC);
    line<WaveKind<false, false, 32, OCC>>("wave closest", OCC);
    line<WaveKind<false, true, 32, OCC>>("wave textured", OCC);
}
int main() { all<16>(); all<24>(); all<28>(); all<32>(); all<40>(); all<48>(); }
"""


@pytest.fixture(scope="module")
def kinds(tmp_path_factory):
    d = tmp_path_factory.mktemp("kinds")
    (d / "t.cu").write_text(SOURCE)
    subprocess.run([B.NVCC, *B.ARCH, "-std=c++17", "-I", B.CSRC, str(d / "t.cu"), "-o", str(d / "t")], check=True)
    out = subprocess.run([str(d / "t")], stdout=subprocess.PIPE, text=True, check=True).stdout
    return [(m[1], int(m[2]), int(m[3]), int(m[4])) for m in re.finditer(r"(\D+) (\d+) (\d+) (\d+)\n", out)]


def test_resident_warps_have_their_shared_memory(kinds):
    assert len(kinds) == 30
    for name, occ, entries, lane in kinds:
        uv = name.strip() in ("query closest", "wave textured")
        warps = 40 if occ == 48 and uv else occ
        threads = 128 if occ == 28 else 256
        blocks = warps * 32 // threads
        # 228 KB an SM, 1 KB reserved for each block, 16 bytes of claimed items a warp
        assert blocks * (threads * lane + threads // 32 * 16 + 1024) <= 228 * 1024, (name, occ)
        assert entries >= 4
