"""The plane codes of a node (csrc/node_quant.h) are the same from device and host
code, where compilers differ in fusing products and sums."""
import subprocess

import pytest

torch = pytest.importorskip("torch")

from paper_2001_02620_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "node_quant.h"
using namespace qrt;

struct Axis {
    float lo[4], hi[4], s, o;
    uint8_t ql[4], qh[4], ok, pad[7];
};

__host__ __device__ void codes(Axis& a) { a.ok = quantize_axis(a.lo, a.hi, 4, &a.s, &a.o, a.ql, a.qh); }

__global__ void on_device(Axis* a, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) codes(a[k]);
}

int main() {
    const int n = 200000;
    std::mt19937 g(7);
    std::vector<Axis> a(n), d(n);
    for (int k = 0; k < n; ++k) {
        Axis& x = a[k];
        x = Axis{};
        // a step of few bits that is no power of two, and children on its codes:
        // every plane is exact, and (plane - o) / s a code's value but for the
        // rounding of 1 / s; every fourth axis is any other
        const float s = (float)(2 * (g() % 128) + 1) / 16.f, o = (float)(int)(g() % 64) - 32.f;
        for (int i = 0; i < 4; ++i) {
            const int p = i ? g() % 256 : 0, q = i ? g() % 256 : 255;
            x.lo[i] = dequant(p < q ? p : q, s, o);
            x.hi[i] = dequant(p < q ? q : p, s, o);
            if (k % 4 == 0) x.hi[i] += (float)(g() % 4096) / 4099.f;
        }
    }
    Axis* p = nullptr;
    if (cudaMalloc(&p, n * sizeof(Axis)) != cudaSuccess) return 1;
    if (cudaMemcpy(p, a.data(), n * sizeof(Axis), cudaMemcpyHostToDevice) != cudaSuccess) return 1;
    on_device<<<(n + 255) / 256, 256>>>(p, n);
    if (cudaMemcpy(d.data(), p, n * sizeof(Axis), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    int differ = 0;
    for (int k = 0; k < n; ++k) {
        codes(a[k]);
        bool same = a[k].ok == d[k].ok && a[k].s == d[k].s && a[k].o == d[k].o;
        for (int i = 0; i < 4; ++i) same = same && a[k].ql[i] == d[k].ql[i] && a[k].qh[i] == d[k].qh[i];
        differ += !same;
    }
    std::printf("%d\n", differ);
    return 0;
}
"""


def test_codes_of_device_and_host(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    (tmp_path / "t.cu").write_text(SOURCE)
    exe = str(tmp_path / "t")
    subprocess.run([B.NVCC, *B.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", B.CSRC,
                    str(tmp_path / "t.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], stdout=subprocess.PIPE, text=True, check=True)
    assert int(r.stdout) == 0
