"""The build option PSATD_TW_HILO: FP32 table twiddles applied as hi + lo pairs.
A small program multiplies by twiddles whose hi parts are off by some 3e-7: with
the option every product, plain and conjugate, in the real split and the merge,
is that of the FP64 twiddle to FP32 rounding; without it the hi part's error
shows."""
import os
import subprocess

import pytest
import torch

from paper_1707_08500_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cmath>
#include <complex>
#include <cstdio>
#include <vector>
#include "psatd_kernels.cuh"
using namespace psatd;
using cd = std::complex<double>;
__global__ void k(const twd<float>* tw, const cpx<float>* a, const cpx<float>* b, cpx<float>* o, int n) {
    const int i = threadIdx.x;
    if (i >= n) return;
    const auto w = ld_tw(tw + i);
    o[i] = mul_tw(a[i], w);
    o[n + i] = mul_tw_conj(a[i], w);
    split_pair_v(a[i], b[i], w, o[2 * n + i], o[3 * n + i]);
    merge_pair_v(a[i], b[i], w, o[4 * n + i], o[5 * n + i]);
}
int main() {
    const int n = 96;
    std::vector<twd<float>> tw(n);
    std::vector<cpx<float>> a(n), b(n), o(6 * n);
    auto part = [](double v, float& hi, float& lo) { hi = float(v) * (1.f + 3e-7f); lo = float(v - double(hi)); };
    for (int i = 0; i < n; ++i) {
        const cd w = std::polar(1.0, -2 * M_PI * i / n);
        part(w.real(), tw[i].hi.x, tw[i].lo.x);
        part(w.imag(), tw[i].hi.y, tw[i].lo.y);
        a[i] = cpx<float>{std::sin(1.f + i), std::cos(2.f * i)};
        b[i] = cpx<float>{std::cos(3.f + i), std::sin(5.f * i)};
    }
    void *dt, *da, *db, *dd;
    cudaMalloc(&dt, n * sizeof(twd<float>));
    cudaMalloc(&da, n * sizeof(cpx<float>));
    cudaMalloc(&db, n * sizeof(cpx<float>));
    cudaMalloc(&dd, 6 * n * sizeof(cpx<float>));
    cudaMemcpy(dt, tw.data(), n * sizeof(twd<float>), cudaMemcpyHostToDevice);
    cudaMemcpy(da, a.data(), n * sizeof(cpx<float>), cudaMemcpyHostToDevice);
    cudaMemcpy(db, b.data(), n * sizeof(cpx<float>), cudaMemcpyHostToDevice);
    k<<<1, 128>>>((twd<float>*)dt, (cpx<float>*)da, (cpx<float>*)db, (cpx<float>*)dd, n);
    if (cudaMemcpy(o.data(), dd, 6 * n * sizeof(cpx<float>), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    double num = 0, den = 0;
    for (int i = 0; i < n; ++i) {
        const cd w = std::polar(1.0, -2 * M_PI * i / n), A(a[i].x, a[i].y), B(b[i].x, b[i].y), I(0, 1);
        // w stands for the halved real-split twiddle
        const cd e = 0.5 * (A + conj(B)), t = w * (A - conj(B)) / I, m = A + conj(B), p = 2.0 * conj(w) * (A - conj(B));
        const cd want[6] = {A * w, A * conj(w), e + t, conj(e - t), m + I * p, conj(m) + I * conj(p)};
        for (int f = 0; f < 6; ++f) {
            num += std::norm(cd(o[f * n + i].x, o[f * n + i].y) - want[f]);
            den += std::norm(want[f]);
        }
    }
    std::printf("%.3e\n", std::sqrt(num / den));
    return 0;
}
"""


@pytest.mark.parametrize("hilo", [0, 1])
def test_products_with_hi_and_lo(tmp_path, hilo):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", f"-DPSATD_TW_HILO={hilo}",
                    "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    err = float(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout)
    # a handful of FP32 roundings (2^-24 each) against the 3e-7 of the hi parts
    assert (err < 1e-7) if hilo else (2e-7 < err < 5e-7), err
