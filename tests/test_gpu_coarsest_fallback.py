"""The coarsest inverse on every cluster size down to one CTA, staged and not: where a device holds no cluster of 16 CTAs
(a part of a shared one) set-up takes a smaller one instead of failing.  The kernel and its rule are compiled from
their source, since an undivided GPU always takes 16."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_16863_gb300", "csrc")

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "mg.cuh"
namespace aao {
std::atomic<long long> g_launches{0};
thread_local long long g_thread_launches = 0;
bool g_prof_on = false;
thread_local double g_bytes_hint = 0.0;
int prof_begin_launch(const void*, cudaStream_t, double) { return -1; }
void prof_end_launch(int, cudaStream_t) {}
void set_error(const std::string& m) { std::fprintf(stderr, "%s\n", m.c_str()); }
}
using namespace aao;
int main() {
    cudaFuncSetAttribute(k_gauss_jordan, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    cudaFuncSetAttribute(k_gauss_jordan, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int n : {1, 2, 7, 16, 17, 31, 100, 256, 512}) {
        const int nm = 3;
        const size_t nn = (size_t)n * n;
        std::vector<double> A(nm * nn), I(nm * nn);
        for (int m = 0; m < nm; ++m)          // symmetric, strictly diagonally dominant with a margin of 1
            for (int i = 0; i < n; ++i)
                for (int j = 0; j < n; ++j)
                    A[m * nn + (size_t)i * n + j] = i == j ? 1.0 + n : std::cos(1.0 + m + i * j + i + j);
        double *a, *v;
        int* fail;
        if (cudaMalloc(&a, nm * nn * 8) || cudaMalloc(&v, nm * nn * 8) || cudaMalloc(&fail, 4)) return 2;
        cudaMemcpy(a, A.data(), nm * nn * 8, cudaMemcpyHostToDevice);
        for (int e = 4; e >= -1; --e) {
            const int ctas = e < 0 ? 1 : 1 << e;
            const bool staged = e >= 0;
            if (gj_smem(n, ctas, staged) > 227 * 1024) continue;
            cudaMemset(v, 0xFF, nm * nn * 8);
            cudaMemset(fail, 0, 4);
            launch_cluster(k_gauss_jordan, dim3(ctas * nm), dim3(kGjThreads), gj_smem(n, ctas, staged), (cudaStream_t)0, ctas,
                           (const double*)a, v, n, ctas, staged ? 1 : 0, fail);
            int f = -1;
            if (cudaMemcpy(&f, fail, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
            cudaMemcpy(I.data(), v, nm * nn * 8, cudaMemcpyDeviceToHost);
            double worst = 0.0;
            for (int m = 0; m < nm; ++m)
                for (int i = 0; i < n; ++i)
                    for (int j = 0; j < n; ++j) {
                        double s = i == j ? -1.0 : 0.0;
                        for (int k = 0; k < n; ++k) s += A[m * nn + (size_t)i * n + k] * I[m * nn + (size_t)k * n + j];
                        if (!(std::fabs(s) <= worst)) worst = std::fabs(s);
                    }
            std::printf("%d %d %d %d %.3e\n", n, ctas, (int)staged, f, worst);
        }
        cudaFree(a);
        cudaFree(v);
        cudaFree(fail);
    }
    return 0;
}
"""


def test_rule_takes_the_largest_cluster_that_fits(tmp_path):
    mg = open(os.path.join(CSRC, "mg.cuh")).read()
    rule = mg[mg.index("template <class Fits> inline int gj_ctas"):]
    rule = rule[:rule.index("\n}\n") + 3]
    most = re.search(r"constexpr int kGjCtas = \d+;", mg).group(0)
    (tmp_path / "t.cpp").write_text("#include <cstdio>\n" + most + "\n" + rule +
                                    'int main() { for (int m = 0; m <= 16; ++m) std::printf("%d ", '
                                    "gj_ctas([&](int c) { return c <= m; })); }\n")
    subprocess.run(["g++", "-std=c++17", "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out] == [0, 1, 2, 2, 4, 4, 4, 4] + [8] * 8 + [16]


@pytest.mark.gpu
def test_inverse_on_every_cluster_size(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    (tmp_path / "t.cu").write_text(MAIN)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                    CSRC, "-I", os.path.join(ROOT, "include"), "-o", str(tmp_path / "t"), str(tmp_path / "t.cu")], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout
    seen = set()
    for line in out.splitlines():
        n, ctas, staged, fail, worst = line.split()
        seen.add((int(n), int(ctas), int(staged)))
        # |A X - I| <= c n u |A| |X|: rows of |A| sum to at most 2 n, |X| to at most 1, c = 4
        assert int(fail) == 0 and float(worst) <= 4 * int(n) * 2.0 ** -53 * 2 * max(int(n), 2), line
    assert {(512, 16, 1), (512, 1, 0), (256, 16, 1), (256, 8, 1), (256, 4, 1), (256, 1, 0), (1, 16, 1), (17, 2, 1)} <= seen
