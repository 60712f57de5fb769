"""Runs one of the library's device functions on arrays: a kernel of a few lines around it is compiled with the
library's own flags and headers, and run by itself (arrays go in and out as files)."""
import os
import subprocess

import numpy as np

from paper_2403_15051_gb300 import build as fbuild

_MAIN = r"""
#include <cstdio>
#include <vector>
#include "device_common.cuh"
#include "kernels_decl.h"
#include "closure_item.cuh"
using namespace fdlb;
using real = %(real)s;
// in: [n_in][n], out: [n_out][n]
__global__ void unit_kernel(const double* in, double* out, int n) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    double x[%(n_in)d], y[%(n_out)d];
    for (int k = 0; k < %(n_in)d; ++k) x[k] = in[(size_t)k * n + t];
    for (int k = 0; k < %(n_out)d; ++k) y[k] = 0.0;
    %(body)s
    for (int k = 0; k < %(n_out)d; ++k) out[(size_t)k * n + t] = y[k];
}
int main(int argc, char** argv) {
    const int n = atoi(argv[1]);
    std::vector<double> h((size_t)n * %(n_in)d), g((size_t)n * %(n_out)d);
    FILE* f = fopen(argv[2], "rb");
    if (!f || fread(h.data(), 8, h.size(), f) != h.size()) return 2;
    fclose(f);
    double *a, *b;
    if (cudaMalloc(&a, h.size() * 8) || cudaMalloc(&b, g.size() * 8)) return 3;
    cudaMemcpy(a, h.data(), h.size() * 8, cudaMemcpyHostToDevice);
    unit_kernel<<<(n + 127) / 128, 128>>>(a, b, n);
    if (cudaMemcpy(g.data(), b, g.size() * 8, cudaMemcpyDeviceToHost)) return 4;
    f = fopen(argv[3], "wb");
    if (!f || fwrite(g.data(), 8, g.size(), f) != g.size()) return 5;
    fclose(f);
    return 0;
}
"""


def run(tmp_path, real, body, x, n_out):
    """y[n_out][n] for x[n_in][n]: `body` maps double x[] to double y[] for one column, `real` the functions' type."""
    x = np.ascontiguousarray(x, dtype=np.float64)
    src, exe, fi, fo = (os.path.join(str(tmp_path), k) for k in ("unit.cu", "unit", "in.bin", "out.bin"))
    with open(src, "w") as f:
        f.write("#include <cstdlib>\n" + _MAIN % dict(real=real, n_in=x.shape[0], n_out=n_out, body=body))
    subprocess.run([fbuild._nvcc(), *fbuild.ARCH, "-O3", "-std=c++17", "-diag-suppress", "549,1886,177", "-I", fbuild.CSRC, src,
                    "-o", exe], check=True)
    x.tofile(fi)
    subprocess.run([exe, str(x.shape[1]), fi, fo], check=True)
    return np.fromfile(fo).reshape(n_out, x.shape[1])
