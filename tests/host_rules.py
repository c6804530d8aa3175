"""Values of the library's host-side rules: C++ expressions over its internal
headers, compiled by nvcc (no GPU needed) and linked with the library."""
import os
import subprocess

from paper_1312_3004_gb300 import build

PROLOGUE = r"""
#include <cstdio>
#include <vector>
#include "rewl_internal.cuh"
#include "rewl_host_internal.hpp"
using namespace rewl;
// The device model of a run on a GPU with 152 SMs and 227 KB of shared memory per CTA
static const int kSms = 152;
static const size_t kShared = 232448;
static Model model(int q, int L, int h, int W, int m, int bits) {
    Model M{};
    M.q = q, M.L = L, M.N = L * L, M.W = W, M.B = W + 1, M.h = h, M.m = m, M.G = h * m;
    M.bits = bits, M.wpc = (M.N * bits + 31) / 32, M.K = 3000;
    return M;
}
int main() {
"""


def evaluate(tmp_path, expressions):
    """The expressions' values, as integers, in order."""
    src = PROLOGUE + "".join("    std::printf(\"%%lld\\n\", (long long)(%s));\n" % e for e in expressions) + "}\n"
    cu, exe = os.path.join(str(tmp_path), "rules.cu"), os.path.join(str(tmp_path), "rules")
    with open(cu, "w") as f:
        f.write(src)
    lib = build.build()
    subprocess.run([build._nvcc()] + build.ARCH + ["-std=c++17", "-cudart", "shared", "-I", build.CSRC, "-I",
                    os.path.join(build.ROOT, "include"), "-o", exe, cu, lib, "-Xlinker", "-rpath," + build.OUT_DIR,
                    "-Xlinker", "-rpath," + build._cuda_lib_dir()], check=True)
    return [int(x) for x in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]
