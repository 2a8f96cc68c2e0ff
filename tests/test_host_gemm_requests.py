"""What the tensor-core GEMM takes and refuses (host logic, no GPU): drain
lengths the MMA issuer has a form for, widths, row strides of C, operands with
a range to watch."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHECK = r'''
#include "gemm_tc.cuh"
#include <cstdio>
using namespace ttnn;
static TcGemm gemm(int type) {
  TcGemm g;
  g.I = 1000; g.K = 500; g.Jn = 20; g.type = type; g.lda = 500; g.ldc = 32;
  g.b[0].n = 20; g.b[0].sk = 1; g.b[0].sj = 500;
  return g;
}
int main() {
  for (int type = 1; type <= 3; ++type) {
    for (int chain = -1; chain <= 33; ++chain) {
      TcGemm g = gemm(type);
      g.chain = chain;
      printf("%d", (int)tcg_supported(g));
    }
    TcGemm w = gemm(type), c = gemm(type), k = gemm(type), s = gemm(type);
    w.Jn = 81; w.ldc = 96;
    c.ldc = 30;
    k.K = 0;
    int32_t shift[64];
    s.shift = shift;   // not a Khatri-Rao operand of two factors
    printf(" %d%d%d%d\n", (int)tcg_supported(w), (int)tcg_supported(c), (int)tcg_supported(k), (int)tcg_supported(s));
  }
}
'''


def test_requests_the_gemm_has_no_form_for_are_refused(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    lib = os.path.join(ROOT, "paper_2412_06111_gb300", "_build")
    if not os.path.exists(nvcc):
        pytest.skip("no CUDA toolkit")
    from paper_2412_06111_gb300 import _native
    _native.build()
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(CHECK)
    subprocess.run([nvcc, "-std=c++17", "-arch=sm_103a", "-cudart", "shared", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2412_06111_gb300", "csrc"), str(src), "-o", str(exe),
                    os.path.join(lib, "libttnn.so"), "-Xlinker", "-rpath=" + lib], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")
    take = lambda ok: "".join("1" if c in ok else "0" for c in range(-1, 34))
    assert out[0] == take((0, 2, 8, 16)) + " 0000"       # binary32
    assert out[1] == take((0, 8, 16)) + " 0000"          # bfloat16
    assert out[2] == take((0, 2, 8, 16)) + " 0000"       # binary64 rounded to binary32
