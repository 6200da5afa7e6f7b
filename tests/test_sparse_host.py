"""Host side of the sparse matrices under the compiler's undefined-behaviour checks: the records of
an observable are formed before anything touches the device."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

MAIN = r"""
#include "sparse.cu"
#include <memory>
namespace qs {
int fail(int code, const char*, ...) { return code; }
}
int main() {
  for (int n = 1; n <= 34; ++n) {
    const uint64_t top = 1ull << (n - 1);
    const uint64_t masks[][2] = {{0, top}, {0, 1}, {0, 1 | top}, {0, 0}, {1, 0}, {top, top}, {1 | top, 1}, {1, top}};
    for (size_t k = 0; k < 8; k += 2) {  // two terms an observable: groups with a table of values
      qs_observable o;
      for (size_t j = k; j < k + 2; ++j) {
        qs_pauli_term t = {};
        t.coeff = 0.5 + n;
        t.x_mask = masks[j][0];
        t.z_mask = masks[j][1];
        o.terms.push_back(t);
      }
      auto T = std::make_unique<qs::SpTerms>();
      auto tab = std::make_unique<qs::SpTable>();
      if (qs::build_terms(&o, n, T.get(), tab.get()) != QS_OK) return 2;
    }
  }
  return 0;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_records_of_every_register_size(tmp_path):
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(MAIN)
    cmd = [NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "--expt-relaxed-constexpr",
           "-I", os.path.join(ROOT, "paper_1912_10877_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
           "-Xcompiler", "-fsanitize=undefined", "-Xcompiler", "-fno-sanitize-recover=undefined", str(src), "-o", str(exe)]
    subprocess.run(cmd, check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "runtime error" not in r.stderr, r.stderr
