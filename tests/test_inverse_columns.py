"""Where the inversion without allocation writes its columns, as compiled code on the CPU.

Its scratch outlives a call.  When a bounded wait gives up, the pivot rows of the
call are incomplete, and what the array holds then may come from an earlier call
with a larger matrix: the columns have to stay inside the caller's matrix all the
same.  (The wait itself is not made to run out on a GPU: the entry point has no
setting for it.)
"""
import os
import subprocess

from paper_1010_3690_gb300 import build

PROGRAM = r"""
#include "ctaux_dev.cuh"
#include "ctaux_inverse.cuh"
int main() {
  using namespace ctaux;
  static int perm[512];
  for (int j = 0; j < 512; ++j) perm[j] = 511 - j;   // left by a call of order 512
  const int m = 137;
  for (int status : {(int)DS_TIMEOUT, DS_TIMEOUT | DS_SINGULAR})
    for (int j = 0; j < m; ++j)
      if (inv_column(status, DS_SINGULAR, perm, j) != j) return 1;
  for (int j = 0; j < m; ++j) perm[j] = (j + 5) % m;   // of a call that ended
  for (int status : {0, (int)DS_SINGULAR})
    for (int j = 0; j < m; ++j)
      if (inv_column(status, DS_SINGULAR, perm, j) != (j + 5) % m) return 2;
  return 0;
}
"""


def test_columns_stay_inside_the_matrix_when_a_wait_gave_up(tmp_path):
    src, exe = tmp_path / "columns.cu", tmp_path / "columns"
    src.write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    "-o", str(exe), str(src)], check=True, capture_output=True)
    assert subprocess.run([str(exe)]).returncode == 0
    # and the kernel that writes the inverse takes them from there
    code = open(os.path.join(build.CSRC, "ctaux_noalloc.cu")).read()
    assert "inv_column(status, DS_SINGULAR, v.perm, j)" in code and "v.perm[j]" not in code
