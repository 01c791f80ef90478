"""pic_field_solve_static: the set-up of the first call on a device reaches
every kernel that any later call may launch, of any size and precision, so that
a warm-up call leaves nothing for lazy loading to load inside a capture or a
region that must not allocate.  A small program includes the source and looks
at what the set-up touches (asking for a kernel's attributes loads it)."""
import os
import subprocess

from paper_0705_0495_gb300 import build

CODE = r"""
#include "o2pic_static.cu"
#include <set>
static std::set<const void *> touched;
namespace o2 {
void set_last_error(const char *) {}
cudaError_t allow_smem(const void *k, size_t) { touched.insert(k); return cudaSuccess; }
}
template <typename... A> static bool has(void (*k)(A...)) { return touched.count(reinterpret_cast<const void *>(k)) != 0; }
int main()
{
    if (static_setup<float>() != cudaSuccess || static_setup<double>() != cudaSuccess) return 1;
    if (!has(k_static_small<float>) || !has(k_static_small<double>)) return 2;
    if (!has(k_static_deposit<float>) || !has(k_static_deposit<double>)) return 3;
    if (!has(k_static_solve<float>) || !has(k_static_solve<double>)) return 4;
    return 0;
}
"""


def test_the_set_up_reaches_every_kernel(tmp_path):
    (tmp_path / "t.cu").write_text(CODE)
    subprocess.run(["nvcc", *build.ARCH, "-std=c++17", "-I", build.CSRC, str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")],
                   check=True, capture_output=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0
