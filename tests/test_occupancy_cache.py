"""The cooperative kernel's occupancy is asked of the runtime once and kept, but not a
failure of that question (the first load of a kernel can find no device memory): the
next call asks again.  The object file of one form is linked against a stand-in for
the CUDA runtime whose first answer is an error."""
import os
import re
import subprocess

import paper_2605_02030_gb300 as pkg

FAKE = r"""
#include <cstddef>
static int asked = 0;
extern "C" int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = asked++ ? 5 : 0;
  return asked > 1 ? 0 : 2;  // cudaErrorMemoryAllocation
}
extern "C" int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                                      unsigned) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, nullptr, 0, 0);
}
namespace uhnsw_dev {
struct WarpShape { int team, cpl, u; bool most; };
int csearch_regs_f32_w2(WarpShape);
}
int main() {
  for (int i = 0; i < 3; ++i) __builtin_printf("%d ", uhnsw_dev::csearch_regs_f32_w2({8, 1, 0, false}));
  __builtin_printf("%d\n", asked);
}
"""


def test_a_failed_question_is_asked_again(tmp_path):
    lib = pkg.build()
    obj = os.path.join(os.path.dirname(lib), "csearch_f32_w2.o")
    if not os.path.exists(obj):
        pkg.build(force=True)
    undefined = subprocess.run(["nm", "-u", obj], capture_output=True, text=True, check=True).stdout
    stubs = [s for s in re.findall(r"\bU (\w+)", undefined)
             if s.startswith(("cuda", "__cuda")) and not s.startswith("cudaOccupancyMax")]
    src = tmp_path / "fake.cpp"
    src.write_text(FAKE + "".join(f'extern "C" long {s}(...) {{ return 0; }}\n' for s in stubs))
    exe = tmp_path / "fake"
    subprocess.run(["g++", "-std=c++17", "-o", exe, src, obj], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    assert out.split() == ["0", "5", "5", "2"]
