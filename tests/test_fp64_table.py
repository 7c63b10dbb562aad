"""The table of sines and cosines of the double-precision step is read with
16-byte loads, which fault on an address that is no multiple of 16: its type
has to ask for that alignment, wherever the linker places it.  Checked by the
compiler alone, without a GPU."""
import subprocess

from paper_2401_14221_gb300 import build as kbuild

SOURCE = """
#include "kf_fp64.cuh"
static_assert(alignof(decltype(kf::f64::kSinCos)) % alignof(double2) == 0 &&
                  alignof(double2) == 16, "the table is aligned for double2 loads");
static_assert(sizeof(kf::f64::kSinCos.v[0]) == sizeof(double2), "an entry is one load");
"""


def test_table_is_aligned_for_its_loads(tmp_path):
    src = tmp_path / "table.cu"
    src.write_text(SOURCE)
    r = subprocess.run([kbuild._nvcc(), *kbuild.ARCH, "-std=c++17", "--expt-relaxed-constexpr",
                        f"-I{kbuild.CSRC}", "-c", str(src), "-o", str(tmp_path / "table.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
