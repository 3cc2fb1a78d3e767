"""Types of the resident COCG kernel's scalars, checked by the compiler: the sums over warps and
blocks, rho, ||r||^2 and its target are FP64 in the FP32 form too, as in the launched
iteration."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_16408_gb300", "csrc")
NVCC = os.environ.get("NVCC", "nvcc")


def compiles(tmp_path, checks, *flags):
    src = tmp_path / "check.cu"
    src.write_text('#include "cocg_resident.cu"\n#include <type_traits>\nnamespace rpa {\n'
                   "template <typename A, typename B>\n"
                   "constexpr bool same = std::is_same<typename std::remove_reference<A>::type, B>::value;\n"
                   + checks + "\n}\n")
    r = subprocess.run([NVCC, "-arch=sm_103a", "-ptx", "-Xcicc", "-O0", "-std=c++17", *flags,
                        "-I" + CSRC, "-I" + os.path.join(ROOT, "include"), str(src), "-o",
                        str(tmp_path / "check.out")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


@pytest.mark.skipif(shutil.which(NVCC) is None, reason="needs nvcc")
def test_scalars_are_fp64(tmp_path):
    compiles(tmp_path, "\n".join(
        f"static_assert(same<decltype(Brick<float>::{m}), double>, \"{m}\");"
        for m in ("rho_r", "rho_i", "rn2", "target2")) + "\n" + "\n".join(
        f"static_assert(same<decltype(Brick<float>::{m}[0]), double>, \"{m}\");"
        for m in ("slots2", "slots3")))
