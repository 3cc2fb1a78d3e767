"""Types of the resident COCG kernel's scalars, checked by the compiler: the sums over warps and
blocks, rho, ||r||^2 and its target are FP64 in the FP32 form too, as in the launched
iteration, and with RPA_DOT_F64 = 1 the threads' and warps' dot products are."""
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


@pytest.mark.skipif(shutil.which(NVCC) is None, reason="needs nvcc")
@pytest.mark.parametrize("flag,want", [("-DRPA_DOT_F64=1", "double"), ("-DRPA_DOT_F64=0", "float")])
def test_dot_products_follow_the_build_flag(tmp_path, flag, want):
    compiles(tmp_path, "\n".join(
        f"static_assert(same<decltype({e}), {want}>, \"{n}\");"
        for n, e in (("p^T w", "part_y<float, 4, 6>().re"),
                     ("r^T r", "phase_update<float, true, true>().v[0]"),
                     ("warp sums", "Brick<float>::red[0]"))), flag)
