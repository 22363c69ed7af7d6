"""The constants that the stage-form kernels take (every FP32 solve, swarm and
per-pixel batch, the finite-element kernel) do not carry the affine map of the
step: it is two thirds of the words and host time that those calls would pay
for without reading it.  Compiled with the host compiler from the library's
header."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "afm_internal.h"
int main() {
    using namespace afm;
    std::printf("%zu %zu %zu %zu %zu %zu\n", sizeof(KConst<float>), sizeof(Affine<float>),
                sizeof(KConst<double>), sizeof(Affine<double>), sizeof(FeConst),
                sizeof(double) * 7 * AFM_FE_MAXN);
}
"""


def test_affine_map_is_apart(tmp_path):
    src, exe = tmp_path / "sizes.cpp", tmp_path / "sizes"
    src.write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1109_0334_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"),
                    str(src), "-o", str(exe)], check=True)
    kf, af, kd, ad, fe, fe_modes = map(int, subprocess.run([str(exe)], check=True,
                                                            capture_output=True, text=True).stdout.split())
    assert kf < af and kd < ad
    assert fe < fe_modes + 200 + kf          # FeConst: its mode arrays, scalars and KConst<float>
