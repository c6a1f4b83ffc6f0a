"""The coefficient table's products round as the source says: the file that forms them is
compiled without contraction, and then gives the same bits whatever the compiler may
inline and whether or not the processor has a fused multiply-add."""
import os
import platform
import re
import subprocess

from paper_2506_03617_gb300 import build as B

MAIN = r"""
#include <cstdio>
#include "coef.inc"
int main()
{
    const mxp::PmlAxis axes[] = {{16, 40, 1.0 / 40, 20.0, 31.4}, {7, 23, 1.0 / 23, 26.3, 13.5}, {1, 31, 1.0 / 31, 19.1, 19.9}};
    for (const auto &a : axes)
        for (long i = 0; i < a.n_interior + 2 * a.npml; ++i)
            for (int b = 0; b < 2; ++b) {
                mxp::cd p, m;
                mxp::pml_neighbours(a, i, b, &p, &m);
                std::printf("%a %a %a %a\n", p.real(), p.imag(), m.real(), m.imag());
            }
}
"""


def _host_only():
    with open(os.path.join(B.CSRC, "coef.cu")) as fh:
        src = fh.read().replace('#include "mxp_internal.h"', "#include <complex>\n#include <cstdint>\n#include \"axis.inc\"")
    with open(os.path.join(B.CSRC, "mxp_internal.h")) as fh:
        axis = re.search(r"struct PmlAxis \{.*?\};\nvoid pml_neighbours[^;]*;", fh.read(), re.S).group(0)
    return src, "namespace mxp {\n" + axis + "\n}\n"


def test_no_contraction_in_the_build():
    assert B.FILE_FLAGS["coef.cu"][-1] == "-ffp-contract=off"
    assert any(os.path.basename(s) == "coef.cu" for s in B.sources())
    with open(os.path.join(B.CSRC, "engine.cu")) as fh:
        assert "inv_stretch" not in fh.read()             # formed in coef.cu only


def test_bits_do_not_depend_on_the_compiler(tmp_path):
    src, axis = _host_only()
    (tmp_path / "coef.inc").write_text(src)
    (tmp_path / "axis.inc").write_text(axis)
    (tmp_path / "main.cpp").write_text(MAIN)
    flags = [f for f in B.FILE_FLAGS["coef.cu"] if f != "-Xcompiler"]
    variants = [["-O0"], ["-O2"], ["-O3"], ["-O3", "-fno-inline"]]
    if platform.machine() == "x86_64" and "fma" in open("/proc/cpuinfo").read():
        variants.append(["-O3", "-mfma"])
    out = []
    for k, v in enumerate(variants):
        exe = str(tmp_path / f"m{k}")
        subprocess.run(["g++", "-std=c++17", *v, *flags, str(tmp_path / "main.cpp"), "-o", exe], check=True)
        out.append(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert len(out[0].splitlines()) == 2 * (72 + 37 + 33)
    assert all(o == out[0] for o in out[1:])
    if len(variants) == 5:                                 # left to the compiler they differ
        exe = str(tmp_path / "c")
        plain = src.replace("std::fma(-ai, bi, ar * br)", "(ar * br - ai * bi)").replace(
            "std::fma(ar, br, -(ai * bi))", "(ar * br - ai * bi)").replace(
            "std::fma(ai, br, ar * bi)", "(ar * bi + ai * br)").replace("std::fma(ar, bi, ai * br)", "(ar * bi + ai * br)")
        (tmp_path / "coef.inc").write_text(plain)
        subprocess.run(["g++", "-std=c++17", "-O3", "-mfma", str(tmp_path / "main.cpp"), "-o", exe], check=True)
        assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout != out[0]
