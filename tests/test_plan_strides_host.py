"""The distance between a tile's block planes, on the host: pass_plan.cpp built with
the host compiler against stub launchers.  Only tiles of the paired peak search in a
kernel specialised to its shape (50 % overlap, blocks of 8, 12, 16, 24 or 32 px, radii 1
to 4) may have their planes spread: the other kernels hold the distance as a constant,
the planes' own size (a 16-bit tile's row groups keep their partial planes beside one
another)."""
import os
import shutil
import subprocess

import pytest

from test_plan_host import CSRC, ROOT, THREADS, _cuda_include

MAIN = r"""
#define main probe_main
#include "plan_probe.cpp"
#undef main
int main()
{
    int w, s, R, nx, ny, prec;
    while (std::scanf("%d %d %d %d %d %d", &w, &s, &R, &nx, &ny, &prec) == 6) {
        rpiv::PassPlan p{};
        const bool ok = rpiv::pass_plan(w, s, R, nx, ny, prec, &p, nullptr);
        std::printf("%d %d %d %d %d\n", ok ? 1 : 0, p.pstride, p.RGx, p.TX, p.TY);
    }
    return 0;
}
"""


def test_planes_are_spread_only_for_kernels_that_read_them_so(tmp_path):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("host C++ compiler or CUDA headers not found")
    src, exe = tmp_path / "strides.cpp", str(tmp_path / "strides")
    src.write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, "-I", CSRC, "-I", os.path.join(ROOT, "tests"), str(src),
                    os.path.join(CSRC, "pass_plan.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    cases = [(w, s, R, n, n, prec) for w in range(8, 130, 2) for s in range(3, w + 1) for R in (0, 1, 2, 3, 4, 5, 6, 8, 16)
             for n in (3, 101) for prec in (0, 1) if prec == 0 or s in (w // 2, w // 4)]
    text = "".join(" ".join(map(str, c)) + "\n" for c in cases)
    env = {k: v for k, v in os.environ.items() if not k.startswith("RPIV_")}
    out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True, env=env).stdout.split("\n")
    spread = 0
    for (w, s, R, _, _, prec), line in zip(cases, out):
        ok, pstride, groups, TX, TY = map(int, line.split())
        if not ok:
            continue
        size = (2 * R + 1) ** 2
        if prec == 0 and w == 2 * s and s in (8, 12, 16, 24, 32) and 1 <= R <= 4 and TX * TY >= 2 * THREADS // 32:
            assert pstride >= size
            spread += pstride > size
        else:
            assert pstride == size * (1 if prec == 0 else groups), (w, s, R, prec)
    assert spread > 0
