"""The kernels that hand registers from warpgroup to warpgroup wait without a
limit if the launch holds fewer than their split's sum: the launchers accept
exactly the compiled count whose launch holds it (regsplit.h, host code)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "regsplit.h"
#include <cstdio>
int main() {
  for (int r = 1; r <= 255; ++r)
    std::printf("%d %d %d\n", r, (int)kvk::kPfRegs.fits(r), (int)kvk::kEvictRegs.fits(r) + 2 * kvk::kMlaQRegs.fits(r));
}
"""


def test_split_fits_only_its_own_launch(tmp_path):
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_37988_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    rows = [tuple(map(int, l.split())) for l in subprocess.run([str(exe)], check=True, capture_output=True,
                                                              text=True).stdout.splitlines()]
    # allocated in units of 8 a thread: 640 x 96 = 512 x 104 + 128 x 64, 896 x 72 = 512 x 88 + 256 x 56 + 128 x 40,
    # 512 x 128 = 128 x 256 + 128 x 96 + 256 x 80
    assert [r for r, pf, _ in rows if pf] == list(range(89, 97))
    assert [r for r, _, x in rows if x & 1] == list(range(65, 73))
    assert [r for r, _, x in rows if x & 2] == list(range(121, 129))

