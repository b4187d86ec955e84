"""The fixed-point marches' host-side conversions, compiled from csrc/swr_fx.cuh and run on the CPU.

fx_limbs splits rint(c 2^61) into two signed 32-bit limbs.  A complex product negates the limbs of
its coefficient, so none may be -2^31, which has no negative."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1503_02564_gb300", "csrc")
PROGRAM = r"""
#include <stdio.h>
#include "swr_fx.cuh"
int main() {
    double re, im;
    while (scanf("%lf %lf", &re, &im) == 2) {
        const int4 c = fx_coef(re, im);
        printf("%d %d %d %d\n", c.x, c.y, c.z, c.w);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def convert(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("fx")
    (d / "limbs.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC,
                    "-o", str(d / "limbs"), str(d / "limbs.cu")], check=True, capture_output=True)

    def run(pairs):
        text = "".join(f"{a!r} {b!r}\n" for a, b in pairs)
        out = subprocess.run([str(d / "limbs")], input=text, capture_output=True, text=True, check=True)
        return [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    return run


def test_limbs(convert):
    # low limb exactly 2^31 (both signs), the edges of a limb, and a spread of ordinary values
    exact = [(2 * k + 1) * 2.0 ** -30 * s for k in (0, 1, 5, 2 ** 20, 2 ** 28 + 3, 2 ** 29) for s in (1, -1)]
    exact += [s * (k * 2.0 ** 32 + e) * 2.0 ** -61 for k in (0, 7, 2 ** 20) for e in (2 ** 31 - 1, 2 ** 31 + 1, 1)
              for s in (1, -1)]
    other = [1.999999, -1.999999, 0.0, 1e-30, -3.7e-12, 0.7071067811865476, 1 / 3, -1e-300]
    vals = exact + other
    got = convert([(v, -v) for v in vals])
    assert len(got) == len(vals)
    for v, (rh, rl, ih, il) in zip(vals, got):
        for c, h, low in ((v, rh, rl), (-v, ih, il)):
            assert -2 ** 31 < low < 2 ** 31 and -2 ** 31 < h < 2 ** 31
            num, den = c.as_integer_ratio()
            assert abs((h * 2 ** 32 + low) * den - num * 2 ** 61) <= den + den // 2   # rounding, and one unit


def test_history_sums_that_wrap_are_out_of_range():
    """sum |beta_s| over 2047 lags is 71.3, the traces stay below 2^58: a history sum in units of 2
    may reach 2^63.2 and wrap.  A wrapped one lies outside the 2^60 at which it is flagged."""
    a, total = 1.0, 0.0
    for k in range(0, 2048, 2):
        total += a + (a if k else 0.0)      # beta_0 belongs to the current step
        a *= (k + 1) / (k + 2)
    assert total < 72
    top = int(total * 2 ** 58) // 2
    assert 2 ** 63 < top < 2 ** 64 - 2 ** 60     # wrapped: from top - 2^64 to -2^63, all below -2^60
    for s in (2 ** 63, top, (2 ** 63 + top) // 2):
        assert abs(((s + 2 ** 63) % 2 ** 64) - 2 ** 63) >= 2 ** 60
