"""Dequantisation by a reciprocal and an exact remainder (as in pac_quant.cuh) equals the correctly rounded quotient code / c: all 2^23 significands of
c, codes 1 to 128 (the sign changes nothing), at the ends and in the middle of the range of scales that takes this route."""
import os
import shutil
import subprocess

import pytest

SOURCE = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
int main(void) {
    const int exps[3] = {127 - 100, 127, 127 + 99};
    for (int k = 0; k < 3; ++k) {
        long bad = 0;
#pragma omp parallel for reduction(+ : bad)
        for (int64_t m = 0; m < (1 << 23); ++m) {
            const uint32_t bits = (uint32_t)exps[k] << 23 | (uint32_t)m;
            float c;
            memcpy(&c, &bits, 4);
            const float rc = 1.f / c;
            int miss = 0;
            for (int i = 1; i <= 128; ++i) {
                const float code = (float)i, y = code * rc, e = __builtin_fmaf(-y, c, code);
                miss += __builtin_fmaf(e, rc, y) != code / c;
            }
            bad += miss;
        }
        if (bad) { printf("exponent %d: %ld quotients differ\n", exps[k], bad); return 1; }
    }
    return 0;
}
"""


def test_every_significand(tmp_path):
    gcc = shutil.which("gcc")
    if not gcc:
        pytest.skip("no C compiler")
    src, exe = tmp_path / "q.c", tmp_path / "q"
    src.write_text(SOURCE)
    subprocess.run([gcc, "-O3", "-march=native", "-ffp-contract=off", "-fopenmp", "-o", str(exe), str(src), "-lm"], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, env={**os.environ, "OMP_NUM_THREADS": "4"})
    assert res.returncode == 0, res.stdout
