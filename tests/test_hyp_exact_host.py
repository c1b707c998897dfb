"""The exact 4-point homographies and their FP32 evaluation forms (csrc/hyp_exact.cuh), compiled for the host, against
rational arithmetic: targets within frames, and imported offsets up to 2^22 beyond them mixed into a sample."""
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1804_03787_gb300 import build_lib

SRC = r"""
#include <cstdio>
#include "hyp_exact.cuh"
using namespace gpm;
int main() {
    int v[16];
    for (;;) {
        for (int k = 0; k < 16; ++k)
            if (scanf("%d", v + k) != 1) return 0;
        i128 H[9];
        Mef m;
        minimal_h_exact(v, v + 4, v + 8, v + 12, H);
        const int ok = make_mef_exact(H, m);
        for (int k = 0; k < 9; ++k) printf("%016llx%016llx ", (unsigned long long)((u128)H[k] >> 64), (unsigned long long)H[k]);
        printf("%d %a %a %a %a %a %a %a %a %a %a %a\n", ok, m.b0, m.h1, m.h2h, m.h2l, m.h3, m.b4, m.h5h, m.h5l, m.g0, m.g1, m.e0);
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("hyp")
    src = d / "hyp.cu"
    src.write_text(SRC)
    exe = str(d / "hyp")
    subprocess.run([build_lib.nvcc(), "-std=c++17", "-I", build_lib.CSRC, str(src), "-o", exe], check=True,
                   capture_output=True)
    return exe


@pytest.mark.parametrize("bits", [7, 15, 19, 22])
def test_exact_homography_and_its_form(program, bits):
    rng = np.random.default_rng(bits)
    n = 200
    p = rng.integers(-48, 48, (n, 2, 4))
    q = p + rng.integers(-20, 20, (n, 2, 4))
    far = rng.integers(-(1 << bits) + 100, (1 << bits) - 100, (n, 2, 4))
    q = np.where(rng.random((n, 1, 4)) < rng.random((n, 1, 1)), far, q)
    text = "\n".join(" ".join(map(str, np.concatenate([a, b]).reshape(-1))) for a, b in zip(p, q))
    out = subprocess.run([program], input=text, check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(out) == n
    u, forms = Fraction(1, 1 << 24), 0
    for (px, py), (qx, qy), line in zip(p.tolist(), q.tolist(), out):
        w = line.split()
        H = [int(h, 16) - (1 << 128 if int(h, 16) >> 127 else 0) for h in w[:9]]
        for k in range(4):  # H (p, 1) is proportional to (q, 1)
            X, Y, Z = (H[3 * r] * px[k] + H[3 * r + 1] * py[k] + H[3 * r + 2] for r in range(3))
            assert X == qx[k] * Z and Y == qy[k] * Z
        dc2 = 2 * H[8] - H[6] - H[7]
        assert int(w[9]) == (dc2 != 0)
        if dc2 == 0:
            continue
        forms += 1
        b0, h1, h2h, h2l, h3, b4, h5h, h5l, g0, g1, e0 = (Fraction(float.fromhex(v)) for v in w[10:])
        r = [Fraction(2 * h, dc2) for h in H]
        for got, want in ((b0, r[0] - 1), (h1, r[1]), (h3, r[3]), (b4, r[4] - 1), (g0, r[6]), (g1, r[7]), (e0, r[8] - 1)):
            assert abs(got - want) <= 6 * u * abs(want)  # three limbs' sums, the reciprocal, the product: 2^-24 each
        for hi, lo, want in ((h2h, h2l, r[2]), (h5h, h5l, r[5])):
            if abs(want) >= Fraction(1, 1 << 19):  # the low part carries what the high part's rounding left
                assert abs(hi + lo - want) <= 6 * u * 4 * u * abs(want)
    assert forms > n // 4
