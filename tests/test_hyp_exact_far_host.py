"""Exact hypotheses whose targets may be any imported integer (csrc/hyp_exact.cuh), compiled for the host: samples that
sample_in_range accepts stay inside the 128-bit products, and it accepts every sample about one or two places."""
import subprocess

import numpy as np
import pytest

from paper_1804_03787_gb300 import build_lib

SRC = r"""
#include <cstdio>
#include "hyp_exact.cuh"
using namespace gpm;
int main() {
    long long v[17];
    for (;;) {
        for (int k = 0; k < 17; ++k)
            if (scanf("%lld", v + k) != 1) return 0;
        int p[8];
        int64_t q[8], a[8];
        for (int k = 0; k < 8; ++k) p[k] = (int)v[k], q[k] = v[8 + k], a[k] = v[8 + k] + v[16];
        i128 H[9], A[9];
        Mef m;
        const int in = sample_in_range(q, q + 4, v[16] < 0 ? -v[16] : v[16]);
        if (in) {
            minimal_h_exact(p, p + 4, q, q + 4, H);
            minimal_h_exact(p, p + 4, a, a + 4, A);
            make_mef_exact(A, m);
        }
        printf("%d", in);
        for (int k = 0; k < 18 && in; ++k) {
            const i128 h = k < 9 ? H[k] : A[k - 9];
            printf(" %016llx%016llx", (unsigned long long)((u128)h >> 64), (unsigned long long)h);
        }
        if (in) printf(" %a %a %a %a", m.h2h, m.h2l, m.h5h, m.h5l);
        printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("hypfar")
    src = d / "hyp.cu"
    src.write_text(SRC)
    exe = str(d / "hyp")
    subprocess.run([build_lib.nvcc(), "-std=c++17", "-I", build_lib.CSRC, str(src), "-o", exe], check=True, capture_output=True)
    return exe


def _exact(px, py, qx, qy):
    """The same homography in Python integers."""
    dx, dy = [a - px[3] for a in px[:3]], [a - py[3] for a in py[:3]]
    X, Y = [a - qx[3] for a in qx[:3]], [a - qy[3] for a in qy[:3]]
    nxt = ((1, 2), (2, 0), (0, 1))
    l = [dx[i] * dy[j] - dx[j] * dy[i] for i, j in nxt]
    mu = [X[i] * Y[j] - X[j] * Y[i] for i, j in nxt]
    h = [[0, 0], [0, 0], [0, 0]]
    for k, (i, j) in enumerate(nxt):
        w = mu[k] * l[i] * l[j]
        for c, d in enumerate((dy[i] - dy[j], dx[j] - dx[i])):
            for r, t in enumerate((X[k], Y[k], 1)):
                h[r][c] += w * d * t
    h8 = l[0] * l[1] * l[2] * sum(mu) - h[2][0] * px[3] - h[2][1] * py[3]
    rows = []
    for r, q3 in ((0, qx[3]), (1, qy[3])):
        rows += [h[r][0] + h[2][0] * q3, h[r][1] + h[2][1] * q3, h8 * q3 - h[r][0] * px[3] - h[r][1] * py[3]]
    return rows + [h[2][0], h[2][1], h8]


@pytest.mark.parametrize("far,wild", [(20, 0), (30, 0), (31, 0), (31, 20), (32, 31)])
def test_samples_of_far_targets_stay_in_range(program, far, wild):
    """A share of each sample's targets moved by one marker of 2^far (wild: each by a random value below 2^wild instead), all
    of them about a reference of up to 2^31."""
    rng = np.random.default_rng(far + wild)
    n = 300
    p = rng.integers(-48, 48, (n, 2, 4))
    q = p + rng.integers(-16000, 16000, (n, 2, 4))
    jump = np.full((n, 2, 4), (1 << far) - 100000) * rng.choice([-1, 1], (n, 2, 1))
    if wild:
        jump = rng.integers(-(1 << wild), 1 << wild, (n, 2, 4))
    q = np.where(rng.random((n, 1, 4)) < 0.5, q + jump, q)
    v0 = rng.integers(-(1 << 31), 1 << 31, n)
    text = "\n".join(" ".join(map(str, [*a.reshape(-1), *b.reshape(-1), c])) for a, b, c in zip(p, q, v0))
    out = subprocess.run([program], input=text, check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(out) == n
    accepted = 0
    for (px, py), (qx, qy), v, line in zip(p.tolist(), q.tolist(), v0.tolist(), out):
        w = line.split()
        accepted += int(w[0])
        if w[0] == "0":
            continue
        H = [int(h, 16) - (1 << 128 if int(h, 16) >> 127 else 0) for h in w[1:19]]
        A = _exact(px, py, [a + v for a in qx], [a + v for a in qy])
        assert H[:9] == _exact(px, py, qx, qy) and H[9:] == A
        dc2 = abs(2 * A[8] - A[6] - A[7])
        assert max(map(abs, A)) < 1 << 126 and dc2 << 24 < 1 << 127
        if dc2:
            s = 1 if 2 * A[8] > A[6] + A[7] else -1
            for hi, lo, num in ((w[19], w[20], 2 * s * A[2]), (w[21], w[22], 2 * s * A[5])):
                want = num / dc2
                # the low part carries the high part's rounding: 24 units of 2^-48, when the quotient is above its own floor
                assert abs(want) < 1 or abs(float.fromhex(hi) + float.fromhex(lo) - want) <= 24 * 2.0**-48 * abs(want)
    assert accepted == n if wild < 22 else accepted < n
