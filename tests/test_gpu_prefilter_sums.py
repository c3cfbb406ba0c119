"""The moving average's sums carry at least what sums in 64 bits carry: frames of opposite sign that cancel, and a huge
value that has slid out of the window, leave no more behind than FP64 sliding sums do.

Bound, per output: half a unit of FP32 rounding of the result (the result below is rounded once), plus what FP64 sums of
the same steps may be off by: 2^-53 of the largest partial sum for each of the steps that formed it, divided by the window.
The exact values are sums of fractions.
"""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_10257_gb300 import rpca
    rpca.load()
    return rpca


def frames(kind, T, m):
    rng = np.random.Generator(np.random.PCG64(11))
    F = (1.0 + 0.1 * rng.standard_normal((T, m))).astype(np.float32)
    if kind == "opposite":      # neighbours of opposite sign, 2^24 and more above what they leave
        big = np.float32(3e7) * (1 + rng.random((T // 2, m))).astype(np.float32)
        F[0:2 * (T // 2):2] = big
        F[1:2 * (T // 2):2] = -big
        F += rng.standard_normal((T, m)).astype(np.float32)
    elif kind == "slides out":  # one frame far above the rest
        F[2] = np.float32(1e15) * (1 + rng.random(m)).astype(np.float32)
        F[T - 2] = -np.float32(1e12) * (1 + rng.random(m)).astype(np.float32)
    elif kind == "constant":    # nothing left by the high-pass
        F[:] = (1 + rng.random(m)).astype(np.float32)
    elif kind == "small":       # means that are subnormal, and just above
        F *= np.float32(2.0 ** -120)
        F[:, ::3] *= np.float32(2.0 ** -14)
    return F


@pytest.mark.parametrize("high_pass", [False, True])
@pytest.mark.parametrize("window", [1, 7, 20])
@pytest.mark.parametrize("kind", ["plain", "opposite", "slides out", "constant", "small"])
def test_window_sums_are_no_further_off_than_fp64(rp, kind, window, high_pass):
    T, m = 44, 24
    F = frames(kind, T, m)
    Y, kept, _ = rp.prefilter(torch.from_numpy(F).cuda(), corr_min=-2.0, window=window, high_pass=high_pass)
    assert kept.cpu().tolist() == list(range(T))
    got = Y.cpu().numpy()
    assert got.shape == (T - window + 1, m)
    for p in range(m):
        col = [Fraction(float(v)) for v in F[:, p]]
        for j0 in range(0, len(got), 16):  # a thread's outputs: one sum formed, then slid
            s, top, steps = Fraction(0), Fraction(0), 0
            for i in range(window):
                s += col[j0 + i]
                top, steps = max(top, abs(s)), steps + 1
            for j in range(j0, min(j0 + 16, len(got))):
                if j > j0:
                    s += col[j + window - 1]
                    top = max(top, abs(s))
                    s -= col[j - 1]
                    top, steps = max(top, abs(s)), steps + 2
                exact = s / window
                off = steps * top / window / 2 ** 53 + abs(exact) / 2 ** 52  # the sums; 1 / window and the product
                if high_pass:
                    exact = col[j + (window - 1) // 2] - exact
                    off += abs(exact) / 2 ** 53
                half = float(np.spacing(np.float32(abs(float(exact)) + float(off)))) / 2
                err = abs(Fraction(float(got[j, p])) - exact)
                assert err <= Fraction(half) + off, (kind, window, p, j, float(err), half, float(off))
