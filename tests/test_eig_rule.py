"""The eigen-step's stopping rule (rpca_eig_rule.cuh), compiled for the host: whatever it accepts, the first-order
formula for Wbar = f(diag(d) + E), f(s^2) = min(1, tau / s), is right to about the Gram's own FP32 rounding, the kink of f at tau included.

Bound: the rule's limits allow 3/8 kEigMaxOff^2 = 6e-8 (smooth), kEigEps / 2 = 5e-7 in the divided difference over the
kink, and kEigEps / 2 where an eigenvalue crosses tau; the sum of the last two, 1e-6, with the next order (a relative 1e-3)
and the FP32 rounding of the rule's own arithmetic (a relative 1e-5), is taken as 1.01e-6.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BOUND = 1.01e-6


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text('#include "rpca_eig_rule.cuh"\n'
                                'extern "C" int accepts(float e, float om, float hi, float lo, float tau) {\n'
                                '  const int kept = (hi > tau) + (lo > tau);\n'
                                '  if (kept && eig_pair_off(e, om, hi, lo, kept)) return 0;\n'
                                '  if (kept == 1) return 1;\n'
                                '  const float w = eig_pair_shift(e, om, hi, lo);\n'
                                '  return !eig_row_off(kept == 2, hi, w, tau) && !eig_row_off(kept == 2, lo, w, tau);\n'
                                '}\n')
    so = str(d / "rule.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2506_10257_gb300", "csrc"), "-o", so,
                    str(d / "rule.cpp")], check=True)
    f = ctypes.CDLL(so).accepts
    f.argtypes = [ctypes.c_float] * 5
    return f


def wbar_error(dp, dq, e, tau):
    """Largest error of the first-order formula for f([[dp, e], [e, dq]])."""
    f = lambda x: np.minimum(1.0, tau / np.sqrt(np.maximum(x, 1e-300)))
    if dp == dq:
        div = -tau / (2 * dp ** 1.5) if dp > tau * tau else 0.0
    else:
        div = (f(dp) - f(dq)) / (dp - dq)
    # f of the matrix through its eigenvalues, in a form without cancellation
    r = np.hypot(dp - dq, 2 * e)
    lp, lm = (dp + dq + r) / 2, (dp * dq - e * e) / ((dp + dq + r) / 2)
    s = (f(lp) - f(lm)) / r if r > 0 else 0.0
    exact = np.array([(f(lp) + f(lm)) / 2 + s * (dp - dq) / 2, s * e, (f(lp) + f(lm)) / 2 - s * (dp - dq) / 2])
    return np.abs(exact - np.array([f(dp), div * e, f(dq)])).max()


# (relative positions of d_p and d_q about tau^2)
NEAR = [0.0, 1e-7, 1e-6, 1e-5, 1e-4, 3e-4, 1e-3, 1e-2, 0.1, 0.5]


@pytest.mark.parametrize("side", ["straddling", "above", "below"])
def test_what_the_rule_accepts_is_right_to_the_bound(rule, side):
    tau, worst, accepted = 1.0, 0.0, 0
    rng = np.random.Generator(np.random.PCG64(7))
    for a in NEAR + [3.0, 100.0]:
        for b in NEAR:
            for e in 10.0 ** np.concatenate([np.arange(-8, -1.9, 0.25), rng.uniform(-6, -3, 20)]):
                if side == "straddling":
                    dp, dq = 1 + a + 1e-9, 1 - b
                elif side == "above":
                    dp, dq = 1 + max(a, b) + 1e-9, 1 + min(a, b) + 1e-9
                else:
                    dp, dq = 1 - min(a, b), 1 - max(a, b)
                    if a > 0.5:
                        continue
                hi, lo = np.float32(np.sqrt(dp)), np.float32(np.sqrt(dq))
                dp, dq = float(hi) ** 2, float(lo) ** 2  # what the rule is given, exactly
                if not rule(e, 0.0, hi, lo, tau):
                    continue
                accepted += 1
                worst = max(worst, wbar_error(dp, dq, float(np.float32(e)), tau))
    assert accepted > 200 and worst <= BOUND, (accepted, worst)


def test_what_the_sweeps_leave_is_accepted_away_from_tau(rule):
    # the rule must not ask for another round where none is needed
    assert rule(3e-4, 0.0, 1.5, 1.2, 1.0)      # both above
    assert rule(2e-4, 0.0, 1.2, 0.5, 1.0)      # straddling, well apart
    assert rule(1e-2, 0.0, 0.5, 0.49, 1.0)     # neither, far below
    assert not rule(1e-3, 0.0, 1.5, 1.2, 1.0)
    assert not rule(1e-6, 3e-4, 1.5, 1.2, 1.0)  # orthonormality lost
