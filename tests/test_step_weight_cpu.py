"""The volume march's step-weight polynomial (1 - exp(-x)) / x = 1 + x P(x) on [0, 1]:
the kernel's coefficients are those its fit script writes, and stay within the stated
error of the function, exactly and in float32."""
import importlib.util
import os
import re

import numpy as np

from paper_1903_03837_gb300 import build as B


def kernel_coefficients():
    src = open(os.path.join(B.CSRC, "lf_precompute.cu")).read()
    body = src[src.index("float one_minus_exp_over_x(float x)"):]
    body = body[:body.index("\n}")]
    first = re.search(r"float h = (\S+)f;", body).group(1)
    rest = re.findall(r"fmaf\(h, x, (\S+)f\)", body)
    return np.array([float(v) for v in [first, *rest]], dtype=np.float32)[::-1]     # 1, c0, c1, ...


def fit_script():
    spec = importlib.util.spec_from_file_location("fit_step_weight", os.path.join(B.CSRC, "fit_step_weight.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def test_coefficients_come_from_the_fit_script():
    c = kernel_coefficients()
    assert len(c) == 7 and c[0] == 1.0
    assert np.array_equal(c[1:], fit_script().coefficients_f32())


def test_error_of_the_polynomial():
    """4e-8 in exact arithmetic; in float32 a rounding of the result (3.0e-8 below 1)
    and of x P(x) (up to 1.5e-8, its own error passed on halved by each x < 1) more."""
    c = kernel_coefficients()[1:]
    x = np.linspace(0.0, 1.0, 400_001)[1:].astype(np.float32).astype(np.float64)
    want = -np.expm1(-x) / x
    assert np.abs(1.0 + x * np.polyval(fit_script().fit()[::-1], x) - want).max() <= 4e-8
    assert np.abs(fit_script().eval_f32(c, x) - want).max() <= 1.1e-7
    assert fit_script().eval_f32(c, np.zeros(1))[0] == 1.0
