"""Coefficients of the step-weight polynomial in lf_precompute.cu
(one_minus_exp_over_x).

(1 - exp(-x)) / x on [0, 1] is taken as 1 + x P(x), P of degree 5: the
interpolation of -1/2! + x/3! - x^2/4! + ... at the 6 Chebyshev nodes of [0, 1], solved
in exact rational arithmetic (nodes as float64) and rounded to float32.

  python fit_step_weight.py            # prints the float32 coefficients, lowest first
"""
import math
from fractions import Fraction

import numpy as np

TERMS = 6
SERIES = 30               # terms of the series: the next is below 1e-32 on [0, 1]


def fit():
    xs = [Fraction(0.5 + 0.5 * math.cos(math.pi * (2 * k + 1) / (2 * TERMS))) for k in range(TERMS)]
    rows = [[x ** k for k in range(TERMS)] + [sum(Fraction((-1) ** (k + 1), math.factorial(k)) * x ** (k - 2)
                                                  for k in range(2, SERIES))] for x in xs]
    for i in range(TERMS):                               # Gauss-Jordan
        rows[i] = [a / rows[i][i] for a in rows[i]]
        for j in range(TERMS):
            if j != i:
                rows[j] = [a - rows[j][i] * b for a, b in zip(rows[j], rows[i])]
    return [float(r[TERMS]) for r in rows]


def coefficients_f32() -> np.ndarray:
    return np.array(fit()).astype(np.float32)


def eval_f32(c: np.ndarray, x: np.ndarray) -> np.ndarray:
    """1 + x P(x) by Horner in float32, one rounding per multiply-add, as the kernel."""
    x = x.astype(np.float32)
    h = np.full_like(x, c[-1])
    for ck in [*c[-2::-1], np.float32(1.0)]:
        h = (h.astype(np.float64) * x.astype(np.float64) + np.float64(ck)).astype(np.float32)
    return h


if __name__ == "__main__":
    c = coefficients_f32()
    print(", ".join(repr(float(v)) + "f" for v in c))
    x = np.linspace(0.0, 1.0, 1_000_001)[1:]
    print("max |error| in float32 evaluation:",
          float(np.abs(eval_f32(c, x) + np.expm1(-x.astype(np.float32).astype(np.float64)) / x.astype(np.float32)).max()))
