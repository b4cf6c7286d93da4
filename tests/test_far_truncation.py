"""Truncation error of the surface sums' local expansions, on the CPU: the degrees and the
separation that the kernels use leave less than one FP32 rounding of the sum of absolute terms."""
import os
import re

import numpy as np
from numpy.polynomial import legendre

import pb_inputs

SOURCE = os.path.join(os.path.dirname(__file__), "..", "paper_2502_09323_gb300", "csrc", "nbody_far.cuh")


def _constant(text, name):
    m = re.search(r"constexpr [^;]*\b%s = (\d+(?:\.\d*)?)" % name, text)
    return float(m.group(1))


def test_truncation():
    with open(SOURCE) as fh:
        text = fh.read()
    P, PD, kappa = int(_constant(text, "P")), int(_constant(text, "PD")), _constant(text, "KAPPA")
    rng = np.random.default_rng(7)
    atoms = pb_inputs.globular_molecule(20000, seed=8)
    y0, q = atoms[:, :3] - atoms[:, :3].mean(0), atoms[:, 4]
    reach = np.linalg.norm(y0, axis=1).max()
    worst = [0.0, 0.0]
    for a in (3.0, 5.0):
        for _ in range(4):
            v = rng.normal(size=3)
            c = v / np.linalg.norm(v) * reach  # a block of the surface
            y = y0 - c
            d = np.linalg.norm(y, axis=1)
            # targets all over the ball, its surface included
            x = rng.normal(size=(12, 3))
            x *= (a * rng.random(12) ** 0.2 / np.linalg.norm(x, axis=1))[:, None]
            x[0] *= a / np.linalg.norm(x[0])
            for t in x:
                rho = np.linalg.norm(t)
                r = np.linalg.norm(y - t, axis=1)
                scale = [(np.abs(q) / r).sum(), (np.abs(q) / r ** 2).sum()]
                rest = [0.0, np.zeros(3)]
                for far, degree in ((d > kappa * a) & (d <= 2 * kappa * a), P), (d > 2 * kappa * a, PD):
                    yh = y[far] / d[far, None]
                    cos = yh @ t / rho
                    pot, grad = 1 / r[far], (y[far] - t) / r[far, None] ** 3
                    for l in range(degree + 1):
                        e = np.zeros(l + 1)
                        e[l] = 1.0
                        p, dp = legendre.legval(cos, e), legendre.legval(cos, legendre.legder(e)) if l else 0 * cos
                        pot = pot - rho ** l / d[far] ** (l + 1) * p
                        if l:
                            grad = grad - (rho ** (l - 1) / d[far] ** (l + 1))[:, None] * (
                                (l * p - cos * dp)[:, None] * t / rho + dp[:, None] * yh)
                    rest[0] += (q[far] * pot).sum()
                    rest[1] = rest[1] + (q[far, None] * grad).sum(0)
                worst[0] = max(worst[0], abs(rest[0]) / scale[0])
                worst[1] = max(worst[1], np.linalg.norm(rest[1]) / scale[1])
    assert max(worst) <= 2.0 ** -24, worst
