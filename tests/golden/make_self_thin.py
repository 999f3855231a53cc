"""Write the singular self rule of drops that are thin along a coordinate axis, in extended precision (test
infrastructure).  The FP64 oracle's own rounding reaches 2e-11 of a component on these shapes.

Calls only the oracle (and the seeded input generators): shapes and densities of `drop(p, axis)`, single and
double layer at the latitudes of `lats(p)`, rounded to FP64.  Output: tests/golden/self_thin.npz.  Needs a
longdouble of at least 64 bits of mantissa (x86).

    python tests/golden/make_self_thin.py
"""
from __future__ import annotations

import os
import sys
from concurrent.futures import ProcessPoolExecutor

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(os.path.dirname(HERE)))

from oracle import extended  # noqa: E402
from paper_1707_02156_gb300 import inputs  # noqa: E402

DEGREES = [(2, 2), (3, 6), (5, 5), (6, 6), (13, 13), (7, 15), (37, 37)]


def lats(p):
    return [1, p // 2] if p < 30 else [p // 2]


def drop(p, axis):
    """Shape coefficients of a deformed sphere, 2^-20 times as thin along the axis, and two densities: without the
    axis's component, and with that one alone."""
    rng = np.random.default_rng(10 * p + axis)
    x = (inputs.sphere_coef(p) + inputs.perturbation(rng, p, 1, min(p, 5), 0.05)).reshape(3, -1).copy()
    x[axis] *= 2.0 ** -20
    dens = inputs.random_bandlimited(rng, p, 3)
    across, along = dens.copy(), np.zeros_like(dens)
    across[axis] = 0
    along[axis] = dens[axis]
    return x, [across, along]


def work(job):
    p, pq, axis = job
    x, dens = drop(p, axis)
    return f"p{p}_pq{pq}_axis{axis}", extended.self_rule(x, p, pq, dens, lats(p)).astype(np.float64)


def main():
    assert np.finfo(np.longdouble).nmant >= 63, "needs an extended-precision longdouble"
    jobs = [(p, pq, axis) for p, pq in sorted(DEGREES, reverse=True) for axis in range(3)]
    with ProcessPoolExecutor() as ex:
        np.savez(os.path.join(HERE, "self_thin.npz"), **dict(ex.map(work, jobs)))


if __name__ == "__main__":
    main()
