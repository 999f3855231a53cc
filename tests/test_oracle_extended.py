"""The extended-precision self rule: equal to the FP64 oracle up to that one's rounding, and the stored values of the
thin drops reproduced."""
import os
import sys

import numpy as np
import pytest

from oracle import extended, layer
from paper_1707_02156_gb300 import inputs

sys.path.insert(0, os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden"))
import make_self_thin as thin  # noqa: E402


def test_extended_rule_equals_the_oracle():
    p, pq, lats = 4, 6, [0, 2]
    rng = np.random.default_rng(4)
    x = inputs.sphere_coef(p, centre=(0.3, -0.2, 0.1)) + inputs.perturbation(rng, p, 1, 3, 0.1)
    f = inputs.random_bandlimited(rng, p, 3)
    q = layer.SelfQuadrature(x, p, pq)
    got = extended.self_rule(x, p, pq, [f], lats)
    for k, kind in enumerate("SD"):
        ref = q.apply(f, kind, lats=lats)[:, lats, :]
        assert np.linalg.norm((got[k, 0] - ref).astype(float)) < 1e-13 * np.linalg.norm(ref)


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="longdouble is no wider than FP64 here")
def test_stored_thin_values():
    z = np.load(os.path.join(os.path.dirname(thin.__file__), "self_thin.npz"))
    assert sorted(z.files) == sorted(f"p{p}_pq{pq}_axis{a}" for p, pq in thin.DEGREES for a in range(3))
    for axis in range(3):
        x, dens = thin.drop(3, axis)
        got = extended.self_rule(x, 3, 6, dens, thin.lats(3))
        ref = z[f"p3_pq6_axis{axis}"]
        for c in range(3):
            assert np.linalg.norm((got[:, :, c] - ref[:, :, c]).astype(float)) < 1e-15 * np.linalg.norm(ref[:, :, c])
