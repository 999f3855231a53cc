"""Precision of the self set-up on drops that are thin along a coordinate axis (tests/golden/self_thin.npz, the
extended-precision rule).

Every component of the shape, and with it every entry of the 3x3 kernel weights, has its own size there (1,
2^-20 and 2^-40 of the largest), and a density along or across the axis brings out one entry at a time.  FP64 keeps each of
them to a few 2^-53 of itself, times the cancellation in x.n and over the surface (about 10^3); the bar is 1e-11 per
component.  One scale for all components would lose 20 or 40 bits."""
import math
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

sys.path.insert(0, os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden"))
import make_self_thin as thin  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_02156_gb300 import api, build
    build.build()
    return api


@pytest.mark.parametrize("p, pq", thin.DEGREES)  # among them one and two latitude pairs a pass in the rotated-grid cache
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_thin_component_keeps_its_precision(api, p, pq, axis):
    raw = np.load(os.path.join(os.path.dirname(thin.__file__), "self_thin.npz"))[f"p{p}_pq{pq}_axis{axis}"]
    x, dens = thin.drop(p, axis)
    ctx = api.Context(0)
    geo = ctx.geometry([p], [pq], torch.as_tensor(x).cuda().ravel(), [3.0])
    out = torch.zeros(3 * (p + 1) * (2 * p + 2), dtype=torch.float64, device="cuda")
    for k, (fn, wt) in enumerate(((geo.apply_single, -1 / (4 * math.pi)), (geo.apply_double, 2 / (4 * math.pi)))):
        for d, density in enumerate(dens):
            fn(torch.as_tensor(density).cuda().ravel(), out, precision=0, grid_out=True)
            got = out.cpu().numpy().reshape(3, p + 1, 2 * p + 2)[:, thin.lats(p), :]
            for c in range(3):
                ref = wt * raw[k, d, c]
                assert np.linalg.norm(got[c] - ref) < TOL * np.linalg.norm(ref), (k, d, c)
    geo.close()
    ctx.close()
