"""When the near-singular rule of an apply sums its check points and when it reads operator rows: both against the
FP64 oracle, and the rows built only for a kind that is applied again."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import layer
from paper_1707_02156_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 5e-6, 2: 1e-11}
P, UP = 8, 3


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_02156_gb300 import api, build
    build.build()
    return api


@pytest.fixture(scope="module")
def case():
    w = inputs.two_drops(p=P, gap=0.05, up=UP, lam=0.5)
    nc = 3 * (P + 1) ** 2
    split = lambda v: [v[:nc].reshape(3, -1), v[nc:].reshape(3, -1)]
    drops = layer.Drops(split(w.xcoef), w.p, w.pq, w.lam, up=UP)
    fs = split(w.density)
    ref = [np.concatenate([v.ravel() for v in fn(fs)]) for fn in (drops.apply_single, drops.apply_double)]
    return w, ref


def relerr(a, b):
    return max(np.linalg.norm(a - b) / np.linalg.norm(b), np.max(np.abs(a - b)) / np.max(np.abs(b)))


def held(api, geo):
    info = api.bie_geom_info()
    assert api.lib().bie_geometry_info(geo.h, ctypes.byref(info)) == 0
    return info.cache_bytes


def rows_bytes(geo):
    return geo.info["near_targets"] * 7 * (((P + 1) ** 2 + 3) & ~3) * 8


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("graphs", [False, True])
def test_rows_from_the_second_apply(api, case, prec, graphs):
    w, ref = case
    ctx = api.Context(0, upsample=UP, use_graphs=graphs)
    x, f = torch.as_tensor(w.xcoef).cuda(), torch.as_tensor(w.density).cuda()
    out = torch.empty_like(f)
    geo = ctx.geometry(w.p, w.pq, x, w.lam)
    base = held(api, geo)
    assert rows_bytes(geo) > 0
    for kind, fn in enumerate((geo.apply_single, geo.apply_double)):
        for k in range(4):
            out.fill_(float("nan"))
            fn(f, out, precision=prec)
            assert held(api, geo) == base + (kind + (k > 0)) * rows_bytes(geo)
            assert relerr(out.cpu().numpy(), ref[kind]) < TOL[prec], (kind, k)
    geo.close()
    ctx.close()


def test_solve_builds_the_double_layers_rows(api, case):
    w, ref = case
    ctx = api.Context(0, upsample=UP)
    x, f = torch.as_tensor(w.xcoef).cuda(), torch.as_tensor(w.density).cuda()
    geo = ctx.geometry(w.p, w.pq, x, w.lam)
    base = held(api, geo)
    b, u, out = torch.empty_like(f), torch.zeros_like(f), torch.empty_like(f)
    geo.rhs(torch.zeros_like(f), f, b, precision=2)
    assert held(api, geo) == base
    assert relerr(b.cpu().numpy(), ref[0]) < TOL[2]
    assert geo.solve(b, u, precision=1, tol=1e-10)["converged"]
    assert held(api, geo) == base + rows_bytes(geo)
    geo.apply_double(u, out, precision=0)
    lam = np.repeat(np.asarray(w.lam), f.numel() // 2)
    r = (lam + 1) * u.cpu().numpy() - out.cpu().numpy() - b.cpu().numpy()
    assert np.linalg.norm(r) < 1e-9 * np.linalg.norm(b.cpu().numpy())
    geo.close()
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_callers_capture_after_one_eager_apply(api, case, prec):
    # nothing may allocate or synchronise in the capture: it takes the check sums, as the eager apply did
    w, ref = case
    ctx = api.Context(0, upsample=UP, use_graphs=False)
    x, f = torch.as_tensor(w.xcoef).cuda(), torch.as_tensor(w.density).cuda()
    out = torch.empty_like(f)
    geo = ctx.geometry(w.p, w.pq, x, w.lam)
    base = held(api, geo)
    geo.apply_double(f, out, precision=prec)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        geo.apply_double(f, out, precision=prec)
    assert held(api, geo) == base
    for k in range(2):
        out.fill_(float("nan"))
        graph.replay()
        assert relerr(out.cpu().numpy(), ref[1]) < TOL[prec]
    geo.apply_double(f, out, precision=prec)  # eager again: the rows, beside the captured check sums
    assert held(api, geo) == base + rows_bytes(geo)
    assert relerr(out.cpu().numpy(), ref[1]) < TOL[prec]
    out.fill_(float("nan"))
    graph.replay()
    assert relerr(out.cpu().numpy(), ref[1]) < TOL[prec]
    geo.close()
    ctx.close()
