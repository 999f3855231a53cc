"""Calls on a stream that is not ordered with the default stream, while that one is busy: the tables a call uploads
and the counters it clears are in place before its kernels read them."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import layer
from oracle import surfactant as sf
from paper_1707_02156_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_02156_gb300 import api, build
    build.build()
    return api


def relerr(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def test_side_stream_beside_a_busy_default_stream(api):
    p, up = 8, 2
    w = inputs.two_drops(p=p, gap=0.5, up=up, lam=0.5)
    nc = (p + 1) ** 2
    split = lambda v, k: [v[: k * nc].reshape(k, -1), v[k * nc:].reshape(k, -1)]
    xs, fs = split(w.xcoef, 3), split(w.density, 3)
    drops = layer.Drops(xs, w.p, w.pq, w.lam, up=up)
    ref = np.concatenate([v.ravel() for v in drops.apply_double(fs)])
    g = inputs.random_bandlimited(np.random.default_rng(5), p, 2)
    ref_y = np.concatenate([sf.solve_implicit(a, c, p, 0.03)[0].ravel() for a, c in zip(xs, g)])
    x, f, gam = (torch.as_tensor(np.ascontiguousarray(v)).cuda().ravel() for v in (w.xcoef, w.density, g))
    torch.cuda.synchronize()
    stop = threading.Event()

    def busy():  # never more than two short waits queued
        ev = [torch.cuda.Event(), torch.cuda.Event()]
        k = 0
        while not stop.is_set():
            ev[k].synchronize()
            torch.cuda._sleep(500_000)
            ev[k].record()
            k = 1 - k

    t = threading.Thread(target=busy)
    t.start()
    side = torch.cuda.Stream()
    try:
        with torch.cuda.stream(side):
            for _ in range(6):
                ctx = api.Context(0, upsample=up)
                geo = ctx.geometry(w.p, w.pq, x, w.lam)
                out, y, u = torch.full_like(f, float("nan")), torch.full_like(gam, float("nan")), torch.zeros_like(f)
                geo.apply_double(f, out, precision=0)
                api.surfactant_implicit(ctx, w.p, x, gam, 0.03, y)
                info = geo.solve(f, u, precision=0, tol=1e-12)
                back = torch.full_like(f, float("nan"))
                geo.apply_double(u, back, precision=0)
                side.synchronize()
                assert info["converged"]
                assert relerr(out.cpu().numpy(), ref) < 1e-12
                assert relerr(y.cpu().numpy(), ref_y) < 1e-11
                lam = np.repeat(np.asarray(w.lam), 3 * nc)
                assert relerr((lam + 1) * u.cpu().numpy() - back.cpu().numpy(), w.density) < 1e-11
                geo.close()
                ctx.close()
    finally:
        stop.set()
        t.join()
