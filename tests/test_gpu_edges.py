"""GPU parity at the sizes where the kernels' folds, paddings and splits have their edges.

The transforms fold latitude pairs (a middle latitude exists for an even degree P) and longitude
quadruples (a middle longitude exists for an odd P), and a block takes more or fewer latitude pairs and
orders with the number of fields; the dense self factors pad (p+1)^2 to whole 16-byte loads; the rows of
the near-singular rule fold the standard and the upsampled grid.  Every parity and remainder is
compared with the FP64 oracle at the bars of the other parity tests."""
import math
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import layer, sh
from oracle import surfactant as sf
from paper_1707_02156_gb300 import inputs

pytestmark = pytest.mark.gpu

FP64_TOL, MIXED_TOL, DF_TOL = 1e-12, 2e-6, 1e-11


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_02156_gb300 import api, build
    build.build()
    return api


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def relerr(a, b):
    a, b = np.asarray(a).ravel(), np.asarray(b).ravel()
    return max(np.linalg.norm(a - b) / np.linalg.norm(b), np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("p, P", [(1, 1), (1, 2), (2, 2), (2, 5), (3, 4), (6, 7), (16, 31), (48, 48), (49, 49), (64, 64), (5, 129)])
@pytest.mark.parametrize("ndrop", [1, 40])
def test_transforms_at_every_grid_parity(api, p, P, ndrop):
    rng = np.random.default_rng(100 * p + P)
    coefs = [inputs.random_bandlimited(rng, p, 3, decay_pow=0.5) for _ in range(2)]
    ctx = api.Context(0)
    c = dev(np.concatenate([coefs[d % 2].ravel() for d in range(ndrop)]))
    g = torch.full((ndrop, 3, (P + 1) * (2 * P + 2)), float("nan"), dtype=torch.float64, device="cuda")
    ctx.sh_synthesize([p] * ndrop, [P] * ndrop, 3, c, g)
    gh = host(g)
    for d in {0, ndrop - 1}:
        for k in range(3):
            assert relerr(gh[d, k], sh.synthesize(coefs[d % 2][k], p, P)) < FP64_TOL
    if p == P:
        back = torch.full_like(c, float("nan"))
        ctx.sh_analyze([p] * ndrop, 3, g, back)
        assert relerr(host(back), host(c)) < FP64_TOL
    ctx.close()


@pytest.mark.parametrize("p, double", [(1, False), (1, True), (2, False), (3, True), (4, False), (7, False), (10, True)])
def test_dense_self_term_at_every_row_padding(api, p, double):
    w = inputs.perturbed_drop(p=p, pq=None if double else p, lam=3.0, nmax=min(p, 6))
    ctx = api.Context(0)
    geo = ctx.geometry(w.p, w.pq, dev(w.xcoef), w.lam)
    drops = layer.Drops([w.xcoef.reshape(3, -1)], w.p, w.pq, w.lam)
    f = dev(w.density)
    out = torch.zeros_like(f)
    for fn, ref in ((geo.apply_single, drops.apply_single), (geo.apply_double, drops.apply_double)):
        r = ref([w.density])[0]
        for prec, tol in ((0, FP64_TOL), (1, MIXED_TOL), (2, DF_TOL)):
            fn(f, out, precision=prec)
            assert relerr(host(out), r) < tol, (prec,)
    geo.close()
    ctx.close()


@pytest.mark.parametrize("p, pq, scale, shift", [(5, 5, 1e-9, 0.0), (6, 13, 1e9, 3e9), (36, 36, 1.0, 0.0), (37, 37, 1.0, 7.0),
                                                  (62, 62, 1.0, 0.0), (63, 63, 1.0, 0.0)])
def test_self_setup_over_sizes_and_scales(api, p, pq, scale, shift):
    # the rotated-grid set-up takes two latitude pairs per pass up to degree 36, one up to 62 and goes through
    # memory above; its fixed-point sums scale with the drop and leave its position out
    w = inputs.perturbed_drop(p=p, pq=pq, lam=3.0, nmax=min(p, 6))
    x = w.xcoef.reshape(3, -1) * scale
    x[:, 0] += shift
    ctx = api.Context(0)
    geo = ctx.geometry(w.p, w.pq, dev(x), w.lam)
    q = layer.SelfQuadrature(x, p, pq)
    lats = [0, p // 2, p] if p < 60 else [p // 2]
    f = dev(w.density)
    out = torch.zeros(3 * (p + 1) * (2 * p + 2), dtype=torch.float64, device="cuda")
    for kind, fn, wt in (("S", geo.apply_single, -1 / (4 * math.pi)), ("D", geo.apply_double, 2 / (4 * math.pi))):
        ref = wt * q.apply(w.density, kind, lats=lats)
        fn(f, out, precision=0, grid_out=True)
        g = host(out).reshape(3, p + 1, 2 * p + 2)
        assert relerr(g[:, lats, :], ref[:, lats, :]) < FP64_TOL, (kind,)
    geo.close()
    ctx.close()


@pytest.mark.parametrize("p, up", [(6, 2), (7, 3), (8, 1), (9, 4)])
def test_near_rows_at_every_grid_parity(api, p, up):
    w = inputs.two_drops(p=p, gap=0.05, up=up, lam=0.5)
    nc = 3 * (p + 1) ** 2
    xs = [w.xcoef[:nc].reshape(3, -1), w.xcoef[nc:].reshape(3, -1)]
    fs = [w.density[:nc].reshape(3, -1), w.density[nc:].reshape(3, -1)]
    drops = layer.Drops(xs, w.p, w.pq, w.lam, up=up)
    ctx = api.Context(0, upsample=up)
    geo = ctx.geometry(w.p, w.pq, dev(w.xcoef), w.lam)
    assert geo.info["near_targets"] == sum(int(np.sum(r == 2)) for r in drops.region.values()) > 0
    f = dev(w.density)
    out = torch.zeros_like(f)
    for fn, ref in ((geo.apply_single, drops.apply_single), (geo.apply_double, drops.apply_double)):
        r = np.concatenate([v.ravel() for v in ref(fs)])
        for prec, tol in ((0, FP64_TOL), (1, 5e-6)):
            for _ in range(3):  # the rows are built by the first apply, the third one is a graph replay
                out.fill_(float("nan"))
                fn(f, out, precision=prec)
                assert relerr(host(out), r) < tol, (prec,)
    geo.close()
    ctx.close()


def test_more_degree_groups_than_a_launch_takes(api):
    # transforms of several degrees share a launch, eight syntheses (two grids per degree for sources) at a time
    ps = [11, 2, 9, 4, 7, 6, 5, 8, 3, 10, 4]
    rng = np.random.default_rng(21)
    xs = [inputs.sphere_coef(p, centre=(4.0 * (i % 4), 4.0 * (i // 4), 0.3 * i)) + inputs.perturbation(rng, p, 2, min(p, 4), 0.05)
          for i, p in enumerate(ps)]
    fs = [inputs.random_bandlimited(rng, p, 3) for p in ps]
    gs = [inputs.random_bandlimited(rng, p, 1)[0] * 0.1 for p in ps]
    lam = np.linspace(0.3, 4.0, len(ps))
    ctx = api.Context(0)
    x, f, g = dev(inputs.pack_drops(xs)), dev(inputs.pack_drops(fs)), dev(np.concatenate(gs))
    geo = ctx.geometry(ps, ps, x, lam)
    drops = layer.Drops([v.reshape(3, -1) for v in xs], ps, ps, lam)
    out = torch.full_like(f, float("nan"))
    for fn, ref in ((geo.apply_single, drops.apply_single), (geo.apply_double, drops.apply_double)):
        fn(f, out, precision=0)
        assert relerr(host(out), np.concatenate([v.ravel() for v in ref(fs)])) < FP64_TOL
    fe, fi, y = torch.full_like(g, float("nan")), torch.full_like(g, float("nan")), torch.full_like(g, float("nan"))
    api.surfactant_rates(ctx, ps, x, f, g, 0.25, fe, fi)
    assert relerr(host(fe), np.concatenate([sf.f_explicit(a, u, c, p) for a, u, c, p in zip(xs, fs, gs, ps)])) < 1e-12
    assert relerr(host(fi), np.concatenate([sf.f_implicit(a, c, p, 4.0) for a, c, p in zip(xs, gs, ps)])) < 1e-12
    api.surfactant_implicit(ctx, ps, x, g, 0.03, y)
    assert relerr(host(y), np.concatenate([sf.solve_implicit(a, c, p, 0.03)[0] for a, c, p in zip(xs, gs, ps)])) < 1e-11
    geo.close()
    ctx.close()


def test_buffers_of_several_threads_and_their_return(api):
    # contexts on threads of their own draw on one memory pool of the device; with the last one gone it is empty
    w = inputs.two_drops(p=8, gap=0.5, up=2, lam=0.5)
    got = [[] for _ in range(3)]

    def work(mine):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            ctx = api.Context(0, upsample=2)
            for _ in range(4):
                geo = ctx.geometry(w.p, w.pq, dev(w.xcoef), w.lam)
                f = dev(w.density)
                out = torch.full_like(f, float("nan"))
                geo.apply_double(f, out, precision=0)
                stream.synchronize()
                mine.append(out.cpu().numpy())
                geo.close()
            ctx.close()

    threads = [threading.Thread(target=work, args=(g,)) for g in got]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    nc = 3 * 81
    xs = [w.xcoef[:nc].reshape(3, -1), w.xcoef[nc:].reshape(3, -1)]
    fs = [w.density[:nc].reshape(3, -1), w.density[nc:].reshape(3, -1)]
    ref = np.concatenate([v.ravel() for v in layer.Drops(xs, w.p, w.pq, w.lam, up=2).apply_double(fs)])
    for g in got:
        assert len(g) == 4
        for v in g:
            assert relerr(v, ref) < FP64_TOL
    # in a process of its own: contexts of other tests may still hold the pool here
    code = """
import torch
from paper_1707_02156_gb300 import api, inputs
free = lambda: (torch.cuda.synchronize(), torch.cuda.mem_get_info()[0])[1]
def run(n, p):
    w = inputs.deformed_drops(n, p, box=8.0)
    x = torch.as_tensor(w.xcoef).cuda()
    ctx = api.Context(0)
    geo = ctx.geometry(w.p, w.pq, x, w.lam)
    f = free()
    geo.close()
    ctx.close()
    return f
run(2, 4)
before = free()
used = before - run(8, 20)
assert used > 200e6 and before - free() < used / 4, (used, before - free())
"""
    subprocess.run([sys.executable, "-c", code], check=True, timeout=120, cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
