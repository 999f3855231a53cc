"""Device memory of the library beside other work: a buffer goes back to the pool only after everything on the
device that may still use it has ended, whatever the other threads do meanwhile, graph captures included."""
import ctypes
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import layer
from paper_1707_02156_gb300 import inputs

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12
P, UP = 8, 2


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_02156_gb300 import api, build
    build.build()
    return api


@pytest.fixture(scope="module")
def case():
    w = inputs.two_drops(p=P, gap=0.5, up=UP, lam=0.5)
    nc = 3 * (P + 1) ** 2
    split = lambda v: [v[:nc].reshape(3, -1), v[nc:].reshape(3, -1)]
    drops = layer.Drops(split(w.xcoef), w.p, w.pq, w.lam, up=UP)
    ref = np.concatenate([v.ravel() for v in drops.apply_double(split(w.density))])
    return w, ref, drops


def relerr(a, b):
    a, b = np.asarray(a).ravel(), np.asarray(b).ravel()
    return max(np.linalg.norm(a - b) / np.linalg.norm(b), np.max(np.abs(a - b)) / np.max(np.abs(b)))


class Worker(threading.Thread):
    """Runs fn on a stream of its own and keeps what it raises."""

    def __init__(self, fn):
        super().__init__()
        self.fn, self.error, self.stream = fn, None, torch.cuda.Stream()

    def run(self):
        try:
            with torch.cuda.stream(self.stream):
                self.fn(self.stream)
        except BaseException as e:  # noqa: BLE001
            self.error = e


def run_all(workers):
    for t in workers:
        t.start()
    for t in workers:
        t.join()
    for t in workers:
        if t.error is not None:
            raise t.error


def tensors(w):
    x, f = torch.as_tensor(w.xcoef).cuda(), torch.as_tensor(w.density).cuda()
    return x, f, torch.full_like(f, float("nan"))


def test_close_waits_for_the_work_that_uses_the_geometry(api, case):
    w, ref, _ = case
    ctx = api.Context(0, upsample=UP)
    x, f, out = tensors(w)
    torch.cuda.synchronize()
    geo = ctx.geometry(w.p, w.pq, x, w.lam)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)  # about 50 ms
        geo.apply_double(f, out, precision=0)
    geo.close()
    assert side.query()
    assert relerr(out.cpu().numpy(), ref) < FP64_TOL
    ctx.close()


def open_geometry(api, ctx, w, x, f, out):
    geo = ctx.geometry(w.p, w.pq, x, w.lam)
    for _ in range(3):  # lazy allocations, capture, replay
        geo.apply_double(f, out, precision=0)
    out.fill_(float("nan"))
    torch.cuda.synchronize()
    return geo


def check_next_geometry(ctx, w, x, f, out, ref):
    geo = ctx.geometry(w.p, w.pq, x, w.lam)
    for _ in range(3):
        out.fill_(float("nan"))
        geo.apply_double(f, out, precision=0)
        assert relerr(out.cpu().numpy(), ref) < FP64_TOL
    geo.close()


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
def test_release_beside_another_threads_capture(api, case, mode):
    # the main thread captures while another one uses and closes a geometry, and makes and closes the next
    w, ref, _ = case
    ctx = api.Context(0, upsample=UP)
    x, f, out = tensors(w)
    a = torch.ones(1000, device="cuda")
    b = torch.zeros_like(a)
    geo = open_geometry(api, ctx, w, x, f, out)
    got = []

    def work(stream):
        torch.cuda._sleep(20_000_000)
        geo.apply_double(f, out, precision=0)
        geo.close()
        assert stream.query()
        ctx2 = api.Context(0, upsample=UP)
        geo2 = ctx2.geometry(w.p, w.pq, x, w.lam)
        geo2.apply_double(f, out, precision=0)
        geo2.close()
        ctx2.close()
        got.append(out)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode=mode):
        b.copy_(a)
        run_all([Worker(work)])
        b.add_(a)
    graph.replay()
    torch.cuda.synchronize()
    assert float(b.sum()) == 2000.0
    assert relerr(got[0].cpu().numpy(), ref) < FP64_TOL
    check_next_geometry(ctx, w, x, f, out, ref)
    ctx.close()


def test_close_while_a_capture_forbids_the_wait(api, case):
    # in the capture mode "global" no thread may free memory: the buffers are held, and come back later
    w, ref, _ = case
    ctx = api.Context(0, upsample=UP)
    x, f, out = tensors(w)
    geo = open_geometry(api, ctx, w, x, f, out)
    cudart = ctypes.CDLL("libcudart.so.13")
    other, graph = torch.cuda.Stream(), ctypes.c_void_p()
    assert cudart.cudaStreamBeginCapture(ctypes.c_void_p(other.cuda_stream), 0) == 0
    try:
        def work(stream):
            torch.cuda._sleep(20_000_000)
            geo.apply_double(f, out, precision=0)
            geo.close()
        t = Worker(work)
        run_all([t])
    finally:
        cudart.cudaStreamEndCapture(ctypes.c_void_p(other.cuda_stream), ctypes.byref(graph))
        if graph.value:
            cudart.cudaGraphDestroy(graph)
        cudart.cudaGetLastError()
    t.stream.synchronize()
    assert relerr(out.cpu().numpy(), ref) < FP64_TOL
    check_next_geometry(ctx, w, x, f, out, ref)
    ctx.close()


def test_threads_capture_and_release_beside_one_another(api, case):
    # every geometry's second apply is a capture, its third a replay, and its end a release
    w, ref, _ = case
    got = [[] for _ in range(3)]

    def work(k):
        def fn(stream):
            x, f, out = tensors(w)
            ctx = api.Context(0, upsample=UP)
            for _ in range(6):
                geo = ctx.geometry(w.p, w.pq, x, w.lam)
                for _ in range(4):
                    out.fill_(float("nan"))
                    geo.apply_double(f, out, precision=0)
                    stream.synchronize()
                    got[k].append(out.cpu().numpy())
                if k == 0:  # the steps of a solve are captures, too
                    u = torch.zeros_like(f)
                    info = geo.solve(f, u, precision=0, tol=1e-12)
                    assert info["converged"]
                    A = torch.full_like(f, float("nan"))
                    geo.apply_double(u, A, precision=0)
                    stream.synchronize()
                    lam = np.repeat(np.asarray(w.lam), f.numel() // 2)
                    un = u.cpu().numpy()
                    r = (lam + 1) * un - A.cpu().numpy() - w.density
                    assert np.linalg.norm(r) < 1e-11 * np.linalg.norm(w.density)
                geo.close()
            ctx.close()
        return fn

    run_all([Worker(work(k)) for k in range(3)])
    for g in got:
        assert len(g) == 24
        for v in g:
            assert relerr(v, ref) < FP64_TOL


def test_threads_with_different_degrees(api):
    # the kernels of the three threads take different amounts of shared memory above the default
    ps = [26, 40, 54]
    shapes = [inputs.perturbed_drop(p=p, pq=p, lam=3.0, nmax=6) for p in ps]

    def run(w, n):
        got = []
        ctx = api.Context(0)
        x, f, out = tensors(w)
        for _ in range(n):
            geo = ctx.geometry(w.p, w.pq, x, w.lam)
            for prec in (0, 1, 2):
                out.fill_(float("nan"))
                geo.apply_double(f, out, precision=prec)
                got.append(out.cpu().numpy())
            geo.close()
        ctx.close()
        return got

    ref = [run(w, 1) for w in shapes]
    got = [None] * len(ps)

    def work(k):
        def fn(stream):
            got[k] = run(shapes[k], 8)
        return fn

    run_all([Worker(work(k)) for k in range(len(ps))])
    for r, g in zip(ref, got):
        for i, v in enumerate(g):
            assert np.array_equal(v, r[i % 3])


def test_near_contact_applies_on_a_full_device(api):
    # 12 contacts of 8 drops: the near rule's rows would take 82 MB, more than the device has left after the set-up.
    # Rows and check-point sums are the same sum in another order; the bar is its rounding (some 2^-53 a term), which
    # the interpolation amplifies by up to 1.9e3
    code = """
import numpy as np, torch
from paper_1707_02156_gb300 import api, inputs
p, d = 32, 2.05
xs = [inputs.sphere_coef(p, centre=(d * (k & 1), d * (k >> 1 & 1), d * (k >> 2))) for k in range(8)]
rng = np.random.default_rng(3)
x = torch.as_tensor(inputs.pack_drops(xs)).cuda()
f = torch.as_tensor(inputs.pack_drops([inputs.random_bandlimited(rng, p, 3) for _ in xs])).cuda()
lam = [0.5] * 8
out = torch.empty_like(f)
ctx = api.Context(0)

def applies(geo):
    got = []
    for fn in (geo.apply_single, geo.apply_double):
        for prec in (0, 0, 0, 1, 1):
            out.fill_(float("nan"))
            fn(f, out, precision=prec)
            got.append(out.cpu().numpy())
    return got

geo = ctx.geometry([p] * 8, [p] * 8, x, lam)
assert geo.info["near_targets"] * 7 * (p + 1) ** 2 * 8 > 80e6, geo.info
ref = applies(geo)
geo.close()
geo = ctx.geometry([p] * 8, [p] * 8, x, lam)
fill = []

def fill_up(leave):
    torch.cuda.synchronize()
    n = torch.cuda.mem_get_info()[0] - leave
    if n > 4 << 20:
        fill.append(torch.empty(n >> 21 << 21, dtype=torch.uint8, device="cuda"))

spare = torch.empty(40 << 20, dtype=torch.uint8, device="cuda")
fill_up(60 << 20)
kept = []  # what the library keeps for the next geometry goes to small ones, until no room for the smallest is left
for q in (32, 20, 12, 6):
    try:
        while True:
            kept.append(ctx.geometry([q], [q], torch.as_tensor(inputs.sphere_coef(q).ravel()).cuda(), [0.5]))
    except api.BIEError as e:
        assert e.status == 2, e
del spare
torch.cuda.empty_cache()
assert torch.cuda.mem_get_info()[0] < 75e6, torch.cuda.mem_get_info()
got = applies(geo)
for k, (a, b) in enumerate(zip(got, ref)):
    e = np.linalg.norm(a - b) / np.linalg.norm(b)
    assert e < 1e-11, (k, e)
for g in [geo] + kept:
    g.close()
ctx.close()
print(len(kept), "ok")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=180,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), r.stdout + r.stderr
