"""The mixed kernels' parts (N = 1,024, N = 512, N <= 256) chained in one call:
a candidate's results do not depend on what else the call holds, so every
window must get the same bits alone as beside windows of the other parts.
Candidate counts give items of one, an odd number and the most candidates."""
import numpy as np
import pytest
import torch

from paper_2307_03763_gb300 import api
from paper_2307_03763_gb300 import workloads as wk

from tests.test_gpu_tchannel import _c, _problem

pytestmark = pytest.mark.gpu

SPECS = [(16e-3, 1024), (4e-3, 256), (11e-3, 512), (2e-3, 128), (15e-3, 1024), (1e-3, 64), (0.4e-3, 32), (9e-3, 512)]


@pytest.mark.parametrize("name", ["loglik", "loglik_aet", "loglik_phase", "loglik_phase_aet", "loglik_grad",
                                  "loglik_grad_aet"])
@pytest.mark.parametrize("n", [1, 33, 1500, 6001])
def test_parts_do_not_interact(name, n):
    ctx = api.Context(wk.YEAR)
    wins, th, data, weights = _problem(n, SPECS, n)
    d, w, th = [_c(x, torch.complex128) for x in data], [_c(x, torch.float64) for x in weights], _c(th, torch.float64)
    if not name.endswith("_aet"):
        d, w = d[:2], w[:2]
    call = getattr(ctx, name)
    joint = [x.clone() for x in call(wins, *d, *w, th, prec="mixed")]
    for k0, W, N, off, coff, m in wins:
        rows, bins = slice(coff, coff + m), slice(off, off + W)
        alone = call([(k0, W, N, 0, 0, m)], *[x[bins].clone() for x in d], *[x[bins].clone() for x in w],
                     th[rows].clone(), prec="mixed")
        for a, b in zip(joint, alone):
            assert torch.isfinite(b).all() and torch.equal(a[rows], b)


NAMES = ["loglik_aet", "loglik_phase", "loglik_grad", "loglik_grad_aet"]


def _args(name, n, seed):
    wins, th, data, weights = _problem(seed, SPECS, n)
    d, w = [_c(x, torch.complex128) for x in data], [_c(x, torch.float64) for x in weights]
    if not name.endswith("_aet"):
        d, w = d[:2], w[:2]
    return wins, d, w, _c(th, torch.float64)


@pytest.mark.parametrize("name", ["loglik"] + NAMES)
@pytest.mark.parametrize("n", [5, 2000])
def test_parts_read_this_calls_data(name, n):
    """One layout, other data and weights in each call, eager and replayed:
    every part must see what the call's own preparation wrote, not the floats
    that the call before left."""
    ctx = api.Context(wk.YEAR)
    sets = [_args(name, n, seed) for seed in (n, n + 1, n + 2)]
    wins, d, w, th = sets[0]
    ref = [[x.clone() for x in getattr(api.Context(wk.YEAR), name)(wins, *s[1], *s[2], th, prec="mixed")] for s in sets]
    assert not torch.equal(ref[0][0], ref[1][0])
    call = getattr(ctx, name)
    for k in (0, 1, 2, 1, 0):
        for a, b in zip(call(wins, *sets[k][1], *sets[k][2], th, prec="mixed"), ref[k]):
            assert torch.equal(a, b)
    buf = [x.clone() for x in (*d, *w)]
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        call(wins, *buf, th, prec="mixed")
        stream.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            out = call(wins, *buf, th, prec="mixed")
        for k in (0, 1, 2, 1, 0):
            for x, y in zip(buf, (*sets[k][1], *sets[k][2])):
                x.copy_(y)
            graph.replay()
            for a, b in zip(out, ref[k]):
                assert torch.equal(a, b)
    stream.synchronize()


@pytest.mark.parametrize("name", ["loglik"] + NAMES)
def test_time_budget_and_events_over_all_parts(name):
    """A budget that is not used up, kernel events around the likelihood, and a
    budget that ends in the middle: the rows that are written are the same bits."""
    wins, d, w, th = _args(name, 12000, 3)
    ctx = api.Context(wk.YEAR)
    call = getattr(ctx, name)
    ref = [x.clone() for x in call(wins, *d, *w, th, prec="mixed")]
    ctx.set_time_budget(10.0)
    for a, b in zip(call(wins, *d, *w, th, prec="mixed"), ref):
        assert torch.equal(a, b)
    ctx.check()
    if "grad" not in name:
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        end.record()
        ctx.set_kernel_events(start, end)
        for a, b in zip(call(wins, *d, *w, th, prec="mixed"), ref):
            assert torch.equal(a, b)
        torch.cuda.synchronize()
        assert start.elapsed_time(end) > 0.0
    for budget in (5e-9, 10e-6, 200e-6):   # the first: warps may end before they take an item
        ctx.set_time_budget(budget)
        got = call(wins, *d, *w, th, prec="mixed")
        try:
            ctx.check()
            full = True
        except api.GBError:
            full = False
        for a, b in zip(got, ref):
            assert torch.equal(a, b) if full else ((a == b) | (a == 0.0)).all()
    ctx.set_time_budget(0.0)
    for a, b in zip(call(wins, *d, *w, th, prec="mixed"), ref):
        assert torch.equal(a, b)
    ctx.check()


@pytest.mark.parametrize("grad", [False, True])
def test_time_budget_leaves_the_preparation_out(grad):
    """A window of four million bins takes the preparation many times as long
    as the kernel takes for its candidates: a budget between the two suffices."""
    n = 200000
    src = wk.source(2e-3, 1e-17, 1e-22, np.random.default_rng(1))
    th = torch.as_tensor(wk.uniform_box(src, np.array([1e-8, 1e-17, 0.1, 0.1, 1e-23, 0.1, 0.1, 0.1]), n,
                                        np.random.default_rng(2)), device="cuda")
    ctx = api.Context(wk.YEAR)

    def problem(W):
        win = [(int(2e-3 * wk.YEAR) - 64, W, 128, 0, 0, n)]
        d, w = torch.zeros(W, dtype=torch.complex128, device="cuda"), torch.ones(W, dtype=torch.float64, device="cuda")
        call = ctx.loglik_grad if grad else ctx.loglik
        return lambda: call(win, d, d, w, w, th, prec="mixed")

    def seconds(f):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        f()
        a.record()
        out = f()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) * 1e-3, [x.clone() for x in out]

    kernel, _ = seconds(problem(128))
    long = problem(1 << 22)
    total, ref = seconds(long)
    assert total > 8 * kernel
    ctx.set_time_budget(total / 4)
    for a, b in zip(long(), ref):
        assert torch.equal(a, b)
    ctx.check()


def test_entry_points_share_a_layouts_fp64_plan():
    """A plan cannot be made while a stream is captured; the likelihood's serves
    the listed rows, the certified round and the Gram matrices of its layout."""
    n = 24000
    wins, d, w, th = _args("loglik", n, 4)
    win, th = wins[1][:4] + (0, n), th[n:2 * n].clone()
    ctx = api.Context(wk.YEAR)
    rows = torch.arange(n, dtype=torch.int32, device="cuda")
    lo, hi = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((1,), 100, dtype=torch.int32, device="cuda")
    zero = torch.zeros((1, n), dtype=torch.float64, device="cuda")
    log_u = torch.log(torch.rand((1, n), dtype=torch.float64, device="cuda"))
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    pairs = [wins[1][:4] + (2 * k, 2) for k in range(n // 2)]
    other = [(win[0] + 1,) + win[1:]]
    ctx.mh_certified(other, *d, *w, th, zero, log_u, one)   # scratch of this size
    for lay in ([win], pairs):
        for prec in ("fp64", "mixed"):
            ctx.loglik(lay, *d, *w, th, prec=prec)
    want = ctx.loglik([win], *d, *w, th)[0][:100].clone()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            got = ctx.loglik_rows([win], *d, *w, th, rows, lo, hi)[0]
            pending = ctx.mh_certified([win], *d, *w, th, zero, log_u, one)[-1]
            rho = ctx.snr_multi(pairs, *d, *w, th)[0]
        graph.replay()
    stream.synchronize()
    assert torch.equal(got[:100], want) and int(pending) == 0
    assert torch.equal(rho, ctx.snr_multi(pairs, *d, *w, th)[0])
