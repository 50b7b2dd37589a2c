"""One window's or a few windows' searches in one cooperative launch: a control
block each with the queue in its shared memory while it fits, evaluating blocks that poll for the
next round.  Results, counts and traces are the oracle's whatever the queue's
place (never, sometimes or always in shared memory), and windows beyond the
launch's size limit go through the graph with the same result.
"""
import functools

import pytest

import oracle as O
from synth import make_window
from synth.descent import serve_spec5

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2209_13168_gb300 as dd  # noqa: E402

KEYS = ("D_star", "D_end", "K_hat", "gap_K", "nodes_expanded", "point_evals", "bound_evals", "event_warps",
        "cell_increments", "bound_increments", "rounds", "max_queue")


# 160-pixel frames: dynamic shared memory of the block (bytes) decides how many
# intervals fit: none, a few tens (the queue of this window reaches 98) or all
@pytest.mark.parametrize("threads,band_rows", [(32, 4), (96, 50), (480, 90)])
@pytest.mark.parametrize("pop_k", [1, 16, 64])
def test_queue_in_and_out_of_shared_memory(threads, band_rows, pop_k):
    w = make_window(160, 90, 80.0, 45.0, 16000, 444, 5333, 0.35, 0.3, seed=74)
    want = O.solve(O.Window.of(w), -1.0, 1.0, 1e-4, 0.0, pop_k, trace_cap=4096)
    ctx = dd.Context(160, 90, 80.0, 45.0, pop_k=pop_k, threads=threads, band_rows=band_rows)
    for _ in range(2):
        got = ctx.solve(dd.Events.of(w, device="cuda"), trace_cap=4096)
        for k in KEYS:
            assert got[k] == want[k], (k, got[k], want[k])
        assert got["trace"] == want["trace"]
    ctx.close()


# A wait that runs out ends the launch, and the same searches run through the
# graph: at the first round (one poll) or wherever a round outlasts the polls.
# What the unfinished round left in the sums (of tasks, and of bands split by
# events: 140,000 of them on a wide frame) must not reach the rerun or what
# the context evaluates next.
@pytest.mark.parametrize("polls", [1, 16, 64])
@pytest.mark.parametrize("windows,n", [(1, 3000), (1, 140000), (3, 3000)])
def test_a_wait_that_runs_out(polls, windows, n):
    ws = [make_window(640, 480, 320.0, 240.0, n - n // 4, n // 36, n // 4, 0.35, 0.3, seed=60 + i)
          for i in range(windows)]
    evs = [dd.Events.of(w, device="cuda") for w in ws]
    ctx = dd.Context(640, 480, 320.0, 240.0, pop_k=16)
    ctx.set_wait_limit(polls)
    for _ in range(2):
        ctx.reset_stats()
        rc, got = ctx.solve_batch(evs, [(-1.0, 1.0, 2e-2, 0.0)] * windows)
        assert rc == dd.DD_OK
        if polls == 1:
            assert ctx.stats()["eval_launches"] == 1 + max(r["rounds"] for r in got) + 1   # the root's round too
        for w, r in zip(ws, got):
            want = O.solve(O.Window.of(w), -1.0, 1.0, 2e-2, 0.0, 16)
            for k in KEYS:
                assert r[k] == want[k], (k, r[k], want[k])
        win = O.Window.of(ws[0])
        assert ctx.contrast(evs[0], [0.1, 0.35])[0] == [O.contrast(win, D)[0] for D in (0.1, 0.35)]
        assert ctx.bound(evs[0], [-1.0, 0.3], [1.0, 0.4])[0] == [O.bound(win, a, b)[0] for a, b in ((-1.0, 1.0), (0.3, 0.4))]
    ctx.set_wait_limit(0)
    trace = ctx.solve(evs[0], -1.0, 1.0, 2e-2, 0.0, trace_cap=4096)["trace"]
    ctx.set_wait_limit(polls)
    assert ctx.solve(evs[0], -1.0, 1.0, 2e-2, 0.0, trace_cap=4096)["trace"] == trace
    with pytest.raises(dd.DDError):
        ctx.set_wait_limit(-1)
    ctx.close()


# The one launch takes every SM: searches of two contexts on their own threads
# and streams take turns, and a search takes turns with a server's rounds.
def test_searches_beside_other_work():
    import threading
    ws = [make_window(160, 90, 80.0, 45.0, 4000 + 900 * i, 110, 1300, 0.35, 0.3, seed=75 + i) for i in range(2)]
    want = [O.solve(O.Window.of(w), -1.0, 1.0, 1e-3, 0.0, 8) for w in ws]
    evs = [dd.Events.of(w, device="cuda") for w in ws]
    ctxs = [dd.Context(160, 90, 80.0, 45.0, pop_k=8) for _ in range(3)]
    srv = dd.Server(ctxs[2], max_slots=4, max_events=1 << 13)
    got = [[], [], []]

    def search(i):
        for _ in range(30):
            got[i].append(ctxs[i].solve(evs[i], -1.0, 1.0, 1e-3, 0.0))

    threads = [threading.Thread(target=search, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for _ in range(5):
        tickets = [srv.submit(evs[k % 2], (-1.0, 1.0, 1e-3, 0.0)) for k in range(8)]
        got[2] += [srv.wait(k) for k in tickets]
    for t in threads:
        t.join()
    srv.stop()
    assert [len(g) for g in got] == [30, 30, 40]
    for i in range(3):
        for j, r in enumerate(got[i]):
            for k in KEYS:
                assert r[k] == want[i if i < 2 else j % 2][k], (i, j, k)
    for c in ctxs:
        c.close()


def test_round_and_queue_limits():
    w = make_window(160, 90, 80.0, 45.0, 4000, 110, 1300, 0.35, 0.3, seed=75)
    ev = dd.Events.of(w, device="cuda")
    for kw, status in (({"max_rounds": 5}, dd.DD_ERR_TIMEOUT), ({"queue_capacity": 3}, dd.DD_ERR_QUEUE_OVERFLOW)):
        ctx = dd.Context(160, 90, 80.0, 45.0, pop_k=4, **kw)
        with pytest.raises(dd.DDError) as e:
            ctx.solve(ev)
        assert e.value.status == status
        ctx.close()


def test_window_beyond_the_launch_limit():
    from synth.gpu import make_window_gpu
    n = (1 << 22) + 33
    spec = list(serve_spec5(0, 100))
    spec[4], spec[5], spec[6] = n - n // 8, n // 40, n // 8
    ev = dd.Events.of(make_window_gpu(tuple(spec)))
    got = []
    for kw in ({}, {"host_loop": 1}):
        ctx = dd.Context(1280, 720, 640.0, 360.0, pop_k=16, **kw)
        got.append(ctx.solve(ev, -1.0, 1.0, 1e-2, 0.0))
        ctx.close()
    for k in KEYS:
        assert got[0][k] == got[1][k], k


# one interval a round, so that bands (the default height, one row, a height
# that the slices do not divide, the whole frame) are cut into slices of rows;
# above 131,072 events a long bound's unit (64 cells; the root of the longest
# window here has 157) holds a share of the events and is not cut
@pytest.mark.parametrize("n,tau", [(900, 0.3), (20000, 0.3), (140000, 0.3), (140000, 0.7)])
@pytest.mark.parametrize("band_rows", [0, 1, 13, 97])
def test_bands_cut_into_slices(n, tau, band_rows):
    w, want = _window_to_slice(n, tau)
    ctx = dd.Context(131, 97, 64.0, 50.5, pop_k=1, band_rows=band_rows)
    got = ctx.solve(dd.Events.of(w, device="cuda"), -1.0, 1.0, 1e-3, 0.0)
    ctx.close()
    for k in KEYS:
        assert got[k] == want[k], (k, got[k], want[k])


@functools.lru_cache(maxsize=None)
def _window_to_slice(n, tau):
    w = make_window(131, 97, 64.0, 50.5, n - n // 3, n // 36, n // 3, 0.35, tau, seed=76)
    return w, O.solve(O.Window.of(w), -1.0, 1.0, 1e-3, 0.0, 1)


# up to 16 windows share one launch, 17 go through the graph; they end in
# different rounds, one has a single event
@pytest.mark.parametrize("windows", [2, 3, 16, 17])
@pytest.mark.parametrize("pop_k,threads", [(1, 480), (16, 480), (16, 32)])
def test_a_few_windows_in_one_launch(windows, pop_k, threads):
    ws = [make_window(96, 64, 48.0, 32.0, 300 + 170 * i, 30, 100 + 40 * i, 0.2 + 0.02 * i, 0.3, seed=80 + i)
          for i in range(windows)]
    ws[1].x, ws[1].y, ws[1].t, ws[1].p = ws[1].x[:1], ws[1].y[:1], ws[1].t[:1], ws[1].p[:1]
    evs = [dd.Events.of(w, device="cuda") for w in ws]
    got = {}
    for host_loop in (0, 1):
        ctx = dd.Context(96, 64, 48.0, 32.0, pop_k=pop_k, threads=threads, host_loop=host_loop)
        rc, got[host_loop] = ctx.solve_batch(evs, [(-1.0, 1.0, 1e-3, 0.0)] * windows)
        assert rc == dd.DD_OK
        ctx.close()
    for i, w in enumerate(ws):
        want = O.solve(O.Window.of(w), -1.0, 1.0, 1e-3, 0.0, pop_k)
        for k in KEYS:
            assert got[0][i][k] == got[1][i][k] == want[k], (i, k)


def test_a_few_windows_with_limits():
    ws = [make_window(96, 64, 48.0, 32.0, 900, 40, 300, 0.3, 0.4, seed=90 + i) for i in range(3)]
    evs = [dd.Events.of(w, device="cuda") for w in ws]
    for kw, status in (({"max_rounds": 5}, dd.DD_ERR_TIMEOUT), ({"queue_capacity": 3}, dd.DD_ERR_QUEUE_OVERFLOW)):
        ctx = dd.Context(96, 64, 48.0, 32.0, pop_k=4, **kw)
        rc, out = ctx.solve_batch(evs)
        assert rc == status and all(r["status"] == status for r in out)
        ctx.close()
