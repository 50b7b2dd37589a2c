"""The evaluation kernel at the sizes its units are cut by: chunks of 32
events, runs of 7 major cells, a warp's list of 320 unstable events, the three
10-bit counts a fused unit keeps in one cell, bands of one row, and the ends of
the search domain -- keys, sums and images against the oracle, exactly.
"""
import numpy as np
import pytest

import oracle as O
from synth import make_window

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2209_13168_gb300 as dd  # noqa: E402

KEYS = ("D_star", "D_end", "K_hat", "gap_K", "nodes_expanded", "point_evals", "bound_evals", "event_warps",
        "cell_increments", "bound_increments", "rounds", "max_queue")


def images_match(w, ctx, Ds, intervals, **kw):
    win = O.Window.of(w, **kw)
    ev = dd.Events.of(w, device="cuda")
    K, S, N, img = ctx.contrast(ev, np.asarray(Ds, np.float32), want_iwe=True)
    for j, D in enumerate(Ds):
        k, s, n, im = O.contrast(win, float(np.float32(D)), want_iwe=True)
        assert (K[j], int(S[j]), int(N[j])) == (k, s, n), D
        assert np.array_equal(img[j], im), D
    lo, hi = np.asarray(intervals, np.float32).T
    K, S, N, img = ctx.bound(ev, lo, hi, want_iwe=True)
    for j in range(len(lo)):
        k, s, n, im = O.bound(win, float(lo[j]), float(hi[j]), want_iwe=True)
        assert (K[j], int(S[j]), int(N[j])) == (k, s, n), (lo[j], hi[j])
        assert np.array_equal(img[j], im), (lo[j], hi[j])


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 480 * 4 - 1, 480 * 4 + 33])
@pytest.mark.parametrize("threads", [32, 480])
def test_chunk_edges(n, threads):
    w = make_window(70, 50, 33.5, 21.0, n - n // 4, max(1, n // 12), n // 4, 0.4, 0.5, seed=6000 + n)
    for rows in (1, 50):
        ctx = dd.Context(70, 50, 33.5, 21.0, threads=threads, band_rows=rows)
        images_match(w, ctx, [-0.9, 0.4], [(-0.9, 0.9), (0.3, 0.31), (0.4, 0.4)])
        ctx.close()


# a call of few points or short bounds divides its bands (the default height,
# one row, a height that the slices do not divide, the whole frame)
@pytest.mark.parametrize("band_rows", [0, 1, 13, 97])
@pytest.mark.parametrize("polarity", [0, 1])
def test_few_tasks_in_slices(band_rows, polarity):
    w = make_window(131, 97, 64.0, 50.5, 6000, 170, 2000, 0.35, 0.3, seed=79)
    ctx = dd.Context(131, 97, 64.0, 50.5, band_rows=band_rows, polarity=polarity)
    win, ev = O.Window.of(w, polarity=bool(polarity)), dd.Events.of(w, device="cuda", polarity=bool(polarity))
    for Ds in ([0.35], [-0.9, 0.0, 0.9]):
        K, S, N, img = ctx.contrast(ev, Ds, want_iwe=True)
        for j, D in enumerate(Ds):
            k, s, n, im = O.contrast(win, D, want_iwe=True)
            assert (K[j], int(S[j]), int(N[j])) == (k, s, n) and np.array_equal(img[j], im), D
    for lo, hi in (([0.35], [0.36]), ([-0.5, 0.3], [-0.49, 0.32])):
        lo, hi = np.asarray(lo, np.float32), np.asarray(hi, np.float32)
        K, S, N, img = ctx.bound(ev, lo, hi, want_iwe=True)
        for j in range(len(lo)):
            k, s, n, im = O.bound(win, float(lo[j]), float(hi[j]), want_iwe=True)
            assert (K[j], int(S[j]), int(N[j])) == (k, s, n) and np.array_equal(img[j], im), (lo[j], hi[j])
    ctx.close()


@pytest.mark.parametrize("foe", [(0.0, 0.0), (160.0, 60.0), (320.0, 119.75)])
def test_segments_of_run_lengths(foe):
    # intervals whose longest segments cover 1, 6-8, 13-15 and over 100 major cells
    w = make_window(320, 120, foe[0], foe[1], 1500, 60, 900, 0.3, 0.4, seed=71)
    ctx = dd.Context(320, 120, foe[0], foe[1], band_rows=17)
    far = max(foe[0], 320 - foe[0], foe[1], 120 - foe[1])
    spans = [c / (far * 0.4) for c in (0.4, 1, 2, 6, 7, 8, 13, 14, 15, 40, 100)]
    images_match(w, ctx, [0.1], [(0.1 - 0.5 * s, 0.1 + 0.5 * s) for s in spans])
    ctx.close()


@pytest.mark.parametrize("to_start", [0, 1])
def test_domain_ends_far_outside_the_frame(to_start):
    # at D tau = -60 a segment from the window's start reaches 60 frames away
    w = make_window(1280, 40, 1280.0, 0.0, 500, 30, 300, 0.3, 0.5, seed=72)
    ctx = dd.Context(1280, 40, 1280.0, 0.0, band_rows=5, warp_to_start=to_start)
    images_match(w, ctx, [-120.0, 1.4], [(-120.0, 0.2), (-120.0, -119.0), (1.2, 1.5)],
                 t_ref=0.0 if to_start else None)
    ctx.close()


def test_more_than_32_bits_of_increments_in_one_warp():
    # n copies of one event whose segment is long although the bound counts as
    # sparse (far from the reference time, at the domain's end), all walked by
    # the one warp of one block: counts grow with n, keys with its square
    n, tau = 21_000_000, 0.5
    x, y, t = np.array([60], np.int16), np.array([0], np.int16), np.array([tau], np.float32)
    one = O.solve(O.Window(4096, 1, 0.0, 0.0, x, y, t, 0.0, tau, t_ref=0.0), -128.0, -121.0, 10.0, 0.0, 1)
    assert one["nodes_expanded"] == 1 and n * one["bound_increments"] > 1 << 32
    ev = dd.Events(*(torch.from_numpy(a).cuda().repeat(n) for a in (x, y, t)), 0.0, tau)
    torch.cuda.synchronize()
    ctx = dd.Context(4096, 1, 0.0, 0.0, threads=32, warp_to_start=1)
    got = ctx.solve(ev, -128.0, -121.0, 10.0, 0.0)
    ctx.close()
    for k in ("bound_increments", "cell_increments"):
        assert got[k] == n * one[k], (k, got[k], n * one[k])
    for k in ("K_hat", "gap_K"):
        assert got[k] == n * n * one[k], k


@pytest.mark.parametrize("hot", [1022, 1023, 1024, 2500])
@pytest.mark.parametrize("threads", [32, 480])
def test_fused_units_with_a_hot_pixel(hot, threads):
    # a pixel that fires `hot` times at one instant fills a fused cell's fields
    w = make_window(96, 64, 48.0, 32.0, 900, 40, 300, 0.3, 0.4, seed=73)
    x = np.concatenate([w.x, np.full(hot, 60, np.int16)])
    y = np.concatenate([w.y, np.full(hot, 41, np.int16)])
    t = np.concatenate([w.t, np.full(hot, 0.2, np.float32)])
    w.x, w.y, w.t, w.p = x, y, t, np.ones(x.size, np.int8)
    want = O.solve(O.Window.of(w), -1.0, 1.0, 1e-3, 0.0, 8, trace_cap=4096)
    ctx = dd.Context(96, 64, 48.0, 32.0, pop_k=8, threads=threads, fuse_span=100)
    got = ctx.solve(dd.Events.of(w, device="cuda"), -1.0, 1.0, 1e-3, 0.0, trace_cap=4096)
    for k in KEYS:
        assert got[k] == want[k], (k, got[k], want[k])
    assert got["trace"] == want["trace"]
    ctx.close()


def test_fused_units_whose_listed_events_overflow():
    # every band holds a pixel of 1,200 events that moves over a border in most
    # intervals: its events are listed (80 a warp) and a field overflows only
    # in the second part of the unit, which the warps reach one by one
    w = make_window(96, 64, 48.0, 32.0, 900, 40, 300, 0.3, 0.4, seed=78)
    rows, hot = np.arange(2, 64, 4), 1200
    x = np.concatenate([w.x, np.full(rows.size * hot, 70, np.int16)])
    y = np.concatenate([w.y, np.repeat(rows, hot).astype(np.int16)])
    t = np.concatenate([w.t, np.full(rows.size * hot, 0.1, np.float32)])
    w.x, w.y, w.t, w.p = x, y, t, np.ones(x.size, np.int8)
    want = O.solve(O.Window.of(w), -1.0, 1.0, 1e-3, 0.0, 16, trace_cap=4096)
    ev = dd.Events.of(w, device="cuda")
    ctx = dd.Context(96, 64, 48.0, 32.0, pop_k=16, band_rows=4, fuse_span=1_000_000)
    for _ in range(20):
        got = ctx.solve(ev, -1.0, 1.0, 1e-3, 0.0, trace_cap=4096)
        for k in KEYS:
            assert got[k] == want[k], (k, got[k], want[k])
        assert got["trace"] == want["trace"]
    ctx.close()


def test_fused_units_with_a_full_list():
    # one warp per block: bands with more than 320 unstable events
    w = make_window(160, 90, 80.0, 45.0, 9000, 250, 3000, 0.35, 0.3, seed=74)
    want = O.solve(O.Window.of(w), -1.0, 1.0, 1e-3, 0.0, 4, trace_cap=4096)
    for threads in (32, 96):
        ctx = dd.Context(160, 90, 80.0, 45.0, pop_k=4, threads=threads, fuse_span=100, band_rows=45)
        got = ctx.solve(dd.Events.of(w, device="cuda"), -1.0, 1.0, 1e-3, 0.0, trace_cap=4096)
        for k in KEYS:
            assert got[k] == want[k], (k, got[k], want[k])
        assert got["trace"] == want["trace"]
        ctx.close()


@pytest.mark.parametrize("n", [(1 << 21) - 512, (1 << 21) + 512])
def test_fused_units_at_the_most_chunks(n):
    # one warp per block and one band: 65,536 chunks are the most whose sums
    # one warp keeps in 32 bits; a unit with more runs its tasks one by one
    w = make_window(256, 90, 128.0, 45.0, 900, 40, 300, 0.3, 0.4, seed=77)
    rng = np.random.default_rng(77)
    w.x, w.y = rng.integers(0, 256, n).astype(np.int16), rng.integers(0, 90, n).astype(np.int16)
    w.t = np.sort(rng.random(n) * 0.3).astype(np.float32)
    w.p = np.ones(n, np.int8)
    want = O.solve(O.Window.of(w), -1e-3, 1e-3, 5e-4, 0.0, 4)
    ctx = dd.Context(256, 90, 128.0, 45.0, pop_k=4, threads=32, fuse_span=100, band_rows=90)
    got = ctx.solve(dd.Events.of(w, device="cuda"), -1e-3, 1e-3, 5e-4, 0.0)
    ctx.close()
    for k in KEYS:
        assert got[k] == want[k], (k, got[k], want[k])
