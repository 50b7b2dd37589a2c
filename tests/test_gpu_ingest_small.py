"""Windows of at most 8,192 events are sorted by one block: counts around a
block's and the limit's edges, with malformed events, on one plane and two,
against the oracle (and against the three-launch sort just beyond the limit)."""
import numpy as np
import pytest

import oracle as O
from synth import make_window

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2209_13168_gb300 as dd  # noqa: E402


@pytest.mark.parametrize("polarity", [0, 1])
@pytest.mark.parametrize("n", [0, 1, 1023, 1024, 1025, 8191, 8192, 8193])
def test_counts_around_the_edges(n, polarity):
    w = make_window(330, 250, 165.0, 125.0, n - n // 3, max(1, n // 50), n // 3, 0.3, 0.4, seed=8000 + n)
    win = O.Window.of(w, polarity=bool(polarity))
    ctx = dd.Context(330, 250, 165.0, 125.0, polarity=polarity)
    ev = dd.Events.of(w, device="cuda", polarity=bool(polarity))
    for _ in range(2):
        K, S, N, img = ctx.contrast(ev, np.array([-0.5, 0.3], np.float32), want_iwe=True)
        for j, D in enumerate((-0.5, 0.3)):
            k, s, c, im = O.contrast(win, float(np.float32(D)), want_iwe=True)
            assert (K[j], int(S[j]), int(N[j])) == (k, s, c)
            assert np.array_equal(img[j], im)
        K, _, _, _ = ctx.bound(ev, np.array([0.1], np.float32), np.array([0.6], np.float32))
        assert K[0] == O.bound(win, float(np.float32(0.1)), float(np.float32(0.6)))[0]
    ctx.close()


@pytest.mark.parametrize("field,value", [("x", 330), ("y", -1), ("t", np.nan), ("t", 0.5)])
def test_malformed_events_are_reported(field, value):
    w = make_window(330, 250, 165.0, 125.0, 2000, 60, 500, 0.3, 0.4, seed=8100)
    good = dd.Events.of(w, device="cuda")
    a = getattr(w, field).copy()
    a[1777] = value
    setattr(w, field, a)
    ctx, fresh = (dd.Context(330, 250, 165.0, 125.0, pop_k=8) for _ in range(2))
    calls = (lambda c, e: c.contrast(e, [0.1])[0], lambda c, e: c.bound(e, [0.1], [0.4])[0],
             lambda c, e: c.solve(e, -1.0, 1.0, 1e-2))
    want = [call(fresh, good) for call in calls]
    for bad in calls:
        with pytest.raises(dd.DDError) as e:
            bad(ctx, dd.Events.of(w, device="cuda"))
        assert e.value.status == dd.DD_ERR_ARG
        assert [call(ctx, good) for call in calls] == want        # the next calls on the context are unaffected
    fresh.close()
    ctx.close()
