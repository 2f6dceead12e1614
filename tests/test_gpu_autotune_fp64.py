"""The FP64 autotuner times the hop at work: a hop over zeros leaves out its
projections and products, so candidates would be ranked by memory traffic."""

import time

import pytest

from paper_2203_17119_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2203_17119_gb300 import dwf as G  # noqa: E402


def _hop_seconds(h, out, src):
    """Fastest of a few hops, host clock around each."""
    best = 1e9
    for _ in range(8):
        torch.cuda.synchronize()
        t = time.perf_counter()
        h.hop(out, src, 0)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


def test_candidates_do_the_work():
    dims, Ls = (24, 24, 16, 16), 16
    h = G.Handle(dims, Ls, G.Action(1.8, 0.01), boxes=[((0, 0, 0, 0), dims)])
    h.set_gauge(torch.from_numpy(inputs.gauge_field(dims, "haar", seed=3).reshape(-1)).cuda())
    src, out = h.empty_cb(1), h.empty_cb(0)
    src.normal_(generator=torch.Generator(device="cuda").manual_seed(4))
    h.hop(out, src, 0)
    want = out.clone()
    h.autotune(1, G.FP64)                 # the tile tables of all candidates
    n0, t = G.launch_count(), time.perf_counter()
    h.autotune(1, G.FP64)
    t, hops = time.perf_counter() - t, G.launch_count() - n0 - 1   # a launch is a hop, but for the input's
    assert h.tuning(1)[0] in (4, 8, 16, 32, 64, 128)
    busy, idle = _hop_seconds(h, out, src), _hop_seconds(h, out, torch.zeros_like(src))
    assert torch.equal(out, torch.zeros_like(out)) and idle < 0.6 * busy
    # the tuned configuration is the fastest of those timed, and each was: more
    # than hops that skip their work would take, flushing L2 between them (0.1 ms)
    assert hops >= 9 and t >= hops * 0.9 * busy
    h.hop(out, src, 0)
    assert torch.equal(out, want)
