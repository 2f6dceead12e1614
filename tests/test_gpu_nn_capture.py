"""New weights of K while other threads and streams are at work: a change of
weights neither waits for unrelated streams nor disturbs a graph that another
thread captures, and waits for replays of a graph that applies K."""

import threading

import pytest

from oracle import dwf as O
from paper_2203_17119_gb300 import inputs
from tests import test_gpu_nn as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DIMS, LS = (4, 4, 2, 4), 6


def _setup(seed):
    rng, U, h = T.setup(DIMS, LS, 1, seed)
    r, e = (T.odd_gpu([O.parity_part(inputs.gaussian_source(DIMS, LS, rng=rng), 1)], DIMS) for _ in range(2))
    return rng, h, r, e


def test_training_beside_a_capture():
    rng, h, r, e = _setup(18)
    w = T.rand_weights(rng)
    nets = [T.G.NN(), T.G.NN()]
    for K in nets:
        K.set_weights(*w)
        K.apply(h, torch.empty_like(r), r)
        K.train_step(h, r, e, lr=1e-3)
    want = nets[0].train_step(h, r, e, lr=1e-3)
    got, failed = [], []
    own = torch.cuda.Stream()

    def train():
        try:
            got.append(nets[1].train_step(h, r, e, lr=1e-3, stream=own))
        except Exception as err:   # noqa: BLE001: reported by the assertion below
            failed.append(err)

    x = torch.ones(1000, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        x.mul_(2.0)
        t = threading.Thread(target=train)
        t.start()
        t.join()
    assert not failed and got == [want]
    graph.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 2000.0
    assert all((a == b).all() for a, b in zip(nets[0].get_weights(), nets[1].get_weights()))


def test_unrelated_stream_is_not_waited_for():
    rng, h, r, e = _setup(19)
    K = T.G.NN()
    K.set_weights(*T.rand_weights(rng))
    K.train_step(h, r, e, lr=1e-3)
    side, own, done = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(2_000_000_000)   # about a second; the step takes some milliseconds
        done.record()
    K.train_step(h, r, e, lr=1e-3, stream=own)
    assert not done.query()
    torch.cuda.synchronize()


def test_replayed_application():
    rng, h, r, e = _setup(20)
    K = T.G.NN()
    K.set_weights(*T.rand_weights(rng))
    want, out = torch.empty_like(r), torch.empty_like(r)
    K.apply(h, want, r)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        K.apply(h, out, r, stream=torch.cuda.current_stream())
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)
        graph.replay()
    K.set_weights(*T.rand_weights(rng))
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def test_more_streams_than_events():
    rng, h, r, e = _setup(21)
    K = T.G.NN()
    K.set_weights(*T.rand_weights(rng))
    want, outs = torch.empty_like(r), [torch.empty_like(r) for _ in range(3)]
    K.apply(h, want, r)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1, -2) for _ in range(32)]   # distinct handles
    assert len({s.cuda_stream for s in streams}) > 64
    for s in streams:
        K.apply(h, outs[0], r, stream=s)
        s.synchronize()
    for i, s in enumerate(streams[-3:]):
        outs[i].zero_()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            torch.cuda._sleep(50_000_000)
            if i:
                s.wait_stream(streams[-3 + i - 1])   # one workspace: one after the other
            K.apply(h, outs[i], r, stream=s)
    K.set_weights(*T.rand_weights(rng))
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for o in outs)
