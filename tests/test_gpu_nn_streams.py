"""New weights while an application of K is still queued on another stream:
the queued one uses the weights it was called with."""

import pytest

from oracle import dwf as O
from paper_2203_17119_gb300 import inputs
from tests import test_gpu_nn as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("how", ["set_weights", "train_step"])
def test_weights_of_the_call(how):
    dims, Ls = (4, 4, 2, 4), 6
    rng, U, h = T.setup(dims, Ls, 1, 17)
    h2 = T.G.Handle(dims, Ls, T.G.Action(1.8, 0.01, 1.5, 0.5))   # its own workspace
    h2.set_gauge(torch.from_numpy(U.reshape(-1)).cuda())
    old, new = T.rand_weights(rng), T.rand_weights(rng)
    K = T.G.NN()
    K.set_weights(*old)
    r, e = (T.odd_gpu([O.parity_part(inputs.gaussian_source(dims, Ls, rng=rng), 1)], dims) for _ in range(2))
    want, out = torch.empty_like(r), torch.empty_like(r)
    K.apply(h, want, r)
    K.train_step(h2, r, e, lr=0.0)            # its workspace exists
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)        # some 50 ms of queued work
        K.apply(h, out, r)
    if how == "set_weights":
        K.set_weights(*new)
    else:
        K.train_step(h2, r, e, lr=1.0)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    K.apply(h, out, r)
    torch.cuda.synchronize()
    assert not torch.equal(out, want)
