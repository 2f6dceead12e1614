"""The inference form of K where its odd-site part has walls everywhere (Ls of
2 and 4: the shifts by two lanes), on a Dirichlet box with odd extents, and in
place, against the FP64 oracle."""

import numpy as np
import pytest

from oracle import dwf as O
from oracle import nn as N
from paper_2203_17119_gb300 import inputs
from tests import layout as LY
from tests import test_gpu_nn as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# FP32 rounding 6e-8 through sums of up to 8 x 32 + 80 products on each of two
# levels, with a factor of five
TOL = 5e-6


@pytest.mark.parametrize("dims,Ls,nrhs,boxes", [((2, 2, 2, 2), 2, 1, None), ((4, 2, 2, 4), 4, 3, None),
                                                ((6, 2, 4, 2), 10, 2, None),
                                                ((4, 4, 2, 4), 6, 1, [((0, 1, 0, 1), (3, 2, 2, 3))])])
@pytest.mark.parametrize("in_place", [False, True])
def test_walls_boxes_in_place(dims, Ls, nrhs, boxes, in_place):
    rng = np.random.default_rng(31)
    U = inputs.gauge_field(dims, "haar", rng=rng)
    h = T.G.Handle(dims, Ls, T.G.Action(1.8, 0.01, 1.5, 0.5), boxes=boxes, nrhs_max=nrhs)
    h.set_gauge(torch.from_numpy(U.reshape(-1)).cuda())
    W1, W2 = T.rand_weights(rng)
    K = T.G.NN()
    K.set_weights(W1, W2)
    mask = O.box_mask(dims, boxes[0]) if boxes else np.ones(dims[::-1], bool)
    Uc = O.cut_gauge(U, boxes) if boxes else U
    r = [O.restrict(O.parity_part(inputs.gaussian_source(dims, Ls, rng=rng), 1), mask) for _ in range(nrhs)]
    x = torch.view_as_real(torch.from_numpy(LY.to_cb([r], dims, boxes, 1))).to("cuda", torch.float32).contiguous()
    out = x if in_place else torch.empty_like(x)
    K.apply(h, out, x, nrhs)
    torch.cuda.synchronize()
    got = LY.from_cb(torch.view_as_complex(out.double().cpu().contiguous()).numpy(), dims, boxes, 1, Ls)[0]
    for k in range(nrhs):
        want = O.restrict(N.apply_K(Uc, r[k], W1, W2), mask)
        assert LY.rel_l2(got[k], want) <= TOL, k
