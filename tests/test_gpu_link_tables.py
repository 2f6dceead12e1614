"""Loading a gauge field: two launches, and only the links inside the domain
count for its tables -- what lies outside a box, or crosses a cut, may be of
any size, or not a number."""

import numpy as np
import pytest

from oracle import dwf as O
from paper_2203_17119_gb300 import inputs
from tests import layout as LY
from tests import test_gpu_hop_fx as FX

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2203_17119_gb300 import dwf as G  # noqa: E402

DIMS, LS = (6, 4, 4, 6), 8
BOXES = [((1, 0, 2, 3), (3, 4, 2, 5)), ((4, 1, 0, 0), (2, 2, 2, 3))]


def _inside(U, boxes):
    """Links whose ends lie in the same box (of `boxes`), per box."""
    out = []
    for b in boxes:
        m = O.box_mask(DIMS, b)
        out.append(np.stack([m & np.roll(m, -1, axis=O.AXIS[mu]) for mu in range(4)], axis=-1))
    return out


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("outside", [1e-9, 1e200, np.nan])
def test_boxes(outside, dagger):
    rng = np.random.default_rng(21)
    U0 = inputs.gauge_field(DIMS, "haar", rng=rng)
    keep = np.any(_inside(U0, BOXES), axis=0)
    U = np.where(keep[..., None, None], U0, outside * U0)
    masks = [O.box_mask(DIMS, b) for b in BOXES]
    psi = [[O.restrict(inputs.gaussian_source(DIMS, LS, rng=rng), m)] for m in masks]
    h = G.Handle(DIMS, LS, G.Action(1.8, 0.01), boxes=BOXES)
    n0 = G.launch_count()
    h.set_gauge(torch.from_numpy(np.ascontiguousarray(U).reshape(-1)).cuda())
    assert G.launch_count() - n0 == 2
    src = torch.view_as_real(torch.from_numpy(LY.to_cb(psi, DIMS, BOXES, 1))).cuda().contiguous()
    out = h.empty_cb(0)
    h.hop(out, src, 0, dagger=dagger)
    got = LY.from_cb(torch.view_as_complex(out.cpu().contiguous()).numpy(), DIMS, BOXES, 0, LS)
    for g, p, m, inside in zip(got, psi, masks, _inside(U0, BOXES)):
        Ub = np.where(inside[..., None, None], U0, 0.0)
        want = O.restrict(O.parity_part(O.hop(Ub, O.parity_part(p[0], 1), dagger), 0), m)
        assert np.abs(g[0] - want).max() <= FX.TOL * np.abs(p[0]).max()


def test_cut():
    rng = np.random.default_rng(22)
    U0 = inputs.gauge_field(DIMS, "haar", rng=rng)
    cut = [BOXES[0]]
    Uc = O.cut_gauge(U0, cut)
    crossing = (np.abs(Uc).max(axis=(-1, -2)) == 0)[..., None, None]
    assert crossing.any()
    psi = inputs.gaussian_source(DIMS, LS, rng=rng)
    h = G.Handle(DIMS, LS, G.Action(1.8, 0.01), cut=cut)
    h.set_gauge(torch.from_numpy(np.where(crossing, 1e200 * U0, U0).reshape(-1)).cuda())
    got = FX._hop(h, [psi], DIMS, False)[0]
    want = O.parity_part(O.hop(Uc, O.parity_part(psi, 1)), 0)
    assert np.abs(got - want).max() <= FX.TOL * np.abs(psi).max()
