"""(d + e S5)^-1 where |e| > |d| (Moebius coefficients with c5 well above b5):
the recurrence in a = -e / d grows like |a|^Ls there, so what it leaves of the
result after the wall term depends on its direction.  Against the closed form
of the oracle, whose entries do not cancel."""

import numpy as np
import pytest

from oracle import dwf as O
from paper_2203_17119_gb300 import inputs
from tests import layout as LY

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2203_17119_gb300 import dwf as G  # noqa: E402

DIMS = (4, 4, 2, 4)
# sums of up to 32 terms in FP32, 32 x 2^-24; BF16 results are rounded to 2^-9,
# and M_pc rounds its intermediate fields too
TOL = {G.FP32: 2e-6, G.BF16: 4e-3}
TOL_MPC = {G.FP32: 4e-6, G.BF16: 1.5e-2}
# (b5, c5, mf): |a| = 1.75, 2.14, 1.75 without a wall, 1.02, and 0.32 for comparison
ACTIONS = [(1.0, 3.0, 0.01), (0.5, 2.5, 0.01), (1.0, 3.0, 0.0), (1.0, 1.93, 0.3), (1.5, 0.5, 0.01)]


def _setup(Ls, b5, c5, mf, nrhs=1):
    rng = np.random.default_rng(41)
    U = inputs.gauge_field(DIMS, "exp", rng=rng)
    h = G.Handle(DIMS, Ls, G.Action(1.8, mf, b5, c5), nrhs_max=nrhs)
    h.set_gauge(torch.from_numpy(U.reshape(-1)).cuda())
    psi = [O.parity_part(inputs.gaussian_source(DIMS, Ls, rng=rng), 1) for _ in range(nrhs)]
    return U, h, psi, O.DWFParams(M5=1.8, mf=mf, b5=b5, c5=c5)


def _dev(psi, prec):
    """The odd field on the GPU, and the values it has there."""
    t = torch.view_as_real(torch.from_numpy(LY.to_cb([psi], DIMS, None, 1))).cuda().to(G._DTYPE[prec]).contiguous()
    return t, LY.from_cb(_host(t), DIMS, None, 1, psi[0].shape[4])[0]


def _host(t):
    return torch.view_as_complex(t.double().cpu().contiguous()).numpy()


@pytest.mark.parametrize("prec", [G.FP32, G.BF16])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("Ls,nrhs", [(2, 1), (10, 2), (24, 1), (32, 1), (32, 2)])
@pytest.mark.parametrize("b5,c5,mf", ACTIONS)
def test_inverse(b5, c5, mf, Ls, nrhs, dagger, prec):
    U, h, psi, prm = _setup(Ls, b5, c5, mf, nrhs)
    src, vals = _dev(psi, prec)
    out = torch.empty_like(src)
    h.mooee_inv(out, src, 1, dagger, prec, nrhs)
    got = LY.from_cb(_host(out), DIMS, None, 1, Ls)[0]
    for g, v in zip(got, vals):
        assert LY.rel_l2(g, O.mooee_inv(v, prm, dagger)) <= TOL[prec]


@pytest.mark.parametrize("prec", [G.FP32, G.BF16])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("Ls", [24, 32])
def test_schur_operator(Ls, dagger, prec):
    U, h, psi, prm = _setup(Ls, 1.0, 3.0, 0.01)
    src, vals = _dev(psi, prec)
    out = torch.empty_like(src)
    h.mpc(out, src, dagger, prec)
    got = LY.from_cb(_host(out), DIMS, None, 1, Ls)[0][0]
    assert LY.rel_l2(got, O.mpc(U, vals[0], prm, dagger)) <= TOL_MPC[prec]


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("Ls,nrhs", [(2, 1), (10, 2), (24, 1), (32, 2)])
@pytest.mark.parametrize("b5,c5,mf", ACTIONS)
def test_inverse_fp64(b5, c5, mf, Ls, nrhs, dagger):
    U, h, psi, prm = _setup(Ls, b5, c5, mf, nrhs)
    src, vals = _dev(psi, G.FP64)
    out = torch.empty_like(src)
    h.mooee_inv(out, src, 1, dagger, G.FP64, nrhs)
    got = LY.from_cb(_host(out), DIMS, None, 1, Ls)[0]
    for g, v in zip(got, vals):   # sums of up to 32 terms, a few roundings of 2^-53 each, on both sides
        assert LY.rel_l2(g, O.mooee_inv(v, prm, dagger)) <= 128 * 2.0 ** -53


@pytest.mark.parametrize("prec", [G.FP32, G.BF16])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("Ls", [16, 32])
def test_schur_operator_with_fusion_chosen(Ls, dagger, prec):
    U, h, psi, prm = _setup(Ls, 0.5, 2.5, 0.01)
    h.set_fusion(1, True)
    src, vals = _dev(psi, prec)
    out = torch.empty_like(src)
    h.mpc(out, src, dagger, prec)
    got = LY.from_cb(_host(out), DIMS, None, 1, Ls)[0][0]
    assert LY.rel_l2(got, O.mpc(U, vals[0], prm, dagger)) <= TOL_MPC[prec]
