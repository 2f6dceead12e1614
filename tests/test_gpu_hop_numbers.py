"""Every number of the FP64 hop to FP64's own precision, in both of its
kernels: where components differ in size and links or projectors keep them
apart, a number may not lose precision to a larger one that does not reach it.
And what the fixed-point form hands to the FP64 form, above the line of the
small-domain kernel."""

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
from tests import test_gpu_hop_fx as FX  # noqa: E402

# Against S, the sum of the moduli of a number's terms W_ab (P psi)_b (|z| = |re| + |im|):
# the FP64 form rounds each term at most 16 times by 2^-53.  The fixed-point
# form is off by 2.8 of its units in each of eight directions (2^-2 for each of
# six low-word products, 1/2 for the rounded high word, 0.1 for the links, 0.7
# for the half spinor) and by 2 from changes of the unit, and is kept only where S is at
# least 1.25 2^52 units: 39 2^-53 S; three more roundings to FP64.
TOL = 42 * 2.0 ** -53

SMALL = ((4, 4, 2, 4), 8, 1)          # one warp per direction
MAIN = [((8, 8, 6, 8), 16, 1), ((8, 8, 8, 8), 12, 1), ((6, 6, 6, 8), 12, 2)]
LONG = np.clongdouble


def _terms(U, psi, dagger):
    """Sum of |W_ab|_1 |(P psi)_b|_1 over directions and colours."""
    g, _ = O.gammas()
    one = np.eye(4)
    m1 = lambda z: np.abs(z.real) + np.abs(z.imag)  # noqa: E731
    out = np.zeros(psi.shape)
    for mu in range(4):
        ax = O.AXIS[mu]
        for s in (1, -1):
            P = one - (s if not dagger else -s) * g[mu]
            W = U[..., mu, :, :] if s > 0 else np.conj(np.swapaxes(np.roll(U[..., mu, :, :], 1, axis=ax), -1, -2))
            h = np.einsum("ij,tzyxsja->tzyxsia", P, np.roll(psi, -s, axis=ax))
            out += np.einsum("tzyxab,tzyxsib->tzyxsia", m1(W), m1(h))
    return out


def _field(kind, dims, Ls, rng):
    psi = inputs.gaussian_source(dims, Ls, rng=rng)
    U = inputs.gauge_field(dims, "haar", rng=rng)
    if kind == "colours":            # unit links do not mix them
        U = np.broadcast_to(np.eye(3, dtype=complex), U.shape).copy()
        psi[..., 1] *= 1e-10
        psi[..., 2] *= 1e-17
    elif kind == "eigenvectors":     # large sites that the projector of one direction annihilates
        g, _ = O.gammas()
        big = rng.random(psi.shape[:4]) < 0.06
        for mu in range(4):
            for s in (1, -1):
                pick = big & (rng.random(big.shape) < 0.25)
                psi[pick] = 1e9 * np.einsum("ij,nsja->nsia", np.eye(4) + s * g[mu], psi[pick])
                big &= ~pick
        psi[big] *= 1e9
    elif kind == "components":
        psi *= 10.0 ** rng.uniform(-6, 6, psi.shape)
    return U, psi


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("kind", ["plain", "colours", "eigenvectors", "components"])
@pytest.mark.parametrize("dims,Ls,nrhs", [SMALL] + MAIN)
def test_each_number(dims, Ls, nrhs, kind, dagger):
    rng = np.random.default_rng(12)
    U, first = _field(kind, dims, Ls, rng)
    psi = [first] + [_field(kind, dims, Ls, rng)[1] for _ in range(nrhs - 1)]
    got = FX._hop(FX._handle(dims, Ls, U, nrhs), psi, dims, dagger)
    for f, g in zip(psi, got):
        f = O.parity_part(f, 1)
        want = O.parity_part(O.hop(U.astype(LONG), f.astype(LONG), dagger), 0)
        S = O.parity_part(_terms(U, f, dagger), 0)
        err = np.maximum(np.abs(g.real - want.real), np.abs(g.imag - want.imag)).astype(float)
        assert (err <= TOL * S).all(), float((err / np.maximum(S, 1e-300)).max())


@pytest.mark.parametrize("dims,Ls,nrhs", MAIN)
@pytest.mark.parametrize("scale", [1e-290, 1e-270, 1e15, 1e18])
def test_ends_of_the_range(dims, Ls, nrhs, scale):
    rng = np.random.default_rng(13)
    U = inputs.gauge_field(dims, "exp", rng=rng)
    psi = [inputs.gaussian_source(dims, Ls, rng=rng) * scale for _ in range(nrhs)]
    FX._check(U, psi, FX._hop(FX._handle(dims, Ls, U, nrhs), psi, dims, False), False)


@pytest.mark.parametrize("dims,Ls,nrhs", MAIN)
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e20])
def test_lanes_of_the_fp64_form_among_others(dims, Ls, nrhs, bad):
    """NaN, infinity or a number above the range on a few lanes, reached from
    every direction: D (whose M_oo part shares lanes by shuffles) is
    unaffected off their neighbours and s-neighbours."""
    rng = np.random.default_rng(14)
    prm = O.DWFParams(M5=1.8, mf=0.01)
    U = inputs.gauge_field(dims, "haar", rng=rng)
    psi = [inputs.gaussian_source(dims, Ls, rng=rng) for _ in range(nrhs)]
    hit = [rng.random(f.shape[:5]) < 3e-4 for f in psi]
    for f, b in zip(psi, hit):
        assert b.any()
        f[b, 2, 1] = bad
    h = FX._handle(dims, Ls, U, nrhs)
    src = torch.view_as_real(torch.from_numpy(LY.to_full([psi], dims, None))).cuda().contiguous()
    out = torch.empty_like(src)
    h.apply_d(out, src, nrhs=nrhs)
    got = LY.from_full(torch.view_as_complex(out.cpu()).numpy(), dims, None, Ls)[0]
    for f, b, g in zip(psi, hit, got):
        near = np.any([np.roll(b, s, axis=a) for a in range(4) for s in (1, -1)], axis=0)
        own = b | np.roll(b, 1, axis=4) | np.roll(b, -1, axis=4)   # M_ee: lanes s, s +- 1
        far = ~(near | own)
        finite = np.isfinite(g).all(axis=(-1, -2))
        assert finite[far].all()
        if not np.isfinite(bad):
            assert not finite[near].any()
        clean = np.where(b[..., None, None], 0.0, f)
        want = O.apply_D(U, clean, prm)
        assert np.abs(g - want)[far].max() <= FX.TOL * np.abs(clean).max()
        if np.isfinite(bad):
            want = O.apply_D(U, f, prm)
            assert np.abs(g - want).max() <= FX.TOL * bad


@pytest.mark.parametrize("dims,Ls,nrhs", MAIN)
def test_links_of_other_sizes(dims, Ls, nrhs):
    rng = np.random.default_rng(15)
    U0 = inputs.gauge_field(dims, "haar", rng=rng)
    psi = [inputs.gaussian_source(dims, Ls, rng=rng) for _ in range(nrhs)]
    h = FX._handle(dims, Ls, U0, nrhs)
    uneven = U0.copy()
    uneven[..., 1, :, :] *= 1e-9
    m = rng.integers(-2 ** 27, 2 ** 27, U0.shape)
    lowest = 0.9 * U0.real + 1j * np.ldexp(2.0 * m + 1.0, -30)   # low words of -2^31
    for U in (6.5 * U0, uneven, lowest, U0):
        h.set_gauge(torch.from_numpy(np.ascontiguousarray(U).reshape(-1)).cuda())
        FX._check(U, psi, FX._hop(h, psi, dims, True), True)
