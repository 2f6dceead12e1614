"""The FP64 hop's fixed-point form where it could lose precision or leave its
range: neighbours of very different size (the unit changes along the eight
directions), zeros, values it hands to the FP64 form (very small, very large,
NaN), links it does not cover, and the shapes of its thread groups."""

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

# FP64 sums of 8 x 12 products: 2^-53 per operation on both sides, a factor of
# ten above sqrt(96) 1.1e-16, relative to the largest neighbour
TOL = 1e-14


def _handle(dims, Ls, U, nrhs=1):
    h = G.Handle(dims, Ls, G.Action(1.8, 0.01, 1.0, 0.0), nrhs_max=nrhs)
    h.set_gauge(torch.from_numpy(np.ascontiguousarray(U).reshape(-1)).cuda())
    return h


def _hop(h, psi, dims, dagger):
    """Dh on even sites as an oracle array (odd sites zero)."""
    src = torch.view_as_real(torch.from_numpy(LY.to_cb([psi], dims, None, 1))).cuda().contiguous()
    out = h.empty_cb(0, len(psi))
    h.hop(out, src, 0, dagger=dagger, nrhs=len(psi))
    torch.cuda.synchronize()
    cb = torch.view_as_complex(out.cpu().contiguous()).numpy()
    return LY.from_cb(cb, dims, None, 0, psi[0].shape[4])[0]


def _check(U, psi, got, dagger):
    for f, g in zip(psi, got):
        f = O.parity_part(f, 1)
        want = O.parity_part(O.hop(U, f, dagger), 0)
        size = np.abs(f).max(axis=(-1, -2))                    # per site and s
        near = np.max([np.roll(size, s, axis=a) for a in range(4) for s in (1, -1)], axis=0)
        err = np.abs(g - want).max(axis=(-1, -2))
        links = max(1.0, np.abs(U).max())
        assert (err <= TOL * links * near).all(), float((err / np.maximum(near, 1e-300)).max())


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("dims,Ls,nrhs,span", [((4, 4, 4, 4), 8, 1, 0), ((2, 2, 2, 2), 2, 1, 6), ((6, 4, 2, 4), 12, 1, 12),
                                               ((4, 2, 6, 4), 16, 1, 3), ((4, 4, 2, 2), 6, 5, 12),
                                               ((2, 4, 2, 2), 32, 8, 2),
                                               # above the small-domain kernel's line
                                               ((8, 8, 8, 8), 16, 1, 3), ((8, 6, 8, 10), 12, 1, 6),
                                               ((8, 4, 4, 8), 12, 3, 2), ((4, 4, 4, 4), 32, 8, 1)])
def test_uneven_neighbours(dims, Ls, nrhs, span, dagger):
    rng = np.random.default_rng(5)
    U = inputs.gauge_field(dims, "haar", rng=rng)
    psi = [inputs.gaussian_source(dims, Ls, rng=rng) for _ in range(nrhs)]
    for f in psi:   # sites differ by up to 10^span, a tenth of them is zero
        f *= 10.0 ** rng.uniform(-span, span, f.shape[:4])[..., None, None, None]
        f[rng.random(f.shape[:4]) < 0.1] = 0.0
    h = _handle(dims, Ls, U, nrhs)
    _check(U, psi, _hop(h, psi, dims, dagger), dagger)


@pytest.mark.parametrize("scale", [1e-290, 1e-270, 1e15, 1e18, 1e290])
def test_ends_of_the_range(scale):
    dims, Ls = (4, 4, 2, 4), 8
    rng = np.random.default_rng(6)
    U = inputs.gauge_field(dims, "exp", rng=rng)
    psi = [inputs.gaussian_source(dims, Ls, rng=rng) * scale]
    _check(U, psi, _hop(_handle(dims, Ls, U), psi, dims, False), False)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_stays_with_its_neighbours(bad):
    dims, Ls = (4, 4, 4, 4), 8
    rng = np.random.default_rng(7)
    U = inputs.gauge_field(dims, "haar", rng=rng)
    psi = O.parity_part(inputs.gaussian_source(dims, Ls, rng=rng), 1)
    psi[1, 2, 3, 1, 5, 2, 1] = bad        # t, z, y, x odd; lane s = 5
    got = _hop(_handle(dims, Ls, U), [psi], dims, False)[0]
    hit = np.zeros(psi.shape[:5], bool)
    hit[1, 2, 3, 1, 5] = True
    near = np.any([np.roll(hit, s, axis=a) for a in range(4) for s in (1, -1)], axis=0)
    finite = np.isfinite(got).all(axis=(-1, -2))
    assert (finite == ~near).all()
    psi[1, 2, 3, 1, 5] = 0.0
    want = O.parity_part(O.hop(U, psi, False), 0)
    assert np.abs(got - want)[~near].max() <= TOL * np.abs(psi).max()


def test_links_of_other_sizes():
    """Links a few times larger than SU(3), then links too uneven for a common
    unit (the FP64 form), then SU(3) again, on one handle."""
    dims, Ls = (4, 4, 2, 4), 12
    rng = np.random.default_rng(8)
    U0 = inputs.gauge_field(dims, "haar", rng=rng)
    psi = [inputs.gaussian_source(dims, Ls, rng=rng)]
    h = _handle(dims, Ls, U0)
    uneven = U0.copy()
    uneven[..., 1, :, :] *= 1e-9
    for U in (6.5 * U0, uneven, U0):
        h.set_gauge(torch.from_numpy(np.ascontiguousarray(U).reshape(-1)).cuda())
        _check(U, psi, _hop(h, psi, dims, True), True)


def test_links_whose_low_word_is_the_lowest():
    """Imaginary parts (2 m + 1) 2^-30: a fixed-point low word of exactly -2^31,
    whose negative is not a 32-bit number."""
    dims, Ls = (4, 4, 2, 4), 8
    rng = np.random.default_rng(9)
    U = inputs.gauge_field(dims, "exp", rng=rng)
    m = rng.integers(-2 ** 27, 2 ** 27, U.shape)
    U = 0.9 * U.real + 1j * np.ldexp(2.0 * m + 1.0, -30)
    psi = [inputs.gaussian_source(dims, Ls, rng=rng)]
    _check(U, psi, _hop(_handle(dims, Ls, U), psi, dims, False), False)


@pytest.mark.parametrize("dims,nrhs,inner", [((6, 6, 6, 6), 4, G.FP64), ((12, 8, 8, 12), 16, G.FP32)])
def test_solves_with_lanes_in_chunks(dims, nrhs, inner):
    """Many right-hand sides go through the hop in chunks of 32 lanes, each with
    its own part of the per-tile norms: every system of a batched solve (Ls = 16)
    reaches its tolerance, and the first equals its solve alone."""
    Ls, tol = 16, 1e-11
    rng = np.random.default_rng(10)
    U = torch.from_numpy(inputs.gauge_field(dims, "exp", rng=rng).reshape(-1)).cuda()
    act = G.Action(1.8, 0.05, 1.5, 0.5)
    h, h1 = G.Handle(dims, Ls, act, nrhs_max=nrhs), G.Handle(dims, Ls, act)
    h.set_gauge(U)
    h1.set_gauge(U)
    b = torch.randn(h.full_shape(nrhs), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(11))
    x = torch.zeros_like(b)
    stats, rc = h.cgne_solve(x, b, nrhs=nrhs, tol=tol, inner=inner)
    assert rc == 0 and all(st["true_resid"] <= tol for st in stats)
    b1 = b[:, :, :1].contiguous()
    x1 = torch.zeros_like(b1)
    h1.cgne_solve(x1, b1, tol=tol, inner=inner)
    # both within tol of the residual: the condition of D (below 1e2 here) times tol, doubled
    assert float((x[:, :, :1] - x1).norm() / x1.norm()) <= 2e2 * tol
