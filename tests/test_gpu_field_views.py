"""Fields that are views into a larger buffer, aligned to one complex number
(the site-local operators) or to two BF16 ones (those with a hop), give what
aligned copies give."""

import pytest

from paper_2203_17119_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2203_17119_gb300 import dwf as G  # noqa: E402

DIMS = (4, 4, 2, 6)


def _view(t, offset):
    """A copy of t that starts `offset` complex numbers into its buffer (256-byte aligned)."""
    buf = torch.empty(t.numel() + 2 * offset, dtype=t.dtype, device="cuda")
    v = buf[2 * offset:].view(t.shape)
    v.copy_(t)
    assert v.is_contiguous() and v.data_ptr() % 16 == (2 * offset * t.element_size()) % 16
    return v


def _close(got, want, prec):
    # the same sums by other groups of lanes: FP32 rounding 2^-24 over up to 32 terms; one BF16 rounding 2^-8
    tol = 2e-6 if prec == G.FP32 else 2.0 ** -8
    return float((got.double() - want.double()).abs().max()) <= tol * float(want.double().abs().max())


@pytest.mark.parametrize("prec,offset", [(G.FP32, 1), (G.BF16, 1), (G.BF16, 2), (G.BF16, 3)])
@pytest.mark.parametrize("Ls,nrhs", [(2, 1), (6, 3), (8, 1), (12, 2), (32, 1)])
def test_site_local(Ls, nrhs, prec, offset):
    h = G.Handle(DIMS, Ls, G.Action(1.8, 0.01, 1.5, 0.5), nrhs_max=nrhs)
    h.set_gauge(torch.from_numpy(inputs.gauge_field(DIMS, "exp", seed=5).reshape(-1)).cuda())
    src = h.empty_cb(1, nrhs, prec)
    src.normal_(generator=torch.Generator(device="cuda").manual_seed(6))
    for op in (h.mooee, h.mooee_inv):
        want = torch.empty_like(src)
        op(want, src, 1, False, prec, nrhs)
        for o, i in ((0, offset), (offset, 0), (offset, offset)):
            out, inp = _view(torch.zeros_like(src), o), _view(src, i)
            op(out, inp, 1, False, prec, nrhs)
            assert _close(out, want, prec), (op.__name__, o, i)


@pytest.mark.parametrize("Ls,nrhs", [(6, 3), (8, 1), (12, 1), (16, 1)])
def test_bf16_operators(Ls, nrhs):
    h = G.Handle(DIMS, Ls, G.Action(1.8, 0.01, 1.5, 0.5), nrhs_max=nrhs)
    h.set_gauge(torch.from_numpy(inputs.gauge_field(DIMS, "exp", seed=5).reshape(-1)).cuda())
    src = h.empty_cb(1, nrhs, G.BF16)
    src.normal_(generator=torch.Generator(device="cuda").manual_seed(6))
    for dagger in (False, True):
        want, eo = torch.empty_like(src), h.empty_cb(0, nrhs, G.BF16)
        h.mpc(want, src, dagger, G.BF16, nrhs)
        h.dslash_eo(eo, src, 0, dagger, G.BF16, nrhs)
        inp, out, out_eo = _view(src, 2), _view(torch.zeros_like(src), 2), _view(torch.zeros_like(eo), 2)
        h.mpc(out, inp, dagger, G.BF16, nrhs)
        h.dslash_eo(out_eo, inp, 0, dagger, G.BF16, nrhs)
        # M_pc rounds four intermediate fields to BF16
        assert float((out.double() - want.double()).norm() / want.double().norm()) <= 4 * 2.0 ** -8
        assert float((out_eo.double() - eo.double()).norm() / eo.double().norm()) <= 4 * 2.0 ** -8
