"""A handle on a GPU with too little memory left for the fixed-point link
table (1152 bytes a site): it is created all the same, and its FP64 hop runs
the FP64 form."""

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2203_17119_gb300 import dwf as G  # noqa: E402


def test_created_without_the_table():
    dims, Ls, sites = (32, 32, 32, 16), 2, 32 ** 3 * 16
    table = 1152 * sites

    def handle():
        return G.Handle(dims, Ls, G.Action(1.8, 0.01))

    g = torch.Generator(device="cuda").manual_seed(8)
    U = 0.2 * torch.randn(sites * 4 * 9, dtype=torch.complex128, device="cuda", generator=g)   # (any links serve)
    h = handle()
    h.set_gauge(U)
    src = h.empty_cb(1)
    src.normal_(generator=g)
    want, out = h.empty_cb(0), h.empty_cb(0)
    h.hop(want, src, 0)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h2 = handle()
    torch.cuda.synchronize()
    need = before - torch.cuda.mem_get_info()[0]
    h2.close()
    torch.cuda.empty_cache()
    assert need > 1.5 * table
    held = torch.empty(torch.cuda.mem_get_info()[0] - (need - table // 2), dtype=torch.uint8, device="cuda")
    h2 = handle()
    del held
    torch.cuda.empty_cache()
    h2.set_gauge(U)
    h2.hop(out, src, 0)
    # both forms within 16 2^-53 of sums of 8 x 12 products that make up numbers of this size
    assert float((out - want).abs().max()) <= 16 * 2.0 ** -53 * 100 * float(want.abs().max())
    assert not torch.equal(out, want)
