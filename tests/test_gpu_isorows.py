"""The isovalue map of strided ensembles of short rows, several rows to a CTA, against the same cells
as one contiguous ensemble, bit for bit: row lengths around the number of threads that share a row,
rows that fill the last CTA only in part, more rows than the grid's y axis has blocks for."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,ld", [(5, 1, 3), (300, 3, 4), (300, 16, 32), (1000, 33, 36), (1001, 32, 32), (77, 129, 131),
                                    (130, 130, 132), (64, 513, 516), (40, 1025, 1028), (9, 2047, 2050),
                                    (5, 4095, 4096), (3, 5000, 5004), (5000000, 2, 3)])
@pytest.mark.parametrize("kind", ["normal", "level"])
def test_short_rows(N, M, ld, kind):
    import torch
    from paper_2512_15187_gb300 import binding, build
    build.build()
    h = binding.Handle(0)
    F = torch.rand((N, ld), device="cuda", generator=torch.Generator("cuda").manual_seed(N))[:, :M]
    want = h.soft_masks(F.contiguous(), 0.5, 0.2, kind=kind)
    out = torch.full((N, ld), -1.0, device="cuda")
    h.soft_masks(F, 0.5, 0.2, kind=kind, out=out)
    b16 = h.soft_masks(F, 0.5, 0.2, kind=kind, dtype=torch.bfloat16)
    h.sync()
    assert torch.equal(out[:, :M], want) and (out[:, M:] == -1.0).all()
    assert torch.equal(b16, want.to(torch.bfloat16))
    h.close()
