"""Both register variants of the lane kernels against the line-parallel kernels.

A level of more tiles than one wave takes the variant with more blocks per SM, a
smaller one or one whose tiles mostly hang the variant with more registers.  Mesh
61,440 cells (1,920 tiles of 32: more than one wave at every degree) and its
coarser levels, a sphere mesh whose tiles mostly hang; domain lengths of a power of
two (a cell's scale is one) and not.  Each path is within 1e-12 (fp64) or 2e-6
(fp32) of the oracle elsewhere, so two of them differ by at most twice that of the
result's norm.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("length", [1.0, 3.0])
@pytest.mark.parametrize("k", [2, 3, 4])
@pytest.mark.parametrize("mesh", ["octant", "sphere"])
def test_register_variants(gcmg, mesh, k, length):
    steps = [(0,)] * 5 + [(1, 0.0, 0.5 * length)] if mesh == "octant" else [(2, 0.5 * length, 0.3 * length)] * 6
    m = gcmg.Mesh(0.0, length, steps)
    ref, new = gcmg.Multigrid(m, k, cell_kernel=1), gcmg.Multigrid(m, k, cell_kernel=3)
    for l in (new.finest, new.finest - 1):
        for dtype, tol in ((torch.float64, 2e-12), (torch.float32, 4e-6)):
            x = torch.randn(new.n_free(l), dtype=dtype, device="cuda",
                            generator=torch.Generator(device="cuda").manual_seed(l))
            a, b = torch.empty_like(x), torch.empty_like(x)
            ref.vmult(l, x, a)
            new.vmult(l, x, b)
            assert float((a - b).double().norm()) <= tol * float(a.double().norm()), (l, dtype)
