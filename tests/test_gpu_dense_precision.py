"""Precision of the V-cycle matrix of the smallest levels under an fp32 cycle.

A handle whose finest level is in the matrix (at most 1,024 DoFs) and whose
V-cycle is fp32, against the same handle in fp64, on a right-hand side that is
exact in fp32.  The set-up is fp64 in both, so the matrix is the same and the two
results may differ by one rounding of the entry to fp32 (2^-24) and by the order
of an fp64 sum of at most 1,024 products (1e-13 of the largest entry).
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(synth.cube_octant(1, 0), 4), (synth.cube_octant(2, 1), 2), (synth.octant(3), 1), (synth.sphere(4), 1)]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_matrix_keeps_fp64_under_an_fp32_cycle(gcmg, i):
    recipe, k = CASES[i]
    m = gcmg.Mesh.from_recipe(recipe)
    lo, hi = gcmg.Multigrid(m, k, mg_fp32=True), gcmg.Multigrid(m, k, mg_fp32=False)
    n = hi.n_free(hi.finest)
    assert 0 < n <= 1024
    b = torch.randn(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5)).double()
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    lo.vcycle(b, x)
    hi.vcycle(b, y)
    assert bool(((x - y).abs() <= 2.0 ** -24 * y.abs() + 1e-13 * y.abs().max()).all())
