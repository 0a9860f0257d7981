"""Route of the fp64 operator between cell vectors and one lane per cell.

At degrees 1 and 2 the bare operator leaves the cell vectors at fewer cells than the
smoother does: beyond the line it gives the bits of cell_kernel = 3 (one lane per cell),
below it another order of sums.  The two agree to twice 1e-12, each kernel's distance
to the oracle elsewhere; the host-vector operator takes the same route by tile groups.
The smoother stays with the cell vectors on both sides.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# degree, mesh, cells, beyond the line
CASES = [(1, synth.uniform_cube(5), 32768, True), (1, synth.sphere(6), 21512, False),
         (2, synth.sphere(6), 21512, True), (2, synth.cube_octant(4, 1), 7680, False),
         (3, synth.cube_octant(4, 1), 7680, False)]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_route(gcmg, i):
    k, recipe, cells, beyond = CASES[i]
    m = gcmg.Mesh.from_recipe(recipe)
    assert m.level_cells(m.num_levels - 1) == cells
    a, b = gcmg.Multigrid(m, k), gcmg.Multigrid(m, k, cell_kernel=3)
    L = a.finest
    x = torch.randn(a.n_free(L), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(3))
    y, z = torch.empty_like(x), torch.empty_like(x)
    a.vmult(L, x, y)
    b.vmult(L, x, z)
    assert float((y - z).norm()) <= 2e-12 * float(z.norm())
    assert torch.equal(y, z) == beyond
    host = np.empty(len(x))
    a.vmult_host(L, x.cpu().numpy(), host)
    assert np.array_equal(host, y.cpu().numpy()) or not beyond
    assert float((torch.tensor(host) - y.cpu()).norm()) <= 2e-12 * float(y.norm())
    s = [x.clone(), x.clone()]
    a.smooth(L, s[0], y, False)
    b.smooth(L, s[1], y, False)
    assert not torch.equal(s[0], s[1])
    assert float((s[0] - s[1]).norm()) <= 8e-12 * float(s[1].norm())


@pytest.mark.parametrize("k,recipe", [(1, synth.sphere(6)), (1, synth.cube_octant(5, 1)), (2, synth.sphere(6)),
                                      (3, synth.cube_octant(4, 1))])
def test_cell_vectors_beyond_two_tiles_per_sm(gcmg, k, recipe):
    """the larger levels of low degree that take the cell vectors, against one lane per cell"""
    m = gcmg.Mesh.from_recipe(recipe)
    a, b = gcmg.Multigrid(m, k), gcmg.Multigrid(m, k, cell_kernel=3)
    L = a.finest
    for dtype, tol in ((torch.float64, 2e-12), (torch.float32, 4e-6)):
        gen = torch.Generator(device="cuda").manual_seed(21)
        x, f = (torch.randn(a.n_free(L), dtype=dtype, device="cuda", generator=gen) for _ in range(2))
        y, z = torch.empty_like(x), torch.empty_like(x)
        a.vmult(L, x, y)
        b.vmult(L, x, z)
        assert float((y - z).double().norm()) <= tol * float(z.double().norm())
        for zero in (False, True):  # three applications: four times the tolerance
            s, t = x.clone(), x.clone()
            a.smooth(L, s, f, zero)
            b.smooth(L, t, f, zero)
            assert not torch.equal(s, t)
            assert float((s - t).double().norm()) <= 4 * tol * float(t.double().norm())
