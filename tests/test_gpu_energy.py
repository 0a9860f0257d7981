"""Energy of a smooth field under the fp32 operator.

x = sin(pi x) sin(pi y) sin(pi z) on [0, 1]^3: the energy x^T A x is h^2 of the
products that the cell operator forms, so a cell matrix whose rows do not sum to
zero shows here (with one sign in every cell, growing like h^-2) where the 2-norm
on random vectors hides it.  x is rounded to fp32 once; both operators get these
values, and the sums are fp64.  The fp64 operator is exact to 1e-11 here.  What the
fp32 operator may add: every transform and product rounds relative to the part of
x that it acts on once constants drop out, about ten roundings of 2^-24 in one
chain whatever the mesh size: 16 2^-24.  Meshes: cell vectors (4,096 cells), whole
tiles (32,768 cells), tiles with hanging cells, one lane per cell and cell vectors.
"""
import math

import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(synth.uniform_cube(4), 0), (synth.uniform_cube(4), 3), (synth.uniform_cube(5), 3),
         (synth.cube_octant(4, 1), 0), (synth.cube_octant(4, 1), 3)]


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("i", range(len(CASES)))
def test_energy_of_a_smooth_field(gcmg, i, k):
    recipe, kernel = CASES[i]
    mg = gcmg.Multigrid(gcmg.Mesh.from_recipe(recipe), k, cell_kernel=kernel)
    L = mg.finest
    xyz = torch.tensor(mg.dof_coords(L), device="cuda")
    x = torch.sin(math.pi * xyz).prod(1).float()
    y32, x64 = torch.empty_like(x), x.double()
    y64 = torch.empty_like(x64)
    mg.vmult(L, x, y32)
    mg.vmult(L, x64, y64)
    e32, e64 = float(x64 @ y32.double()), float(x64 @ y64)
    assert abs(e32 - e64) <= 16 * 2.0 ** -24 * e64
