"""Energy of a smooth field under the fp64 (double-float) operator.

x = sin(pi x) sin(pi y) sin(pi z) on a uniform [0, 1]^3: x^T A x = 3 E_K E_M^2 with
the 1D energies E_K and E_M, formed here by Gauss quadrature of differences, in
which constants drop out exactly (1e-15).  As for fp32, the rows of the cell matrix
have to sum to zero: rounded entry by entry to pairs they did not, 1.9e-12 at degree
3 on 32^3 cells, growing like h^-2.  A pair that is not normalised between two
steps of a line keeps at least 46 bits; about ten such roundings in one chain:
16 2^-46.  Whole tiles (cell_kernel 3) and cell vectors (4,096 cells, default).
"""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NODES = {1: [-1, 1], 2: [-1, 0, 1], 3: [-1, -(1 / 5) ** 0.5, (1 / 5) ** 0.5, 1],
         4: [-1, -(3 / 7) ** 0.5, 0, (3 / 7) ** 0.5, 1]}


def _energies(k, cells):
    """(E_K, E_M) of sin(pi x) on `cells` 1D cells of degree k"""
    x = 0.5 + 0.5 * np.array(NODES[k])
    t, w = np.polynomial.legendre.leggauss(k + 2)
    t, w = 0.5 + 0.5 * t, 0.5 * w
    v, d = np.empty((len(t), k + 1)), np.zeros((len(t), k + 1))
    for a in range(k + 1):
        others = [b for b in range(k + 1) if b != a]
        v[:, a] = np.prod([(t - x[b]) / (x[a] - x[b]) for b in others], axis=0)
        for m in others:
            d[:, a] += np.prod([(t - x[b]) / (x[a] - x[b]) for b in others if b != m], axis=0) / (x[a] - x[m])
    s = np.sin(math.pi * (np.arange(cells)[:, None] + x) / cells)
    ds = (s - s[:, :1]) @ d.T  # constants drop out
    return float((ds ** 2 @ w).sum() * cells), float(((s @ v.T) ** 2 @ w).sum() / cells)


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("depth,kernel", [(4, 0), (4, 3), (5, 3)])
def test_energy_of_a_smooth_field(gcmg, depth, kernel, k):
    mg = gcmg.Multigrid(gcmg.Mesh.from_recipe(synth.uniform_cube(depth)), k, cell_kernel=kernel)
    L = mg.finest
    x = torch.sin(math.pi * torch.tensor(mg.dof_coords(L), device="cuda")).prod(1).contiguous()
    y = torch.empty_like(x)
    mg.vmult(L, x, y)
    ek, em = _energies(k, 2 ** depth)
    assert abs(float(x @ y) - 3 * ek * em ** 2) <= 16 * 2.0 ** -46 * 3 * ek * em ** 2
