"""Precision of the fp64 operator on levels of few cells (the cell vectors).

Their pairs must be no worse than those of the line-parallel kernel that runs such
a level with cell_kernel = 1: the same random vector through both, errors against
the operator of a uniform cube as a sum of products of assembled 1D matrices in
native fp64 (a few 1e-16).  The two errors are sums of independent roundings over
at least 3,000 DoFs: a tenth of a per cent to a per cent of scatter, so 2 %.
"""
import numpy as np
import pytest

import synth
from test_gpu_energy_fp64 import NODES

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _one_dimension(k, cells):
    """assembled interior stiffness and mass matrices and the interior points"""
    x = 0.5 + 0.5 * np.array(NODES[k])
    t, w = np.polynomial.legendre.leggauss(k + 2)
    t, w = 0.5 + 0.5 * t, 0.5 * w
    v, d = np.empty((len(t), k + 1)), np.zeros((len(t), k + 1))
    for a in range(k + 1):
        others = [b for b in range(k + 1) if b != a]
        v[:, a] = np.prod([(t - x[b]) / (x[a] - x[b]) for b in others], axis=0)
        for m in others:
            d[:, a] += np.prod([(t - x[b]) / (x[a] - x[b]) for b in others if b != m], axis=0) / (x[a] - x[m])
    n = cells * k + 1
    K, M = np.zeros((n, n)), np.zeros((n, n))
    for c in range(cells):
        s = slice(c * k, c * k + k + 1)
        K[s, s] += cells * (d.T * w) @ d
        M[s, s] += (v.T * w) @ v / cells
    points = ((np.arange(cells)[:, None] + x[None, :-1]) / cells).reshape(-1)
    return K[1:-1, 1:-1], M[1:-1, 1:-1], points[1:]


@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_pairs_are_no_worse_than_the_line_kernel(gcmg, k):
    m = gcmg.Mesh.from_recipe(synth.uniform_cube(4))
    K, M, points = _one_dimension(k, 16)
    K, M = torch.tensor(K, device="cuda"), torch.tensor(M, device="cuda")
    n = len(points)
    err = []
    for kernel in (0, 1):
        mg = gcmg.Multigrid(m, k, cell_kernel=kernel, mg_fp32=False)
        L = mg.finest
        near = np.searchsorted((points[1:] + points[:-1]) / 2, mg.dof_coords(L))
        at = torch.tensor((near[:, 2] * n + near[:, 1]) * n + near[:, 0], device="cuda")
        X = torch.randn(n ** 3, dtype=torch.float64, device="cuda",
                        generator=torch.Generator(device="cuda").manual_seed(11))
        x = X[at].contiguous()
        y = torch.empty_like(x)
        mg.vmult(L, x, y)
        X = X.reshape(n, n, n)
        R = sum(torch.einsum("zc,yb,xa,cba->zyx", *([K if e == d else M for e in range(3)]), X) for d in range(3))
        R = R.reshape(-1)[at]
        err.append(float((y - R).norm() / R.norm()))
    assert err[0] <= 1.02 * err[1], err
