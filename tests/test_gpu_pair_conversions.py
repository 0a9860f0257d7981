"""Conversions between fp64 and pairs in the fp64 operator.

Inputs at which a conversion on the bits can go wrong: upper parts exactly half way
between two floats, powers of two and their neighbours (the low part crosses the
binade), zeros, both signs, and the same scaled by powers of two up to the exponents
at which the conversion on the bits hands over to the plain one.  A pair holds 48
bits, so the result is that of native fp64 1D matrices to 1e-12, the operator's bound,
at every scale.  One lane per cell (conversion on the bits) and cell vectors.
"""
import numpy as np
import pytest

import synth
from test_gpu_small_fp64 import _one_dimension

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _values(n):
    r = np.random.RandomState(8)
    one = 1.0 + r.randint(0, 1 << 23, n) * 2.0 ** -23
    kinds = [one + 2.0 ** -24,  # ties, even and odd
             one + 2.0 ** -24 + r.choice([-1, 1], n) * 2.0 ** -52, 2.0 ** r.randint(-3, 4, n),
             2.0 ** r.randint(-3, 4, n) * (1 - 2.0 ** -53), 2.0 ** r.randint(-3, 4, n) * (1 + 2.0 ** -52),
             1.0 - 2.0 ** -30 * r.rand(n), np.zeros(n), r.randn(n), one * (2 - 2.0 ** -23)]
    pick = r.randint(0, len(kinds), n)
    return np.choose(pick, kinds) * r.choice([-1.0, 1.0], n)


@pytest.mark.parametrize("kernel", [0, 3])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_conversions(gcmg, k, kernel):
    mg = gcmg.Multigrid(gcmg.Mesh.from_recipe(synth.uniform_cube(3)), k, cell_kernel=kernel, mg_fp32=False)
    L = mg.finest
    K, M, points = _one_dimension(k, 8)
    n = len(points)
    near = np.searchsorted((points[1:] + points[:-1]) / 2, mg.dof_coords(L))
    at = (near[:, 2] * n + near[:, 1]) * n + near[:, 0]
    X = _values(n ** 3)
    T = X.reshape(n, n, n)
    R = sum(np.einsum("zc,yb,xa,cba->zyx", *([K if e == d else M for e in range(3)]), T, optimize=True) for d in range(3))
    want = torch.tensor(R.reshape(-1)[at], device="cuda")
    for s in (-68, -40, 0, 40, 110):
        x = torch.tensor(X[at] * 2.0 ** s, device="cuda")
        y = torch.empty_like(x)
        mg.vmult(L, x, y)
        assert float((y * 2.0 ** -s - want).norm()) <= 1e-12 * float(want.norm()), s
