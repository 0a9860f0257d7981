"""Operator variants on one mesh and numbering against the line-parallel kernels.

cell_kernel = 1 runs one thread per line; the default takes the cell vectors on
levels of few cells, cell_kernel = 3 one lane per cell.  Each path is within
1e-12 (fp64, 48-bit pairs) or 2e-6 (fp32) of the oracle elsewhere, so two of them
differ by at most twice that of the result's norm.  Smoothing chains three
applications (factor 4), a V-cycle about 40 (fp64 1e-10, fp32 1e-4).  Meshes:
hanging faces and edges, one cell more than a multiple of the cells per warp, a
level with a single DoF, a coefficient.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MESHES = {"octant4": synth.octant(4), "shell5": synth.shell(5), "cube2+2": synth.cube_octant(2, 2),
          "sphere5": synth.sphere(5), "cube1": synth.uniform_cube(1)}


def _rand(n, dtype, seed):
    return torch.randn(n, dtype=dtype, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


def _close(a, b, tol):
    return float((a - b).double().norm()) <= tol * max(float(b.double().norm()), 1e-300)


@pytest.mark.parametrize("coef", [False, True])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("mesh", sorted(MESHES))
def test_variants_agree(gcmg, mesh, k, coef):
    m = gcmg.Mesh.from_recipe(MESHES[mesh])
    ref = gcmg.Multigrid(m, k, cell_kernel=1, mg_fp32=False)
    if ref.n_free(ref.finest) == 0:
        return
    new, lanes = gcmg.Multigrid(m, k, mg_fp32=False), gcmg.Multigrid(m, k, cell_kernel=3, mg_fp32=False)
    if coef:
        nu = 1.0 + torch.rand(ref.n_cells(ref.finest), dtype=torch.float64, device="cuda",
                              generator=torch.Generator(device="cuda").manual_seed(5))
        for g in (ref, new, lanes):
            g.set_coefficient(nu)
    for l in range(ref.num_levels):
        n = ref.n_free(l)
        if n == 0:
            continue
        for dtype, tol in ((torch.float64, 2e-12), (torch.float32, 4e-6)):
            x, b = _rand(n, dtype, l), _rand(n, dtype, 50 + l)
            y = [torch.empty_like(x) for _ in range(3)]
            for g, v in zip((ref, new, lanes), y):
                g.vmult(l, x, v)
            assert _close(y[1], y[0], tol) and _close(y[2], y[0], tol), (l, dtype)
            if l == 0:
                continue
            for zero in (False, True):
                s = [x.clone() for _ in range(2)]
                ref.smooth(l, s[0], b, zero)
                new.smooth(l, s[1], b, zero)
                assert _close(s[1], s[0], 4 * tol), (l, dtype, zero)
    b = _rand(ref.n_free(ref.finest), torch.float64, 99)
    for fp32, tol in ((False, 1e-10), (True, 1e-4)):
        a = gcmg.Multigrid(m, k, cell_kernel=1, mg_fp32=fp32)
        c = gcmg.Multigrid(m, k, mg_fp32=fp32)
        x, y = torch.zeros_like(b), torch.zeros_like(b)
        a.vcycle(b, x)
        c.vcycle(b, y)
        assert _close(y, x, tol), fp32
