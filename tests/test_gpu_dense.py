"""The V-cycle matrix of the smallest levels against the level-by-level cycle.

With timers on, the cycle runs level by level; with them off, the levels of at
most 1,024 DoFs take one matrix.  Both are the same linear map: fp64 to 1e-11
of the result's norm (the parity of the V-cycle with the oracle is 1e-10; the
matrix is built in native fp64, the level operators run in 48-bit pairs), fp32
to 1e-5 (chains of about 100 roundings of 6e-8 over the levels).  Meshes whose
finest level is itself that small, that have empty coarse levels (k = 1), the
polynomial hierarchy, a coefficient; a changed Chebyshev interval falls back.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(synth.octant(5), 1, False), (synth.cube_octant(2, 1), 2, False), (synth.cube_octant(3, 1), 3, False),
         (synth.octant(3), 4, False), (synth.sphere(5), 4, True), (synth.shell(5), 2, True),
         (synth.cube_octant(1, 0), 4, False), (synth.cube_octant(3, 0), 1, False)]


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("i", range(len(CASES)))
@pytest.mark.parametrize("coef", [False, True])
def test_dense_cycle_is_the_level_by_level_cycle(gcmg, i, fp32, coef):
    rec, k, p = CASES[i]
    mg = gcmg.Multigrid(gcmg.Mesh.from_recipe(rec), k, p_coarsening=p, mg_fp32=fp32)
    if coef:
        mg.set_coefficient(1.0 + torch.rand(mg.n_cells(mg.finest), dtype=torch.float64, device="cuda",
                                            generator=torch.Generator(device="cuda").manual_seed(3)))
    b = torch.randn(mg.n_free(mg.finest), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(7))
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    n0 = gcmg.launch_count()
    mg.vcycle(b, x)
    n1 = gcmg.launch_count()
    mg.set_profiling(True)
    mg.vcycle(b, y)
    n2 = gcmg.launch_count()
    assert n1 - n0 < n2 - n1  # the matrix replaced launches
    tol = 1e-5 if fp32 else 1e-11
    assert float((x - y).norm()) <= tol * float(y.norm())
    mg.set_profiling(False)
    mg.set_lambda(1, 1.5 * mg.get_lambda(1))  # level by level again, with the new interval
    mg.vcycle(b, x)
    mg.set_profiling(True)
    mg.vcycle(b, y)
    assert torch.equal(x, y)
