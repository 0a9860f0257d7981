"""CG as one graph launch against the host loop of plain launches.

The same kernels run in the same order, so x, the iteration count, the status and
the residual are equal bit for bit: converged, stopped by maxit (0 included), a
zero and a NaN right-hand side, both precisions of the V-cycle, local smoothing,
one reduction block (up to 8,192 DoFs) and several, repeated solves with other
vectors, tolerances and limits on one handle.
"""
import math

import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(synth.cube_octant(2, 1), 2, {}), (synth.octant(5), 3, {}), (synth.octant(4), 2, dict(mg_fp32=False)),
         (synth.shell(5), 2, dict(local_smoothing=True)), (synth.sphere(5), 4, dict(p_coarsening=True))]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_graph_equals_host_loop(gcmg, i):
    rec, k, kw = CASES[i]
    m = gcmg.Mesh.from_recipe(rec)
    a, b = gcmg.Multigrid(m, k, **kw), gcmg.Multigrid(m, k, **kw)
    b.set_graphs(False)
    rhs = a.rhs()
    rand = torch.randn(rhs.numel(), dtype=torch.float64, device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(1))
    nan = rhs.clone()
    nan[0] = math.nan
    for f, rtol, maxit in ((rhs, 1e-8, 100), (rand, 1e-6, 100), (rhs, 1e-8, 2), (rhs, 1e-8, 0), (0 * rhs, 1e-8, 5),
                           (nan, 1e-8, 5), (rhs, 1e-8, 100)):
        x, y = torch.ones_like(rhs), torch.ones_like(rhs)
        s, t = a.cg_solve(f, x, rtol, maxit, raise_on_fail=False), b.cg_solve(f, y, rtol, maxit, raise_on_fail=False)
        assert (s.iterations, s.status) == (t.iterations, t.status), (rtol, maxit)
        assert torch.equal(torch.nan_to_num(x), torch.nan_to_num(y))
        assert s.r0 == t.r0 or (math.isnan(s.r0) and math.isnan(t.r0))
        assert s.rel_residual == t.rel_residual or (math.isnan(s.rel_residual) and math.isnan(t.rel_residual))
