"""The level transfer with one warp per coarse cell against the general kernels.

The restriction with a set chunk size (transfer_chunk = 4) runs the general
kernel, the default the one with one warp per coarse cell, on the same mesh and
numbering.  fp64: both sum at most a few hundred products per coarse entry in
different orders, 1e-14 of the result's norm.  fp32: a chain of about 30
roundings of 6e-8 each side, 1e-6 of the norm.  The prolongation is the
transpose of the restriction: <P c, f> = <c, R f> to 1e-13 of |P c| |f| (fp64).
Meshes: hanging nodes on every level, coarse cell counts that are no multiple of
8 or 32, refined and unrefined coarse cells, 8-, 16- and 32-cell tiles, the
refinement levels of local smoothing (coarse cells without fine ones), and the
polynomial hierarchy (degree k to floor(k / 2) on one mesh).
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MESHES = {"octant5": synth.octant(5), "shell5": synth.shell(5), "cube2+1": synth.cube_octant(2, 1),
          "sphere6": synth.sphere(6), "cube4+1": synth.cube_octant(4, 1)}


def _rand(n, dtype, seed):
    return torch.randn(n, dtype=dtype, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


@pytest.mark.parametrize("variant", ["global", "local", "p"])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("mesh", sorted(MESHES))
def test_lattice_transfer(gcmg, mesh, k, variant):
    m = gcmg.Mesh.from_recipe(MESHES[mesh])
    local, p = variant == "local", variant == "p"
    new = gcmg.Multigrid(m, k, p_coarsening=p, local_smoothing=local)
    old = gcmg.Multigrid(m, k, p_coarsening=p, local_smoothing=local, transfer_chunk=4)
    top = new.num_levels - (2 if local else 1)
    for l in range(1, top + 1):
        nf, nc = new.n_free(l), new.n_free(l - 1)
        if nf == 0 or nc == 0:
            continue
        for dtype, tol in ((torch.float64, 1e-14), (torch.float32, 1e-6)):
            f, c = _rand(nf, dtype, 10 + l), _rand(nc, dtype, 20 + l)
            a, b = c.clone(), c.clone()
            new.restrict_add(l, f, a)
            old.restrict_add(l, f, b)
            assert float((a - b).double().norm() / b.double().norm()) <= tol, (l, dtype)
        pc = torch.zeros(nf, dtype=torch.float64, device="cuda")
        c = _rand(nc, torch.float64, 30 + l)
        f = _rand(nf, torch.float64, 40 + l)
        r = torch.zeros(nc, dtype=torch.float64, device="cuda")
        new.prolongate_add(l, c, pc)
        new.restrict_add(l, f, r)
        assert abs(float(pc @ f - c @ r)) <= 1e-13 * float(pc.norm() * f.norm()), l
