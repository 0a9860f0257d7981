"""Paths of the V-cycle that an option or the hierarchy selects, against one another.

A set chunk size asks for the general restriction on every level: the cycle then
takes it also onto levels of few cells, whose restriction otherwise stays in the cell
vectors.  Both are the same linear map: fp64 1e-11 of the result's norm, as for the
matrix of the smallest levels (`test_gpu_dense.py`); the order of their sums differs,
and with it the last bits.  Under local smoothing that matrix stops at
the first level with copied values; with timers on the cycle runs level by level.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MESHES = {"cube3+1": synth.cube_octant(3, 1), "sphere5": synth.sphere(5), "shell5": synth.shell(5),
          "octant4": synth.octant(4)}


def _cycle(gcmg, mg, b):
    x = torch.zeros_like(b)
    n = gcmg.launch_count()
    mg.vcycle(b, x)
    return x, gcmg.launch_count() - n


def _rhs(mg):
    return torch.randn(mg.n_free(mg.finest), dtype=torch.float64, device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(13))


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("mesh", sorted(MESHES))
def test_chunk_size_reaches_every_level(gcmg, mesh, k, local):
    m = gcmg.Mesh.from_recipe(MESHES[mesh])
    new = gcmg.Multigrid(m, k, mg_fp32=False, local_smoothing=local)
    top = new.num_levels - (2 if local else 1)
    b = _rhs(new)
    x, _ = _cycle(gcmg, new, b)
    for chunk in (4, 8):
        y, _ = _cycle(gcmg, gcmg.Multigrid(m, k, mg_fp32=False, local_smoothing=local, transfer_chunk=chunk), b)
        assert float((x - y).norm()) <= 1e-11 * float(y.norm())
        if new.n_free(top) > 1024:  # at least one restriction above the matrix
            assert not torch.equal(x, y)


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("mesh", sorted(MESHES))
def test_matrix_under_local_smoothing(gcmg, mesh, k):
    mg = gcmg.Multigrid(gcmg.Mesh.from_recipe(MESHES[mesh]), k, mg_fp32=False, local_smoothing=True)
    b = _rhs(mg)
    x, few = _cycle(gcmg, mg, b)
    mg.set_profiling(True)
    y, many = _cycle(gcmg, mg, b)
    assert few < many  # the matrix replaced launches
    assert float((x - y).norm()) <= 1e-11 * float(y.norm())
