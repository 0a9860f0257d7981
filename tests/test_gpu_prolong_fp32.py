"""The fp32 prolongation against the fp64 one (pinned as the restriction's transpose).

Three sweeps of at most five products and the addition: a chain of about 20 roundings of
6e-8, 1e-6 of the result's norm.  Hanging nodes on every level, refined and unrefined
coarse cells, the refinement levels of local smoothing, the polynomial hierarchy.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("variant", ["global", "local", "p"])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("recipe", [synth.octant(5), synth.sphere(5), synth.cube_octant(4, 1)], ids=["octant", "sphere", "cube"])
def test_prolongation(gcmg, recipe, k, variant):
    local = variant == "local"
    mg = gcmg.Multigrid(gcmg.Mesh.from_recipe(recipe), k, p_coarsening=variant == "p", local_smoothing=local)
    for l in range(1, mg.num_levels - (1 if local else 0)):
        nf, nc = mg.n_free(l), mg.n_free(l - 1)
        if nf == 0 or nc == 0:
            continue
        gen = torch.Generator(device="cuda").manual_seed(l)
        c, f = (torch.randn(n, device="cuda", generator=gen) for n in (nc, nf))
        want = f.double()
        mg.prolongate_add(l, c.double(), want)
        mg.prolongate_add(l, c, f)
        assert float((f.double() - want).norm()) <= 1e-6 * float(want.norm()), l
