"""A Chebyshev interval that is changed and set back.

On a level of the matrix of the smallest levels another interval makes the cycle run
level by level; with the set-up's value again the matrix is taken again: the same
launches and the same bits as before.  Levels above it do not touch the matrix.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fp32", [False, True])
def test_interval_set_back(gcmg, fp32):
    mg = gcmg.Multigrid(gcmg.Mesh.from_recipe(synth.octant(4)), 2, mg_fp32=fp32)
    inside = [l for l in range(1, mg.num_levels) if 0 < mg.n_free(l) <= 1024]
    assert inside and mg.n_free(mg.finest) > 1024
    b = torch.randn(mg.n_free(mg.finest), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(2))

    def cycle():
        x = torch.zeros_like(b)
        n = gcmg.launch_count()
        mg.vcycle(b, x)
        return x, gcmg.launch_count() - n

    x, few = cycle()
    lam = {l: mg.get_lambda(l) for l in inside}
    for l in inside:
        mg.set_lambda(l, 1.25 * lam[l])
    y, many = cycle()
    assert many > few and not torch.equal(x, y)
    for l in inside:
        assert cycle()[1] == many  # one interval is still another
        mg.set_lambda(l, lam[l])
    z, again = cycle()
    assert again == few and torch.equal(x, z)
    top = mg.finest
    mg.set_lambda(top, 1.25 * mg.get_lambda(top))
    assert cycle()[1] == few
