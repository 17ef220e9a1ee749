"""The parameter gradient sums each slab of rows in a fixed order: where every net has one slab (at most 128 listed rows,
512 atoms), all its values but those of the first embedding layer (whose kernel adds rows in no fixed order) repeat to
the bit, from call to call and from model to model.  16 atoms of 400 slots: the real rows lie in 25 blocks of rows, which
finish in another order every time.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("one_side", [0, 1])
def test_gradient_repeats_to_the_bit(precision, one_side):
    from paper_2304_09409_gb300 import dpgb
    cfg = I.ModelConfig(ntypes=2, rcut=4.0, rcut_smth=0.5, sel=(200, 200), embed=(5, 10, 20), axis=4, fit=(24, 24),
                        type_one_side=one_side)
    fr = I.random_frame(16, 2, np.eye(3) * 9.0, seed=3, min_dist=1.2)
    nat, box = np.array([16], dtype=np.int32), fr.box[None]
    coord, atype = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    rng = np.random.default_rng(5)
    ge, gf, gv = np.ones(1), rng.normal(size=(16, 3)), rng.normal(size=(1, 3, 3))
    fixed = np.ones(dpgb.n_params(cfg), dtype=bool)
    nets, shapes = (2 if one_side else 4), [(1, 5), (5, 10), (10, 20)]
    per_net = sum((a + 1) * b for a, b in shapes)
    for n in range(nets):
        fixed[n * per_net:n * per_net + 2 * shapes[0][1]] = False
    first = None
    for _ in range(3):
        m = dpgb.Model(cfg, I.make_params(cfg, 0), precision=precision)
        for _ in range(20):
            g = dpgb.param_grad(m, nat, coord, atype, box, ge, gf, g_virial=gv).cpu().numpy()
            first = g if first is None else first
            assert np.array_equal(g[fixed], first[fixed])
        m.free()
    assert np.abs(first[fixed]).max() > 0
