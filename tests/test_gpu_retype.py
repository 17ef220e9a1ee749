"""Device type arrays rewritten in place between calls of one model, to compositions that the calls before had no room
for (every atom of the other type, then back): each call must give what a fresh model gives for the types as they are.

The same kernels run on the same inputs, so the results differ by the order of FP64 additions only (1e-12 of the largest
value); the FP32 parameter gradient also adds slabs of rows in no fixed order (a few FP32 additions per value: 1e-6 of
the largest).
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TWO_BODY = dict(ntypes=2, rcut=6.0, rcut_smth=0.5, sel=(112, 112), embed=(8, 16, 32), axis=4, fit=(32, 32))
CONFIGS = {"a": I.ModelConfig(**TWO_BODY),
           "hybrid": I.ModelConfig(**{**TWO_BODY, "rcut": 4.0}, descriptor=2, rcut_2=6.0, rcut_smth_2=0.5,
                                   sel_2=(112, 112), embed_2=(50, 50))}


def _types(n):
    mixed = np.tile(np.array([0, 1, 1], dtype=np.int32), n // 3)
    return [mixed, np.ones(n, dtype=np.int32), np.zeros(n, dtype=np.int32), mixed[::-1].copy(), np.ones(n, dtype=np.int32)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", list(CONFIGS))
def test_energy_force_after_retyping(kind, precision):
    from paper_2304_09409_gb300 import dpgb
    cfg = CONFIGS[kind]
    p, fr = I.make_params(cfg, 0), I.water_frame(0)
    coord, atype = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    m = dpgb.Model(cfg, p, precision=precision)
    out = None
    for t in _types(fr.natoms):
        atype.copy_(torch.tensor(t, device="cuda"))
        for _ in range(3):  # direct, recorded, replayed
            out = m.compute(coord, atype, fr.box, atom_energy=True, out=out)
            fresh = dpgb.Model(cfg, p, precision=precision)
            for x, y in zip(out, fresh.compute(fr.coord, t, fr.box, atom_energy=True)):
                assert np.abs(x.cpu().numpy() - y).max() <= 1e-12 * np.abs(y).max()
            fresh.free()
    m.free()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_param_grad_after_retyping(precision):
    from paper_2304_09409_gb300 import dpgb
    cfg = CONFIGS["a"]
    p, fr = I.make_params(cfg, 0), I.water_frame(0)
    coord, atype = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    nat, ge = np.array([fr.natoms], dtype=np.int32), np.ones(1)
    gf = np.random.default_rng(5).normal(size=(fr.natoms, 3))
    m = dpgb.Model(cfg, p, precision=precision)
    for t in _types(fr.natoms):
        atype.copy_(torch.tensor(t, device="cuda"))
        got = dpgb.param_grad(m, nat, coord, atype, fr.box[None], ge, gf).cpu().numpy()
        fresh = dpgb.Model(cfg, p, precision=precision)
        ref = dpgb.param_grad(fresh, nat, fr.coord, t, fr.box[None], ge, gf)
        fresh.free()
        assert np.abs(got - ref).max() <= (1e-12 if precision == "fp64" else 1e-6) * np.abs(ref).max()
    m.free()
