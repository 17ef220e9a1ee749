"""CUDA-core dense layers (csrc/dense.cu, csrc/grad.cu) at the widths and row counts where a tile, a K
chunk, a row list or a row slab ends unevenly: FP64 energies and forces against the oracle, FP32 against
FP64, the energy's parameter gradient against central differences of the FP64 path's own energies.

Tolerances: FP64 as the parity tests (1e-10 eV per atom, 1e-9 eV/A).  FP32: a sum of K products is off by
at most K 2^-24 of the sum of their magnitudes (1e-4 at K = 1,600), forward and backward; with the
cancellation of forces within an order of magnitude, 2e-3 of the largest force.  Central differences
at h = 1e-4 along a unit direction: h^2 times a third derivative of order one, 1e-7, taken with a factor
of ten.
"""
import numpy as np
import pytest

import oracle
from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TRI = I.triclinic_box(9.0, (1.1, -0.7, 0.9))


def _cfg(ntypes, sel, embed, axis, fit, one_side=0):
    return I.ModelConfig(ntypes=ntypes, rcut=6.0, rcut_smth=0.5, sel=sel, embed=embed, axis=axis, fit=fit,
                         type_one_side=one_side)


CASES = {
    # widths below, at and just beyond a quad, a 32- and a 52-column tile; skips {x,x} and +x; one row tile
    "tiny_odd": (_cfg(2, (40, 40), (5, 10, 10), 3, (33, 33)), lambda: I.random_frame(14, 2, TRI, 3, 1.2)),
    # a type without atoms (no rows), one-sided nets, one hidden layer each
    "empty_type": (_cfg(3, (40, 40, 8), (7,), 4, (53,), 1), lambda: I.random_frame(17, 2, TRI, 5, 1.2)),
    # the water nets: short lists of tiles, then enough rows for the persistent embedding kernels
    "water_192": (I.water_model(), lambda: I.water_frame(2)),
    "water_1536": (I.water_model(), lambda: I.replicate(I.water_frame(2), (2, 2, 2))),
    # 32 / 64 / 128 columns (whole tiles) over a single type, ragged last tiles
    "metal_500": (_cfg(1, (256,), (32, 64, 128), 16, (240, 240)), lambda: I.fcc_frame((5, 5, 5), seed=4)),
}


def _dev(fr):
    return torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")


@pytest.mark.parametrize("name", list(CASES))
def test_dense_energy_force(name):
    from paper_2304_09409_gb300 import dpgb
    cfg, make = CASES[name]
    fr, p = make(), I.make_params(cfg, 1)
    ref = oracle.compute(cfg, p, fr.coord, fr.atype, fr.box)
    c, t = _dev(fr)
    for prec in ("fp64", "fp32"):
        m = dpgb.Model(cfg, p, precision=prec)
        e, f, _, _ = m.compute(c, t, fr.box)
        de, df = abs(float(e.cpu()[0]) - ref.energy) / fr.natoms, float(np.abs(f.cpu().numpy() - ref.force).max())
        print(f"{name} {prec}: |dE|/atom {de:.1e} |dF| {df:.1e} (max |F| {np.abs(ref.force).max():.1e})")
        if prec == "fp64":
            assert de <= 1e-10 and df <= 1e-9
        else:
            assert df <= 2e-3 * np.abs(ref.force).max() and de <= 1e-4 * max(1.0, abs(ref.energy) / fr.natoms)
        m.free()


@pytest.mark.parametrize("name", list(CASES))
def test_dense_param_grad(name):
    from paper_2304_09409_gb300 import dpgb
    cfg, make = CASES[name]
    fr, p = make(), I.make_params(cfg, 1)
    c, t = _dev(fr)
    nat = np.array([fr.natoms], dtype=np.int32)
    ge, gf = np.ones(1), np.zeros((fr.natoms, 3))
    grads = {}
    m = dpgb.Model(cfg, p, precision="fp64")
    grads["fp64"] = dpgb.param_grad(m, nat, c, t, fr.box[None], ge, gf).cpu().numpy()
    rng = np.random.default_rng(7)
    h = 1e-4
    for _ in range(3):
        v = rng.normal(size=p.size)
        v /= np.linalg.norm(v)
        es = []
        for s in (h, -h):
            m.set_params(p + s * v)
            es.append(float(m.compute(c, t, fr.box)[0].cpu()[0]))
        fd, an = (es[0] - es[1]) / (2 * h), float(grads["fp64"] @ v)
        assert abs(fd - an) <= 1e-6 * max(1.0, fr.natoms), (fd, an)
    m.free()
    m = dpgb.Model(cfg, p, precision="fp32")
    grads["fp32"] = dpgb.param_grad(m, nat, c, t, fr.box[None], ge, gf).cpu().numpy()
    m.free()
    assert np.linalg.norm(grads["fp32"] - grads["fp64"]) <= 2e-3 * np.linalg.norm(grads["fp64"])
