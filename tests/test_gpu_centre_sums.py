"""The warp's sums of force and virial per centre atom (csrc/emb_tc.cu, add_to_centre) where a warp holds the slots of
one atom, of two, and of many (short lists), with a last warp cut short.  FP64 against the oracle (|dF| <= 1e-9 eV/A,
virial relative 1e-10), TF32 against FP64 (FP32 sums of TF32 networks: 5e-2 of the largest force).
"""
import numpy as np
import pytest

import oracle
from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n, sel", [(2, (1, 1)), (4, (2, 3)), (7, (6, 6)), (9, (20, 12)), (9, (33, 30)), (11, (70, 75))])
def test_centre_sums(n, sel):
    from paper_2304_09409_gb300 import dpgb
    cfg = I.ModelConfig(ntypes=2, rcut=6.0, rcut_smth=0.5, sel=sel, embed=(16, 32), axis=4, fit=(32, 32))
    p = I.make_params(cfg, 2)
    rng = np.random.default_rng(n)
    grid = np.stack(np.meshgrid(*[np.arange(3)] * 3, indexing="ij"), -1).reshape(-1, 3)[rng.permutation(27)[:n]]
    coord = 15.0 + 1.3 * grid + rng.uniform(-0.2, 0.2, (n, 3))
    atype = (np.arange(n) % 2).astype(np.int32)
    box = np.eye(3) * 40.0
    ref = oracle.compute(cfg, p, coord, atype, box)
    out = {}
    for prec in ("fp64", "tf32"):
        m = dpgb.Model(cfg, p, precision=prec)
        e, f, v, _ = m.compute(coord, atype, box)
        out[prec] = f
        m.free()
        if prec == "fp64":
            assert np.abs(f - ref.force).max() <= 1e-9
            assert np.abs(v - ref.virial).max() <= 1e-10 * max(np.abs(ref.virial).max(), 1.0)
    assert np.abs(out["tf32"] - ref.force).max() <= 5e-2 * np.abs(ref.force).max()
