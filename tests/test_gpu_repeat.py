"""Every call of a model starts from zero: repeated calls on the same inputs give the first call's result, and another
model's workspace contents are never part of it.

Calls 1 to 4 of one shape run directly, are recorded, and are replayed.  Tolerance: the order of FP64 additions in the
scatter (1e-12 of the largest value) in FP64; in FP32 the se_e3 pair sums are unordered FP32 additions, about a hundred
to a value: 100 * 2^-24 = 6e-6 of the largest value.  A sum left over from the call before is off by 1.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MODELS = {"a": (I.water_model, I.WATER_FORCE_SCALE), "r": (I.water_model_r, I.WATER_R_FORCE_SCALE),
          "e3": (I.water_model_e3, I.WATER_E3_FORCE_SCALE), "hybrid": (I.water_model_hybrid, I.WATER_HYBRID_FORCE_SCALE),
          "hybrid_e3": (I.water_model_hybrid_e3, I.WATER_HYBRID_E3_FORCE_SCALE)}
CASES = [(k, prec, comp) for prec in ("fp64", "fp32") for k, comps in
         (("a", (0, 1)), ("r", (0, 1)), ("e3", (0, 1)), ("hybrid", (0,)), ("hybrid_e3", (0,))) for comp in comps]
CASES += [("a", "bf16", 0), ("a", "bf16", 1), ("a", "tf32", 0)]


@pytest.mark.parametrize("kind,precision,compressed", CASES)
def test_repeated_calls_agree(kind, precision, compressed):
    from paper_2304_09409_gb300 import dpgb
    make, scale = MODELS[kind]
    cfg = make()
    fr = I.water_frame(0)
    m = dpgb.Model(cfg, I.force_scaled(cfg, I.make_params(cfg, 0), scale), precision=precision, compressed=bool(compressed))
    coord, atype = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    out = m.compute(coord, atype, fr.box, atom_energy=True)
    first = [x.cpu().numpy().copy() for x in out]
    tol = 1e-12 if precision == "fp64" else 6e-6
    for _ in range(3):
        out = m.compute(coord, atype, fr.box, atom_energy=True, out=out)
        for x, y in zip(out, first):
            assert np.abs(x.cpu().numpy() - y).max() <= tol * np.abs(y).max()
    m.free()
