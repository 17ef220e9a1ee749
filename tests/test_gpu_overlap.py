"""Atoms on top of one another in a compressed model: s = 1/r lies far beyond the table (and, at 1e-10 A, beyond what an
interval index can hold), the call fails with the range error, nothing is read out of range on the way, and the next call
on the frame put right gives what it gave before (1e-12 of the largest value: the order of FP64 additions; the unordered
FP32 sums of se_e3, 6e-6).
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kind,precision", [("a", "fp32"), ("a", "bf16"), ("a", "fp64"), ("r", "fp32"), ("r", "fp64"),
                                            ("e3", "fp32"), ("e3", "fp64")])
@pytest.mark.parametrize("gap", [1e-3, 1e-8, 1e-10, 1e-13])
def test_overlapping_atoms(kind, precision, gap):
    from paper_2304_09409_gb300 import dpgb
    cfg = {"a": I.water_model, "r": I.water_model_r, "e3": I.water_model_e3}[kind]()
    fr = I.water_frame(0)
    m = dpgb.Model(cfg, I.make_params(cfg, 0), precision=precision, compressed=True)
    coord, atype = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    out = m.compute(coord, atype, fr.box)
    ref = [x.cpu().numpy().copy() for x in out[:3]]
    good = coord.clone()
    coord[190] = coord[3]  # the frame's last row of pairs reads furthest
    coord[190, 0] += gap
    coord[191] = coord[1]
    coord[191, 2] -= gap
    for _ in range(3):
        if precision == "bf16" and gap <= 1e-10:  # below the FP32 cell-local positions' resolution: the distance is zero
            assert np.isnan(float(m.compute(coord, atype, fr.box, out=out)[0].cpu()[0]))
            continue
        with pytest.raises(dpgb.DPError) as err:
            m.compute(coord, atype, fr.box, out=out)
        assert err.value.code == dpgb.DP_E_RANGE
    coord.copy_(good)
    out = m.compute(coord, atype, fr.box, out=out)
    tol = 6e-6 if (kind, precision) == ("e3", "fp32") else 1e-12
    for x, y in zip(out[:3], ref):
        assert np.abs(x.cpu().numpy() - y).max() <= tol * np.abs(y).max()
    m.free()
