"""A type outside the model's in a device array that earlier calls have used: the call fails with the argument error,
nothing is read out of range on the way (the kernels run before the host knows), and the next call with the types put
right gives what it gave before (1e-12 of the largest value: the order of FP64 additions; FP32 parameter gradients 1e-6,
slabs of rows added in no fixed order).
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MODES = [("fp64", False), ("fp32", False), ("tf32", False), ("fp64", True), ("fp32", True), ("bf16", True)]


@pytest.mark.parametrize("precision,compressed", MODES)
@pytest.mark.parametrize("external", [False, True])
def test_bad_type_is_refused(precision, compressed, external):
    from paper_2304_09409_gb300 import dpgb
    cfg, fr = I.water_model(), I.water_frame(0)
    m = dpgb.Model(cfg, I.water_params_scaled(0), precision=precision, compressed=compressed)
    coord, atype = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    nlist = m.build_nlist(coord, atype, fr.box) if external else None
    out = m.compute(coord, atype, fr.box, nlist)
    ref = [x.cpu().numpy().copy() for x in out[:3]]
    for bad, at in ((2, [0]), (-1, [5, 191]), (2**31 - 1, list(range(0, 192, 3))), (100000, list(range(192)))):
        good = atype.clone()
        atype[torch.tensor(at, device="cuda")] = bad
        for _ in range(3):
            with pytest.raises(dpgb.DPError, match="type outside"):
                m.compute(coord, atype, fr.box, nlist, out=out)
        atype.copy_(good)
        out = m.compute(coord, atype, fr.box, nlist, out=out)
        for x, y in zip(out[:3], ref):
            assert np.abs(x.cpu().numpy() - y).max() <= 1e-12 * np.abs(y).max()
    m.free()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_bad_type_is_refused_in_param_grad(precision):
    from paper_2304_09409_gb300 import dpgb
    cfg, fr = I.water_model(), I.water_frame(0)
    m = dpgb.Model(cfg, I.water_params_scaled(0), precision=precision)
    coord, atype = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    nat, ge, gf = np.array([192], dtype=np.int32), np.ones(1), np.zeros((192, 3))
    ref = dpgb.param_grad(m, nat, coord, atype, fr.box[None], ge, gf).cpu().numpy()
    for bad, at in ((2, [0]), (-7, [5, 191]), (100000, list(range(192)))):
        good = atype.clone()
        atype[torch.tensor(at, device="cuda")] = bad
        with pytest.raises(dpgb.DPError, match="type outside"):
            dpgb.param_grad(m, nat, coord, atype, fr.box[None], ge, gf)
        atype.copy_(good)
        got = dpgb.param_grad(m, nat, coord, atype, fr.box[None], ge, gf).cpu().numpy()
        assert np.abs(got - ref).max() <= (1e-12 if precision == "fp64" else 1e-6) * np.abs(ref).max()
    m.free()
