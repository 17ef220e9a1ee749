"""The split-operand fitting kernel (csrc/fit_split.cu) where its buffers change shape: one to four hidden
layers, widths of 16 to 256 (the 256-wide weight slots), layers of different width, a last dE/dD chunk of
every kind, descriptors with M_< other than 16 (dE/dD stored), ragged last tiles of both types.

The FP32 compressed path on a 12,288-atom frame (enough tiles for the one-kernel path) against the FP64
compressed path: every operand keeps about 16 significant bits (2^-17 relative per product), forward and
backward through at most five products, with the cancellation of forces two orders of magnitude above the
roundings' sum: 2e-3 of the largest force, 1e-5 of the largest atomic energy.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("embed_last, axis, fit", [
    (100, 16, (240,)),
    (100, 16, (64, 240)),
    (100, 16, (256, 256, 256)),
    (100, 16, (32, 256, 256, 16)),
    (16, 16, (16, 16, 16)),      # KD 256: a whole chunk and a third of one
    (28, 16, (128, 128)),        # KD 448: a last chunk of 64
    (100, 12, (240, 240, 240)),  # KD 1,200, M_< 12
    (20, 4, (48, 48)),           # KD 80: one short chunk
])
def test_fit_split_shapes(embed_last, axis, fit):
    from paper_2304_09409_gb300 import dpgb
    cfg = I.ModelConfig(ntypes=2, rcut=6.0, rcut_smth=0.5, sel=(46, 92), embed=(10, embed_last), axis=axis, fit=fit)
    p = I.make_params(cfg, 3)
    fr = I.replicate(I.water_frame(1), (4, 4, 4))
    fr = I.Frame(fr.coord[:-37].copy(), fr.atype[:-37].copy(), fr.box)  # ragged tiles of both types
    c, t = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    out = {}
    for prec in ("fp64", "fp32"):
        m = dpgb.Model(cfg, p, precision=prec, compressed=True)
        m.profile(True)
        e, f, v, ae = m.compute(c, t, fr.box, atom_energy=True)
        out[prec] = (f.cpu().numpy(), ae.cpu().numpy())
        if prec == "fp32":
            assert "fit_split_tc" in m.profile_read()
        m.free()
    (f0, a0), (f1, a1) = out["fp64"], out["fp32"]
    df, da = np.abs(f0 - f1).max() / np.abs(f0).max(), np.abs(a0 - a1).max() / np.abs(a0).max()
    print(f"M {embed_last} x {axis}, fit {fit}: |dF|/|F|max {df:.1e}, |dE_i|/max {da:.1e}")
    assert df <= 2e-3 and da <= 1e-5
