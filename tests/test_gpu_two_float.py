"""FP32 compressed frames with their own neighbour search, whose pair displacements come from two-float
positions, against the same frames with a list built beforehand, whose displacements are FP64: the displacement is
the FP64 one rounded to FP32 on both, so the atomic energies are the same to the last bit.  Frames with images, far
from the origin (where the FP64 fallback decides most pairs), skewed, and without a box.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shift", [0.0, 37.25, 1.0e5])
@pytest.mark.parametrize("shape", ["cubic", "skewed", "open"])
def test_two_float_displacement(shape, shift):
    from paper_2304_09409_gb300 import dpgb
    cfg = I.water_model()
    m = dpgb.Model(cfg, I.make_params(cfg, 4), precision="fp32", compressed=True)
    fr = I.replicate(I.water_frame(3), (2, 2, 1))
    box = fr.box.copy()
    if shape == "skewed":
        box[1, 0], box[2, 0], box[2, 1] = 2.5, -1.75, 3.125
    coord = fr.coord @ np.linalg.inv(fr.box) @ box + shift * np.array([1.0, -1.0, 0.5])
    box = None if shape == "open" else box
    e0, f0, v0, a0 = m.compute(coord, fr.atype, box, atom_energy=True)
    nl = m.build_nlist(coord, fr.atype, box)
    e1, f1, v1, a1 = m.compute(coord, fr.atype, box, nlist=nl, atom_energy=True)
    m.free()
    assert np.abs(a0).max() > 0 and np.array_equal(np.asarray(a0), np.asarray(a1))
    assert np.abs(f0 - f1).max() <= 1e-12 * np.abs(f0).max()
