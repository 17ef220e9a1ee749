"""Neighbour lists where the cell grid or the work split of the cell-centred search changes
(csrc/nlist.cu): boxes between one and three cutoffs wide, where half-width cells are taken, cells with
more centre atoms than one block serves, and the batch of such frames whose paddings end early; integer
results, bit-exact against the oracle's brute-force list, and energies and forces of the compressed path
against the same frame evaluated with a fully padded external list.
"""
import numpy as np
import pytest

import oracle
from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _frames():
    yield "metal 3x3x3 (10.9 A, r_c 8)", I.metal_model(), I.fcc_frame((3, 3, 3), seed=1)
    yield "metal 4x4x4 (14.5 A: one whole cell a side, three half cells)", I.metal_model(), I.fcc_frame((4, 4, 4), seed=2)
    yield "metal 4x5x6", I.metal_model(), I.fcc_frame((4, 5, 6), seed=3)
    yield "metal 7x4x3", I.metal_model(), I.fcc_frame((7, 4, 3), seed=4)
    yield "water 12.42 A (two cells a side)", I.water_model(), I.water_frame(5)
    yield "water 9.3 A (one whole cell, three half cells)", I.water_model(), I.water_frame(6, n_side=3)
    yield "water 11.7 x 11.7 x 37 A", I.water_model(), I.replicate(I.water_frame_n(53, 7), (1, 1, 3))
    yield "sheared", I.water_model(), I.random_frame(90, 2, I.triclinic_box(11.5, (3.0, -2.0, 1.5)), 8, 1.3)


@pytest.mark.parametrize("k", range(8))
def test_list_matches_brute_force(k):
    from paper_2304_09409_gb300 import dpgb
    name, cfg, fr = list(_frames())[k]
    m = dpgb.Model(cfg, I.make_params(cfg, 0), precision="fp32", compressed=True)
    c, t = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    nl = m.build_nlist(c, t, fr.box)
    j, s = nl.export()
    ref = oracle.nlist(cfg, fr.coord, fr.atype, fr.box)
    assert np.array_equal(j, ref[0].reshape(j.shape)), name
    assert np.array_equal(s, ref[1].reshape(s.shape)), name
    # the internal list stops its padding after the batch that ends each type block
    e0, f0, v0, _ = m.compute(c, t, fr.box, nlist=nl)
    e1, f1, v1, _ = m.compute(c, t, fr.box)
    scale = float(f0.abs().max())
    assert float((f0 - f1).abs().max()) <= 1e-12 * max(scale, 1e-3)
    assert abs(float(e0 - e1)) <= 1e-12 * abs(float(e0)) and float((v0 - v1).abs().max()) <= 1e-9 * float(v0.abs().max())
    nl.free()
    m.free()


def test_batch_of_narrow_boxes():
    from paper_2304_09409_gb300 import dpgb
    cfg = I.metal_model()
    frames = [I.fcc_frame(n, seed=k) for k, n in enumerate(((4, 4, 4), (3, 3, 3), (9, 9, 9), (4, 5, 4)))]
    m = dpgb.Model(cfg, I.metal_params_scaled(0), precision="fp32", compressed=True)
    nat = np.array([f.natoms for f in frames], dtype=np.int32)
    c = torch.tensor(np.concatenate([f.coord for f in frames]), device="cuda")
    t = torch.tensor(np.concatenate([f.atype for f in frames]), device="cuda")
    e, f, _, _ = dpgb.compute_batch(m, nat, c, t, np.stack([f.box for f in frames]))
    at = 0
    for k, fr in enumerate(frames):
        n = fr.natoms
        e1, f1, _, _ = m.compute(c[at:at + n].contiguous(), t[at:at + n].contiguous(), fr.box)
        # the same atoms alone and in the batch: FP32 rows of the same rounding, forces up to the order of
        # the FP64 scatter
        assert abs(float(e[k] - e1[0])) <= 1e-6 * abs(float(e1[0]))
        assert float((f[at:at + n] - f1).abs().max()) <= 1e-3
        at += n
    m.free()
