"""A frame gives the same energy, forces and virial alone and behind others in a batch, in every mode.

What differs is only where its rows stand: the pairs of an atom lie in other lanes and warps (the sums per centre of the
TF32 and BF16 force kernel: warps that hold one atom's pairs, two or many, and a last warp that is cut short), its atoms
in other tiles, its list came from another work split.  The values added are the same, so the results differ by the
order of FP64 additions: 1e-12 of the largest value; the FP32 sums of se_e3 are unordered: 6e-6.  Where
each pair adds one value to its two atoms (the uncompressed paths; the compressed ones sum an atom's own share in FP32
first) the forces of a frame cancel: their sum is zero to 1e-12 of the sum of their magnitudes.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SMALL = dict(rcut=6.0, rcut_smth=0.5, axis=16, fit=(64, 64))
# slots per atom: odd numbers, fewer than a warp and more than four
SLOTS = {"19 slots": I.ModelConfig(ntypes=2, sel=(8, 11), embed=(16, 32, 64), **{**SMALL, "rcut": 3.0}),
         "171 slots": I.ModelConfig(ntypes=2, sel=(80, 91), embed=(16, 32, 64), **SMALL)}


def _water():
    return [I.water_frame_n(n, seed=n) for n in (23, 64, 8, 107, 41)]


def _narrow():
    return [I.fcc_frame(n, seed=k) for k, n in enumerate(((4, 4, 4), (3, 3, 3), (9, 9, 9), (4, 5, 4)))]


CASES = [("water", I.water_model(), I.WATER_FORCE_SCALE, _water, p, c) for p, c in
         (("fp64", 0), ("fp32", 0), ("tf32", 0), ("bf16", 0), ("fp64", 1), ("fp32", 1), ("bf16", 1))]
CASES += [("metal", I.metal_model(), I.METAL_FORCE_SCALE, _narrow, p, c) for p, c in (("tf32", 0), ("bf16", 0), ("fp32", 1), ("bf16", 1))]
CASES += [("hybrid_e3", I.water_model_hybrid_e3(), I.WATER_HYBRID_E3_FORCE_SCALE, _water, "fp32", 0)]
CASES += [(n, cfg, 1.0, _water, p, 0) for n, cfg in SLOTS.items() for p in ("tf32", "bf16")]


@pytest.mark.parametrize("name,cfg,scale,frames,precision,compressed", CASES,
                         ids=["%s-%s-%d" % (c[0], c[4], c[5]) for c in CASES])
def test_alone_and_in_a_batch(name, cfg, scale, frames, precision, compressed):
    from paper_2304_09409_gb300 import dpgb
    frames = frames()
    m = dpgb.Model(cfg, I.force_scaled(cfg, I.make_params(cfg, 0), scale), precision=precision, compressed=bool(compressed))
    nat = np.array([f.natoms for f in frames], dtype=np.int32)
    e, f, v, _ = dpgb.compute_batch(m, nat, np.concatenate([x.coord for x in frames]),
                                    np.concatenate([x.atype for x in frames]).astype(np.int32), np.stack([x.box for x in frames]))
    tol = 6e-6 if "e3" in name else 1e-12
    at = 0
    for k, fr in enumerate(frames):
        e1, f1, v1, _ = m.compute(fr.coord, fr.atype, fr.box)
        fk = f[at:at + fr.natoms]
        at += fr.natoms
        assert abs(e[k] - e1[0]) <= tol * abs(e1[0])
        assert np.abs(fk - f1).max() <= tol * np.abs(f1).max()
        assert np.abs(v[k] - v1).max() <= tol * np.abs(v1).max()
        if not compressed:
            assert np.abs(f1.sum(0)).max() <= 1e-12 * np.abs(f1).sum()
    m.free()


@pytest.mark.parametrize("name", ["water", "metal"])
def test_tf32_virial_against_fp64(name):
    """The TF32 force kernel's nine virial sums against FP64: TF32 operands (2^-11) through seven layers, the path's own
    5 % of the largest component as for its forces; a lost, doubled or transposed sum is off by far more."""
    from paper_2304_09409_gb300 import dpgb
    make, scale, frames = (I.water_model, I.WATER_FORCE_SCALE, _water) if name == "water" else \
        (I.metal_model, I.METAL_FORCE_SCALE, _narrow)
    cfg = make()
    p = I.force_scaled(cfg, I.make_params(cfg, 0), scale)
    for fr in frames():
        v = {}
        for prec in ("fp64", "tf32"):
            m = dpgb.Model(cfg, p, precision=prec)
            v[prec] = m.compute(fr.coord, fr.atype, fr.box)[2]
            m.free()
        assert np.abs(v["tf32"] - v["fp64"]).max() <= 5e-2 * np.abs(v["fp64"]).max()
