"""The three-pass moment kernels (csrc/mom.cu) at every ring depth and schedule: six forward stages (fewer
tiles than SMs), three (two blocks share an SM), two (long lists); four, three and two backward stages; and
the schedule from the run masks or, with tables of more than 256 intervals (small r_s) and lists of more than
1,024 slots, the plain one.

The depth changes no operation and no order, so a frame alone (six stages) and the same frame next to another
(three or two) have the same atomic energies to the last bit, and forces to the order of their FP64 sums
(1e-12).  Against FP64 compressed the forces agree to 2e-3 of the largest, as in test_gpu_fit_split.py.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sel, rcut_smth", [
    ((46, 92), 0.5),
    ((150, 350), 0.5),
    ((46, 92), 0.3),
    ((500, 540), 0.5),
])
def test_mom_rings(sel, rcut_smth):
    from paper_2304_09409_gb300 import dpgb
    cfg = I.ModelConfig(ntypes=2, rcut=6.0, rcut_smth=rcut_smth, sel=sel, embed=(25, 50, 100), axis=16,
                        fit=(240, 240, 240))
    p = I.make_params(cfg, 5)
    fr = I.replicate(I.water_frame(2), (3, 3, 2))
    fr = I.Frame(fr.coord[:-5].copy(), fr.atype[:-5].copy(), fr.box)  # ragged tiles of both types
    n = len(fr.atype)

    def run(prec, copies):
        m = dpgb.Model(cfg, p, precision=prec, compressed=True)
        out = dpgb.compute_batch(m, np.full(copies, n, dtype=np.int32), np.concatenate([fr.coord] * copies),
                                 np.concatenate([fr.atype] * copies).astype(np.int32), np.stack([fr.box] * copies),
                                 atom_energy=True)
        m.free()
        return out[1], out[3]

    f0, _ = run("fp64", 1)
    f1, a1 = run("fp32", 1)
    f2, a2 = run("fp32", 2)
    fmax = np.abs(f0).max()
    print(f"sel {sel}, r_s {rcut_smth}, {n} atoms: |dF|/|F|max {np.abs(f1 - f0).max() / fmax:.1e} against FP64, "
          f"{np.abs(f2[n:] - f1).max() / fmax:.1e} next to another frame")
    assert np.abs(f1 - f0).max() <= 2e-3 * fmax
    assert np.array_equal(a2[:n], a1) and np.array_equal(a2[n:], a1)
    assert np.abs(f2[:n] - f1).max() <= 1e-12 * fmax and np.abs(f2[n:] - f1).max() <= 1e-12 * fmax
