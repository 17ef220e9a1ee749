"""The moment kernels (csrc/mom.cu) at the longest lists they take, 512 slots: the run lists of a tile fill 32 KB beside the
operand rings (forward six stages alone and two next to another frame, or two both times at 128 outputs; backward
three).  The profile says that these kernels ran.

Ring depths change no operation and no order, so atomic energies alone and in the batch are equal to the last bit and
forces to the order of their FP64 sums (1e-12).  Against FP64 compressed the three-pass forces agree to 2e-3 of the
largest, as in test_gpu_mom_ring.py; the one-pass operands have 8 bits fewer, 256 times that bound is no check, so the
mixed mode is compared with itself only.  One slot more and the model takes the tabulated kernels.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _model(sel, embed, prec):
    from paper_2304_09409_gb300 import dpgb
    cfg = I.ModelConfig(ntypes=2, rcut=6.0, rcut_smth=0.5, sel=sel, embed=embed, axis=16, fit=(64, 64))
    return dpgb.Model(cfg, I.make_params(cfg, 5), precision=prec, compressed=True)


def _run(m, fr, copies):
    from paper_2304_09409_gb300 import dpgb
    m.profile(True)
    out = dpgb.compute_batch(m, np.full(copies, fr.natoms, dtype=np.int32), np.concatenate([fr.coord] * copies),
                             np.concatenate([fr.atype] * copies).astype(np.int32), np.stack([fr.box] * copies),
                             atom_energy=True)
    return out[1], out[3], m.profile_read()


@pytest.mark.parametrize("embed", [(25, 50, 100), (32, 64, 128)])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_longest_lists(embed, prec):
    sel = (170, 342)
    fr = I.replicate(I.water_frame(2), (3, 3, 2))
    fr = I.Frame(fr.coord[:-5].copy(), fr.atype[:-5].copy(), fr.box)  # ragged tiles of both types
    n = fr.natoms
    m = _model(sel, embed, prec)
    f1, a1, prof = _run(m, fr, 1)
    f2, a2, _ = _run(m, fr, 2)
    m.free()
    assert "mom_fwd" in prof and "mom_bwd" in prof
    fmax = np.abs(f1).max()
    assert np.array_equal(a2[:n], a1) and np.array_equal(a2[n:], a1)
    assert np.abs(f2[:n] - f1).max() <= 1e-12 * fmax and np.abs(f2[n:] - f1).max() <= 1e-12 * fmax
    if prec == "fp32":
        ref = _model(sel, embed, "fp64")
        f0, _, _ = _run(ref, fr, 1)
        ref.free()
        assert np.abs(f1 - f0).max() <= 2e-3 * np.abs(f0).max()


def test_one_slot_more():
    m = _model((170, 343), (25, 50, 100), "fp32")
    _, _, prof = _run(m, I.water_frame(0), 1)
    m.free()
    assert "mom_fwd" not in prof


def test_one_pass_kernels_keep_three_blocks_an_sm(tmp_path):
    """The mixed mode's moment kernels on the water lists (138 slots) leave shared memory for three blocks an SM (228 KB,
    1 KB of them per block taken by the system)."""
    import json
    import os

    from torch.profiler import ProfilerActivity, profile

    from paper_2304_09409_gb300 import dpgb
    cfg, fr = I.water_model(), I.water_frame(0)
    m = dpgb.Model(cfg, I.make_params(cfg, 0), precision="bf16", compressed=True)
    c, t = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    path, used = os.path.join(str(tmp_path), "trace.json"), {}
    for _ in range(3):  # a process's first trace can come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            m.compute(c, t, fr.box)
            torch.cuda.synchronize()
        prof.export_chrome_trace(path)
        with open(path) as f:
            for e in json.load(f)["traceEvents"]:
                if "k_mom_fwd" in e.get("name", "") or "k_mom_bwd" in e.get("name", ""):
                    used[e["name"].split("<")[0].split("::")[-1]] = e["args"]["shared memory"]
        if used:
            break
    m.free()
    if not used:
        pytest.skip("the profiler gives no kernel records here")
    assert set(used) == {"k_mom_fwd", "k_mom_bwd"}
    assert all(3 * (b + 1024) <= 228 * 1024 for b in used.values()), used
