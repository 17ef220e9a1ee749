"""Which cell grid the neighbour search of a frame takes: half-width cells where whole ones fit the box badly, by a line that
is higher where half-width cells hold fewer than four atoms and are more than four an SM (csrc/nlist.cu, host_geometry).
The grid is read from the launch of the cell-centred search, which has a block column per cell; the lists themselves are
checked elsewhere.
"""
import json
import os

import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _water(n):
    return I.replicate(I.water_frame_n(1, 3), (n, n, n))


# model, sides, cells along x * y * z: metal boxes of 1.8, 2.3, 5.0 and 7.7 cutoffs, water boxes of 1.5 to 6.7
CASES = [("metal", 4, 3 ** 3), ("metal", 5, 2 ** 3), ("metal", 11, 9 ** 3), ("metal", 17, 15 ** 3),
         ("water", 3, 3 ** 3), ("water", 4, 2 ** 3), ("water", 5, 5 ** 3), ("water", 7, 7 ** 3), ("water", 9, 4 ** 3), ("water", 13, 6 ** 3)]


@pytest.mark.parametrize("name,n,cells", CASES)
def test_grid(name, n, cells, tmp_path):
    from torch.profiler import ProfilerActivity, profile

    from paper_2304_09409_gb300 import dpgb
    cfg = I.metal_model() if name == "metal" else I.water_model()
    fr = I.fcc_frame((n, n, n), seed=1) if name == "metal" else _water(n)
    m = dpgb.Model(cfg, I.make_params(cfg, 0), precision="fp32", compressed=True)
    c, t = torch.tensor(fr.coord, device="cuda"), torch.tensor(fr.atype, device="cuda")
    path, grids = os.path.join(str(tmp_path), "trace.json"), []
    for _ in range(3):  # a process's first trace can come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            nl = m.build_nlist(c, t, fr.box)
            torch.cuda.synchronize()
        nl.free()
        prof.export_chrome_trace(path)
        with open(path) as f:
            grids = [e["args"]["grid"] for e in json.load(f)["traceEvents"] if "k_nlist_cell" in e.get("name", "")]
        if grids:
            break
    m.free()
    if not grids:
        pytest.skip("the profiler gives no kernel records here")
    assert [g[0] for g in grids] == [cells]
