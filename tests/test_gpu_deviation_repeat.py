"""Model deviation again and again on one ensemble.  Every call takes its forces and virials from a fresh stream-ordered
allocation, and each model records its pass as a graph on the second call and replays it from the third, so a replay
runs on addresses that were freed and allocated again.  Same inputs: results equal to the order of FP64 additions
(taken as 1e-9 of the largest: the spread is a difference of forces).
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,compressed", [("fp64", False), ("fp32", True)])
@pytest.mark.parametrize("device", [False, True])
def test_repeated_deviation(precision, compressed, device):
    from paper_2304_09409_gb300 import dpgb
    cfg = I.water_model()
    models = [dpgb.Model(cfg, I.force_scaled(cfg, I.make_params(cfg, s), I.WATER_FORCE_SCALE), precision=precision,
                         compressed=compressed) for s in range(3)]
    frames = [I.water_frame(3), I.replicate(I.water_frame(4), (2, 1, 1))]
    first = {}
    for k in range(12):
        q = 0 if k < 7 else k % 2  # seven calls of one shape, then two shapes in turn
        fr = frames[q]
        c = torch.tensor(fr.coord, device="cuda") if device else fr.coord
        t = torch.tensor(fr.atype, device="cuda") if device else fr.atype
        out = [x.cpu().numpy() if device else x for x in dpgb.model_deviation(models, c, t, fr.box)]
        out = [np.array(x) for x in out]
        for x, y in zip(out, first.setdefault(q, out)):
            assert np.abs(x - y).max() <= 1e-9 * np.abs(y).max()
    for m in models:
        m.free()
