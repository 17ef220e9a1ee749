"""The parameter gradient with force and virial seeds at the widths and row counts of test_gpu_dense.py, where a tile, a K
chunk, a row list or a row slab of the tangent layers ends unevenly: FP64 against central differences of the FP64 path's
own sum(ge E) + sum(gf F) + sum(gv Xi), layer by layer, and FP32 against FP64.

Central differences at h = 1e-4 along a unit direction that weights a layer's parameters by their own gradient: the
truncation is h^2 / 6 times the third derivative, allowed a hundred times the gradient there (2e-7), taken with a factor
of fifty (1e-5 of the layer's gradient); the forces' FP64 rounding (about 1e-13 each) over 2 h adds 1e-9 sqrt(3 N), taken
with a factor of ten.  FP32 as in test_gpu_dense.py, 2e-3 of the gradient's norm.
"""
import numpy as np
import pytest

from paper_2304_09409_gb300 import inputs as I

from test_gpu_dense import CASES, _dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _layers(cfg):
    """Index arrays of the parameters of every layer (embedding layer l of all nets, fitting layer l of all types)."""
    emb, fit = cfg.embed_layer_shapes(), cfg.fit_layer_shapes()
    out, at = [[] for _ in emb + fit], 0
    for count, shapes, first in ((cfg.ntypes if cfg.type_one_side else cfg.ntypes ** 2, emb, 0), (cfg.ntypes, fit, len(emb))):
        for _ in range(count):
            for l, (a, b) in enumerate(shapes):
                out[first + l].append(np.arange(at, at + (a + 1) * b))
                at += (a + 1) * b
    return [np.concatenate(x) for x in out], at


@pytest.mark.parametrize("name", list(CASES))
def test_force_and_virial_seeds(name):
    from paper_2304_09409_gb300 import dpgb
    cfg, make = CASES[name]
    fr, p = make(), I.make_params(cfg, 1)
    c, t = _dev(fr)
    nat = np.array([fr.natoms], dtype=np.int32)
    rng = np.random.default_rng(11)
    ge, gf, gv = np.array([0.3]), rng.normal(size=(fr.natoms, 3)), rng.normal(size=(1, 3, 3))
    layers, total = _layers(cfg)
    assert total == p.size
    m = dpgb.Model(cfg, p, precision="fp64")

    def value(q):
        m.set_params(q)
        e, f, v, _ = m.compute(c, t, fr.box)
        return float(ge[0] * e.cpu()[0]) + float((f.cpu().numpy() * gf).sum()) + float((v.cpu().numpy() * gv[0]).sum())

    g = dpgb.param_grad(m, nat, c, t, fr.box[None], ge, gf, g_virial=gv).cpu().numpy()
    h = 1e-4
    for idx in layers:
        d = np.zeros_like(p)
        d[idx] = g[idx] * rng.uniform(0.5, 1.5, idx.size)
        norm = np.linalg.norm(d)
        if norm == 0.0:
            continue
        d /= norm
        fd, an = (value(p + h * d) - value(p - h * d)) / (2 * h), float(g @ d)
        assert abs(fd - an) <= 1e-5 * np.linalg.norm(g[idx]) + 1e-8 * np.sqrt(3 * fr.natoms), (fd, an)
    m.free()
    m = dpgb.Model(cfg, p, precision="fp32")
    g32 = dpgb.param_grad(m, nat, c, t, fr.box[None], ge, gf, g_virial=gv).cpu().numpy()
    m.free()
    assert np.linalg.norm(g32 - g) <= 2e-3 * np.linalg.norm(g)
