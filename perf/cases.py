"""The performance cases of the framework, each one call as a user's program makes it.

listed() names them, draw() gives more of the same ranges, prepare() builds what a program holds before
the call (a resident model, coordinates and types on the GPU, the cell on the host), run() is one pass
through the public entry points and work() counts what that pass cannot do without.  exact() evaluates the
same inputs with the plain FP64 torch code at the end of this file, which uses nothing of the library.
"""
import functools
import math

import numpy as np
import torch

from paper_2304_09409_gb300 import dpgb
from paper_2304_09409_gb300 import inputs as I
from paper_2304_09409_gb300.autograd import DPForce, efv_loss

WATER_SPACING = 3.105  # A between O sites: 1 g/cm^3
SERVE_BATCH_ATOMS = 65536  # the server's batch budget
# Energies per atom (eV, by type) of the seed-0 water model at unit force scale: training labels lie
# near the model's own energies, as they do once a data set's energy bias has been set.
WATER_ATOM_ENERGY = (0.311535, -1.809837)

MODELS = {
    "water": (I.water_model, I.WATER_FORCE_SCALE),
    "metal": (I.metal_model, I.METAL_FORCE_SCALE),
    "water_r": (I.water_model_r, I.WATER_R_FORCE_SCALE),
    "water_hybrid": (I.water_model_hybrid, I.WATER_HYBRID_FORCE_SCALE),
    "water_e3": (I.water_model_e3, I.WATER_E3_FORCE_SCALE),
    "water_hybrid_e3": (I.water_model_hybrid_e3, I.WATER_HYBRID_E3_FORCE_SCALE),
}


def listed():
    return [
        # Molecular dynamics with the production mode (FP32 arithmetic, compressed embedding): one step
        # of the smallest benchmark box, where the latency of the call decides.
        {"name": "md_water_192", "kind": "md", "model": "water", "precision": "fp32", "compressed": True,
         "nx": 4, "ny": 4, "nz": 4, "tilt": 0.0},
        # A mid-size odd box: the step of a typical liquid simulation.
        {"name": "md_water_2145", "kind": "md", "model": "water", "precision": "fp32", "compressed": True,
         "nx": 5, "ny": 11, "nz": 13, "tilt": 0.0},
        # The benchmark's box of 12,288 atoms.
        {"name": "md_water_12288", "kind": "md", "model": "water", "precision": "fp32", "compressed": True,
         "nx": 16, "ny": 16, "nz": 16, "tilt": 0.0},
        # The benchmark's metal crystal of 32,000 atoms (r_c 8, ~180 neighbours).
        {"name": "md_metal_32000", "kind": "md", "model": "metal", "precision": "fp32", "compressed": True,
         "nx": 20, "ny": 20, "nz": 20, "tilt": 0.0},
        # The server at saturation: one batch of uneven water and metal frames of two resident models.
        {"name": "serve_mixed_16", "kind": "serve", "precision": "fp32", "compressed": True, "frames": 16, "mix": 9},
        # The BF16 mixed mode (compressed), on an odd box.
        {"name": "md_water_bf16_8190", "kind": "md", "model": "water", "precision": "bf16", "compressed": True,
         "nx": 13, "ny": 14, "nz": 15, "tilt": 0.0},
        # The reference mode, FP64 networks, on the smallest benchmark box (validation of a model).
        {"name": "md_water_fp64_192", "kind": "md", "model": "water", "precision": "fp64", "compressed": False,
         "nx": 4, "ny": 4, "nz": 4, "tilt": 0.0},
        # The precision sweep's TF32 networks on the metal crystal, as sheared cells of a data set are.
        {"name": "md_metal_tf32_8736", "kind": "md", "model": "metal", "precision": "tf32", "compressed": False,
         "nx": 12, "ny": 13, "nz": 14, "tilt": 0.06},
        # A training step's batch: forward, the loss with its virial term, and the parameter gradient.
        {"name": "train_water_32x192", "kind": "train", "frames": 32, "nx": 4, "ny": 4, "nz": 4},
        # FP32 networks, as a model is run between training and compression.
        {"name": "md_water_fp32_nets_1029", "kind": "md", "model": "water", "precision": "fp32", "compressed": False,
         "nx": 7, "ny": 7, "nz": 7, "tilt": 0.0},
        # The three-body descriptor.
        {"name": "md_water_e3_12288", "kind": "md", "model": "water_e3", "precision": "fp32", "compressed": False,
         "nx": 16, "ny": 16, "nz": 16, "tilt": 0.0},
        # A hybrid descriptor with FP32 networks (two-body part with r_c 4, radial part with r_c 6).
        {"name": "md_water_hybrid_4116", "kind": "md", "model": "water_hybrid", "precision": "fp32", "compressed": False,
         "nx": 7, "ny": 14, "nz": 14, "tilt": 0.0},
    ]


def draw(rng):
    """One more case: a kind, then its sizes spread over the logarithm of the atom count."""

    def sides(lo, hi, per):
        """Three sides with lo <= per * product <= hi, none more than about three times another."""
        while True:
            n = math.exp(rng.uniform(math.log(lo), math.log(hi))) / per
            s = [max(2, round(n ** (1 / 3) * math.exp(rng.uniform(-0.35, 0.35)))) for _ in range(3)]
            if lo <= per * s[0] * s[1] * s[2] <= hi:
                return dict(zip(("nx", "ny", "nz"), s))

    def md(model, precision, compressed, hi, lo=24):
        per = 4 if model == "metal" else 3
        if model == "metal":
            lo = max(lo, 108)
        tilt = rng.choice((0.0, 0.0, 0.03, 0.08))
        return dict(kind="md", model=model, precision=precision, compressed=compressed, tilt=tilt, **sides(lo, hi, per))

    kind = rng.choice(("md_water", "md_water", "md_metal", "md_metal", "serve", "bf16", "fp64", "nets", "train", "other"))
    if kind == "md_water":
        return md("water", "fp32", True, 32000)
    if kind == "md_metal":
        return md("metal", "fp32", True, 32000)
    if kind == "bf16":
        return md(rng.choice(("water", "metal")), "bf16", True, 12288)
    if kind == "fp64":
        return md("water", "fp64", rng.random() < 0.5, 384)
    if kind == "nets":
        model, precision = rng.choice(("water", "metal")), rng.choice(("fp32", "tf32", "bf16"))
        return md(model, precision, False, 3000 if precision == "fp32" else 8736)
    if kind == "other":
        model = rng.choice(("water_r", "water_hybrid", "water_e3", "water_hybrid_e3"))
        return md(model, "fp32", model in ("water_r", "water_e3") and rng.random() < 0.5,
                  4116 if "hybrid" in model else 12288)
    if kind == "serve":
        return dict(kind="serve", precision="fp32", compressed=True, frames=rng.randint(1, 16), mix=rng.randrange(1 << 30))
    size = sides(24, 648, 3)
    return dict(kind="train", frames=rng.randint(1, min(32, 6144 // (3 * size["nx"] * size["ny"] * size["nz"]))), **size)


# ---- inputs ---------------------------------------------------------------------------------------

def _rng(*key):
    return np.random.default_rng([int(k) for k in key])


def _water(nx, ny, nz, seed, tilt=0.0):
    """Water-like frame: O on a lattice with +-0.2 A jitter, two H at 0.96 A and 104.52 degrees."""
    g = _rng(seed, nx, ny, nz)
    n = nx * ny * nz
    site = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1).reshape(-1, 3)
    o = site * WATER_SPACING + g.uniform(-0.2, 0.2, (n, 3))
    u = g.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    w = np.cross(u, g.normal(size=(n, 3)))
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    a = math.radians(I.HOH_ANGLE_DEG)
    coord = np.stack([o, o + I.OH_BOND * u, o + I.OH_BOND * (math.cos(a) * u + math.sin(a) * w)], axis=1)
    box = np.diag(np.array([nx, ny, nz]) * WATER_SPACING)
    return _shear(I.Frame(coord.reshape(-1, 3), np.tile(np.array([0, 1, 1], dtype=np.int32), n), box), tilt)


def _metal(nx, ny, nz, seed, tilt=0.0):
    return _shear(I.fcc_frame((nx, ny, nz), seed=seed), tilt)


def _shear(fr, tilt):
    """The frame under a small simple shear of its cell (x along y, y along z)."""
    if not tilt:
        return fr
    m = np.array([[1.0, 0.0, 0.0], [tilt, 1.0, 0.0], [0.0, 0.5 * tilt, 1.0]])
    return I.Frame(fr.coord @ m, fr.atype, fr.box @ m)


def _sizes(case):
    """Model and sides of every frame of a served batch: as the benchmark's stream, water of 24 to 3,000 and
    metal of 108 to about 20,000 atoms with equal chance, taken oldest first up to the batch budget."""
    g = _rng(case["mix"])
    out, total = [], 0
    for k in range(case["frames"]):
        if g.random() < 0.5:
            s = [int(v) for v in g.integers(2, 11, 3)]
            name, n = "water", 3 * s[0] * s[1] * s[2]
        else:
            s = [int(v) for v in g.integers(3, 18, 3)]
            name, n = "metal", 4 * s[0] * s[1] * s[2]
        if total + n > SERVE_BATCH_ATOMS:
            break
        out.append((name, s))
        total += n
    return sorted(out, key=lambda x: x[0] != "water")  # a batch lists each model's frames together


def _frames(case, seed):
    """(model name, Frame) of every frame of the case."""
    if case["kind"] == "serve":
        sizes = _sizes(case)
    else:
        name = case.get("model", "water")
        sizes = [(name, (case["nx"], case["ny"], case["nz"]))] * case.get("frames", 1)
    make = {"water": _water, "metal": _metal}
    return [(name, make[name.split("_")[0]](*s, seed * 64 + k, case.get("tilt", 0.0))) for k, (name, s) in enumerate(sizes)]


@functools.lru_cache(maxsize=None)
def _weights(name):
    make, scale = MODELS[name]
    return I.force_scaled(make(), I.make_params(make(), 0), scale)


def _labels(frames, seed):
    """Training labels: forces of 1 eV/A, energies and virials a few eV off."""
    g = _rng(seed, 77)
    per = np.array(WATER_ATOM_ENERGY) * I.WATER_FORCE_SCALE
    e = np.array([per[fr.atype].sum() for fr in frames]) + g.normal(size=len(frames)) * 5.0
    f = g.normal(size=(sum(fr.natoms for fr in frames), 3))
    v = g.normal(size=(len(frames), 3, 3)) * 20.0
    return e, f, v + v.transpose(0, 2, 1)


PREFACTORS = (0.02, 100.0, 0.02)  # p_E, p_F, p_Xi early in a training run


def prepare(case, seed):
    frames = _frames(case, seed)
    s = {"kind": case["kind"], "natoms": np.array([fr.natoms for _, fr in frames], dtype=np.int32),
         "coord": torch.tensor(np.concatenate([fr.coord for _, fr in frames]), device="cuda"),
         "atype": torch.tensor(np.concatenate([fr.atype for _, fr in frames]), device="cuda"),
         "boxes": np.stack([fr.box for _, fr in frames])}
    if case["kind"] == "md":
        s["model"] = dpgb.Model(MODELS[case["model"]][0](), _weights(case["model"]), precision=case["precision"],
                                compressed=case["compressed"])
    elif case["kind"] == "serve":
        s["model"] = [dpgb.Model(MODELS[n][0](), _weights(n), precision=case["precision"], compressed=case["compressed"])
                      for n in ("water", "metal")]
        s["frame_model"] = np.array([0 if n == "water" else 1 for n, _ in frames], dtype=np.int32)
    else:
        s["model"] = dpgb.Model(I.water_model(), _weights("water"), precision="fp32")
        s["params"] = torch.tensor(_weights("water"), device="cuda").requires_grad_()
        s["labels"] = [torch.tensor(x, device="cuda") for x in _labels([fr for _, fr in frames], seed)]
    return s


def run(s):
    if s["kind"] == "md":
        return s["model"].compute(s["coord"], s["atype"], s["boxes"][0])[:3]
    if s["kind"] == "serve":
        return dpgb.compute_batch(s["model"], s["natoms"], s["coord"], s["atype"], s["boxes"],
                                  frame_model=s["frame_model"])[:3]
    e, f, v = DPForce.apply(s["params"], s["model"], s["natoms"], s["coord"], s["atype"], s["boxes"])
    loss = efv_loss(e, f, v, *s["labels"], s["natoms"], *PREFACTORS)
    (grad,) = torch.autograd.grad(loss, s["params"])
    return e.detach(), f.detach(), v.detach(), grad


# ---- what a pass cannot do without ------------------------------------------------------------------

def work(case):
    sizes = _sizes(case) if case["kind"] == "serve" else [(case.get("model", "water"), (case["nx"], case["ny"], case["nz"]))]
    natoms = {}
    for name, s in sizes:
        natoms[name] = natoms.get(name, 0) + s[0] * s[1] * s[2] * (4 if name == "metal" else 3) * case.get("frames", 1) ** (case["kind"] == "train")
    total_b = total_f = 0.0
    wide = 8 if case.get("precision", "fp32") == "fp64" else 2 if case.get("precision") == "bf16" else 4
    for name, n in natoms.items():
        cfg = MODELS[name][0]()
        density = 4 / 3.634 ** 3 if name == "metal" else 3 / WATER_SPACING ** 3
        mul = lambda shapes: 2 * sum(a * b for a, b in shapes)  # noqa: E731
        per_atom, nbr = 2 * mul(cfg.fit_layer_shapes()), density * 4 / 3 * math.pi * cfg.rcut ** 3
        nets = cfg.embed_layer_shapes()
        if cfg.descriptor in (0, 2, 4):
            embed = 10 * cfg.m if case.get("compressed", False) else mul(nets)
            per_atom += 2 * nbr * (embed + 8 * cfg.m) + 2 * (8 * cfg.m * cfg.axis)
        if cfg.descriptor == 1:
            per_atom += 2 * nbr * (mul(nets) + 2 * cfg.m)
        if cfg.hybrid:
            nbr_2 = density * 4 / 3 * math.pi * cfg.list_rcut ** 3
            pairs = nbr_2 if cfg.descriptor == 2 else nbr_2 * nbr_2 / 2
            per_atom += 2 * pairs * (mul(cfg.embed_2_layer_shapes()) + 2 * cfg.embed_2[-1])
        if cfg.descriptor == 3:
            per_atom += 2 * nbr * nbr / 2 * (mul(nets) + 2 * cfg.m + 8)
        passes = 4 if case["kind"] == "train" else 1  # tangent and reverse double a gradient's work
        weights = cfg.n_params() - (cfg.embed_params() if case.get("compressed", False) else 0)
        total_f += passes * n * per_atom
        total_b += n * (24 + 4 + 24) + weights * wide + (cfg.n_params() * 16 if case["kind"] == "train" else 0)
    return {"bytes": total_b, "flops": total_f}


# ---- the same in plain torch, FP64 ------------------------------------------------------------------

def _neighbours(coord, atype, box, rcut, sel):
    """The sel[t] nearest neighbours of every atom: index [N, sum(width)], displacement base, type blocks."""
    inv = torch.linalg.inv(box)
    heights = 1.0 / torch.linalg.norm(inv, dim=0)
    frac = coord @ inv
    wrapped = (frac - torch.floor(frac)) @ box
    reach = [int(math.ceil(rcut / float(h))) for h in heights]
    n = torch.cartesian_prod(*[torch.arange(-r, r + 1, device=coord.device) for r in reach]).to(coord.dtype)
    f = (frac - torch.floor(frac))[None] + n[:, None]
    pad = rcut / heights
    keep = ((f >= -pad) & (f <= 1 + pad)).all(-1)
    which, src = torch.nonzero(keep, as_tuple=True)
    pos = f[which, src] @ box
    home = (n[which] == 0).all(-1)
    blocks = []
    for t, width in enumerate(sel):
        m = atype[src] == t
        p, j, h = pos[m], src[m], home[m]
        rows_j, rows_r = [], []
        for i0 in range(0, coord.shape[0], 256):
            c = wrapped[i0:i0 + 256]
            r2 = sum((p[None, :, k] - c[:, None, k]) ** 2 for k in range(3))
            me = torch.arange(i0, i0 + c.shape[0], device=coord.device)
            r2.masked_fill_((r2 >= rcut * rcut) | ((j[None] == me[:, None]) & h[None]), math.inf)
            k = min(width, p.shape[0])
            near, at = torch.topk(r2, k, dim=1, largest=False)
            rows_j.append(torch.where(torch.isinf(near), -1, j[at]))
            rows_r.append(torch.where(torch.isinf(near)[..., None], torch.zeros_like(p[at]), p[at] - c[:, None]))
        full = max(1, max(int((r >= 0).sum(1).max()) for r in rows_j))
        blocks.append((torch.cat([r[:, :full] for r in rows_j]), torch.cat([r[:, :full] for r in rows_r])))
    return blocks


def _net(x, layers, jets=None):
    """Eq. (NN) hidden layers; with jets (x', x'') also the first two derivatives."""
    for w, b in layers:
        t = torch.tanh(x @ w + b)
        skip = (lambda q: 0.0) if w.shape[1] not in (w.shape[0], 2 * w.shape[0]) else \
            (lambda q: q) if w.shape[1] == w.shape[0] else (lambda q: torch.cat([q, q], -1))
        if jets is not None:
            z1, z2, gate = jets[0] @ w, jets[1] @ w, 1 - t * t
            jets = (gate * z1 + skip(jets[0]), gate * z2 - 2 * t * gate * z1 * z1 + skip(jets[1]))
        x = t + skip(x)
    return x if jets is None else (x,) + jets


def _table(layers, top):
    """Quintic pieces of Eq. (compress) on [0, top]: fine on the first 90 %, ten times wider after."""
    h = top / 200
    nodes = torch.cat([torch.arange(181) * h, 180 * h + 10 * h * torch.arange(1, 3)]).to(layers[0][0])
    y, y1, y2 = _net(nodes[:, None], layers, (torch.ones_like(nodes)[:, None], torch.zeros_like(nodes)[:, None]))
    d, w = y[1:] - y[:-1], (nodes[1:] - nodes[:-1])[:, None]
    a0, a1, c0, c1 = y1[:-1], y1[1:], y2[:-1], y2[1:]
    return nodes, torch.stack([
        y[:-1], a0, c0 / 2,
        (20 * d - (8 * a1 + 12 * a0) * w - (3 * c0 - c1) * w ** 2) / (2 * w ** 3),
        (-30 * d + (14 * a1 + 16 * a0) * w + (3 * c0 - 2 * c1) * w ** 2) / (2 * w ** 4),
        (12 * d - 6 * (a1 + a0) * w + (c1 - c0) * w ** 2) / (2 * w ** 5)])


def _embed(x, net):
    if isinstance(net, list):
        return _net(x[..., None], net)
    nodes, coef = net
    at = torch.clamp(torch.searchsorted(nodes, x.detach().contiguous(), right=True) - 1, 0, coef.shape[1] - 1)
    t = (x - nodes[at])[..., None]
    out = coef[5][at]
    for p in range(4, -1, -1):
        out = out * t + coef[p][at]
    return out


class _Reference:
    """E, F and Xi of one model in FP64, as functions of the flat parameters."""

    def __init__(self, cfg, params, compressed=False):
        self.cfg, self.at, self.p = cfg, 0, params
        kind = cfg.descriptor
        self.parts = [dict(e3=kind == 3, r=kind == 1, rcut=cfg.rcut, rs=cfg.rcut_smth, sel=cfg.sel,
                           nets=[self._take(cfg.embed_layer_shapes()) for _ in range(cfg.n_embed_nets)])]
        if cfg.hybrid:
            self.parts.append(dict(e3=kind == 4, r=kind == 2, rcut=cfg.rcut_2, rs=cfg.rcut_smth_2, sel=cfg.sel_2,
                                   nets=[self._take(cfg.embed_2_layer_shapes()) for _ in range(cfg.n_embed_nets_2)]))
        if compressed:
            for p in self.parts:
                p["nets"] = [_table(net, 2.0 / p["rs"] ** 2 if p["e3"] else 1.0 / p["rs"]) for net in p["nets"]]
        self.fit = [self._take(cfg.fit_layer_shapes()) for _ in range(cfg.ntypes)]

    def _take(self, shapes):
        layers = []
        for a, b in shapes:
            w, self.at = self.p[self.at:self.at + a * b].reshape(a, b), self.at + a * b
            c, self.at = self.p[self.at:self.at + b], self.at + b
            layers.append((w, c))
        return layers

    def _descriptor(self, part, t, blocks, rij):
        cfg, nt, nc = self.cfg, self.cfg.ntypes, sum(part["sel"])
        rows = []
        for (j, _), d in zip(blocks, rij):
            real = j >= 0
            r = torch.sqrt(torch.where(real, (d * d).sum(-1), torch.ones_like(d[..., 0])))
            x = (r - part["rs"]) / (part["rcut"] - part["rs"])
            u = torch.where(x < 0, torch.ones_like(x), x ** 3 * (-6 * x * x + 15 * x - 10) + 1)
            s = torch.where(real, u / r, torch.zeros_like(r))
            rows.append(torch.cat([s[..., None], (s / r)[..., None] * d], -1))
        if part["e3"]:
            out = 0.0
            for a, ra in enumerate(rows):
                for b, rb in enumerate(rows):
                    th = ra @ rb.transpose(1, 2)
                    out = out + (th[..., None] * _embed(th, part["nets"][a * nt + b])).sum((1, 2))
            return out / nc ** 2
        gr = 0.0
        for b, rb in enumerate(rows):
            g = _embed(rb[..., 0], part["nets"][b if cfg.type_one_side else t * nt + b])
            gr = gr + g.transpose(1, 2) @ (rb[..., :1] if part["r"] else rb)
        gr = gr / nc
        return gr[..., 0] if part["r"] else (gr @ gr[:, :cfg.axis].transpose(1, 2)).flatten(1)

    def __call__(self, fr, chunk, graph=False):
        """(E [1], F [N, 3], Xi [3, 3]); with graph=True they stay functions of the parameters."""
        dev = self.p.device
        coord, atype = torch.tensor(fr.coord, device=dev), torch.tensor(fr.atype, device=dev).long()
        box = torch.tensor(fr.box, device=dev)
        lists = [_neighbours(coord, atype, box, p["rcut"], p["sel"]) for p in self.parts]
        e, f, v = torch.zeros(1, device=dev, dtype=coord.dtype), torch.zeros_like(coord), torch.zeros_like(box)
        for t in range(self.cfg.ntypes):
            for i in torch.nonzero(atype == t)[:, 0].split(chunk):
                blocks = [[(j[i], d[i]) for j, d in lst] for lst in lists]
                rij = [[d.clone().requires_grad_() for _, d in b] for b in blocks]
                x = torch.cat([self._descriptor(p, t, b, r) for p, b, r in zip(self.parts, blocks, rij)], -1)
                x = _net(x, self.fit[t][:-1]) @ self.fit[t][-1][0] + self.fit[t][-1][1]
                flat = [d for r in rij for d in r]
                grads = torch.autograd.grad(x.sum(), flat, create_graph=graph)
                e = e + (x.sum() if graph else x.sum().detach())
                for (j, _), d, g in zip([q for b in blocks for q in b], flat, grads):
                    f = f.index_add(0, i, g.sum(1))
                    f = f.index_add(0, j.clamp(min=0).flatten(), -torch.where((j >= 0)[..., None], g, 0.0 * g).flatten(0, 1))
                    v = v - g.flatten(0, 1).T @ d.detach().flatten(0, 1)
        return e, f, v


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    frames = _frames(case, seed)
    if case["kind"] == "train":
        params = torch.tensor(_weights("water"), device=dev).requires_grad_()
        le, lf, lv = [torch.tensor(x, device=dev) for x in _labels([fr for _, fr in frames], seed)]
        pe, pf, pv = PREFACTORS
        out, at, grad = [], 0, torch.zeros_like(params)
        for k, (_, fr) in enumerate(frames):
            n = fr.natoms
            e, f, v = _Reference(I.water_model(), params)(fr, 1024, graph=True)
            loss = (pe * (e[0] - le[k]) ** 2 / n + pf * ((f - lf[at:at + n]) ** 2).sum() / (3 * n)
                    + pv * ((v - lv[k]) ** 2).sum() / (9 * n)) / len(frames)
            grad += torch.autograd.grad(loss, params)[0]
            out.append((e.detach(), f.detach(), v.detach()))
            at += n
        return torch.cat([e for e, _, _ in out]), torch.cat([f for _, f, _ in out]), torch.stack([v for _, _, v in out]), grad
    chunk = 48 if "e3" in case.get("model", "") else 1024
    refs = {name: _Reference(MODELS[name][0](), torch.tensor(_weights(name), device=dev), case["compressed"])
            for name, _ in frames}
    res = [refs[name](fr, chunk) for name, fr in frames]
    if case["kind"] == "md":
        return res[0]
    return torch.cat([r[0] for r in res]), torch.cat([r[1] for r in res]), torch.stack([r[2] for r in res])
