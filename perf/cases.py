"""Performance cases of the gamma library: what a user's program calls, over the
range of sizes, criteria and entry points that the library is used with.

A case is a dict of plain values.  Doses are synthetic, with the recipes of
this repository's workloads (sums of Gaussian blobs in 2D, seven coplanar
beams of 10 x 10 beamlets in 3D; the evaluation dose is the shifted, scaled
phantom plus noise), generated on the GPU from the seed.  Every handle keeps
its default options.

  listed()          the cases
  draw(rng)         one more case of the same ranges
  prepare(c, seed)  doses or rows on the GPU (host buffers for the host case),
                    the handle or model, and the outputs
  run(state)        one pass through the public entry points
  work(c)           bytes and FLOPs a pass cannot do without
  exact(c, seed)    the same outputs in 64 bits, from plain torch
"""
import itertools
import math
import os
import struct

import numpy as np
import torch

import paper_1012_1900_gb300 as g

DEV = "cuda"
F64 = torch.float64
MODEL = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                     "paper_1012_1900_gb300", "proposal_2pct2mm.gmlp")
K_IN, K_PAD, K_H, K_OUT, K_OUTPAD = 375, 384, 128, 4, 8      # the network's layers


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def _map(kind, shape, h, dd, dta, local=False, shift=1.5, scale=1.03, **more):
    nz, ny, nx = shape
    return dict(kind=kind, nz=nz, ny=ny, nx=nx, h=h, dd=dd, dta=dta, local=local, shift=shift,
                scale=scale, **more)


def listed():
    cases = [
        # one portal or film plane against its planned dose: the smallest call,
        # a map of a few microseconds of work, where launches count
        ("plane_128", _map("map", (1, 128, 128), 1.0, 0.03, 3.0, shift=0.7, scale=1.02)),
        # a clinical treatment plan at its usual grid and criteria (this
        # library's benchmark workload)
        ("imrt_160", _map("map", (120, 160, 160), 2.5, 0.03, 3.0)),
        # a cropped region of interest: odd extents (rows not 16-byte aligned),
        # tighter criteria
        ("roi_99x113x115", _map("map", (99, 113, 115), 2.0, 0.02, 2.0, shift=2.0, scale=1.02)),
        # a fine grid with a large set-up error: many voxels fail and search far
        ("imrt_320", _map("map", (240, 320, 320), 1.25, 0.03, 3.0, shift=3.0, scale=1.05)),
        # the same with local 1 %/1 mm criteria: the largest call
        ("imrt_320_local", _map("map", (240, 320, 320), 1.25, 0.01, 1.0, local=True, shift=3.0,
                                scale=1.05)),
        # a department's batch: planes and volumes of uneven size and criteria
        # in one batched run
        ("batch_8_8", dict(kind="batch", planes=8, volumes=8, pick=0)),
        # doses on the host (page-locked), as a planning system holds them: map
        # and pass rate back on the host
        ("host_160", _map("host", (120, 160, 160), 2.5, 0.03, 3.0)),
        # Monte Carlo reference on a coarse grid against a fine evaluation grid,
        # half a fine voxel off
        ("grids_160_320", _map("grids", (120, 160, 160), 2.5, 0.03, 3.0, ratio=2.0, offset=0.625)),
        # the search with the committed proposal network attached
        ("learned_200", _map("learned", (150, 200, 200), 2.0, 0.02, 2.0, shift=2.5, scale=1.03)),
        # training rows of one pair: features and labels of sampled voxels
        ("rows_4096", _map("rows", (150, 200, 200), 2.0, 0.02, 2.0, shift=2.5, scale=1.03, rows=4096)),
        # one optimiser step of the proposal network at the training batch
        ("train_8192", dict(kind="train", rows=8192)),
        # the network on its own over a large set of rows
        ("infer_262144", dict(kind="infer", rows=262144)),
    ]
    return [dict(c, name=n) for n, c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plane", "map", "map", "local", "batch", "host", "grids", "learned", "rows",
                       "train", "infer"])
    if kind == "train":
        return dict(kind="train", rows=_log_int(rng, 500, 16384))
    if kind == "infer":
        return dict(kind="infer", rows=_log_int(rng, 1000, 262144))
    if kind == "batch":
        return dict(kind="batch", planes=rng.randint(2, 8), volumes=rng.randint(2, 8),
                    pick=rng.randint(1, 1000))
    dd, dta = rng.choice([(0.01, 1.0), (0.02, 2.0), (0.03, 3.0)])
    shift, scale = round(rng.uniform(0.0, 3.0), 3), round(rng.uniform(0.97, 1.05), 4)
    if kind == "plane":
        return _map("map", (1, _log_int(rng, 64, 512), _log_int(rng, 64, 512)), 1.0, dd, dta,
                    local=rng.random() < 0.3, shift=shift, scale=scale)
    h = rng.choice([1.25, 2.0, 2.5])
    top = {"map": 24.0e6, "local": 8.0e6, "host": 8.0e6, "grids": 3.0e6, "learned": 6.0e6,
           "rows": 6.0e6}[kind]
    while True:
        shape = (_log_int(rng, 24, 240), _log_int(rng, 40, 320), _log_int(rng, 40, 320))
        if shape[0] * shape[1] * shape[2] <= top:
            break
    if kind == "local":
        return _map("map", shape, h, dd, dta, local=True, shift=shift, scale=scale)
    if kind == "grids":
        return _map("grids", shape, 2.5, dd, dta, shift=shift, scale=scale,
                    ratio=rng.choice([1.25, 1.6, 2.0]), offset=round(rng.uniform(0.0, 1.25), 3))
    if kind == "learned":
        return _map("learned", shape, 2.0, 0.02, 2.0, shift=shift, scale=scale)
    if kind == "rows":
        return _map("rows", shape, 2.0, 0.02, 2.0, shift=shift, scale=scale,
                    rows=_log_int(rng, 256, 16384))
    return _map(kind, shape, h, dd, dta, shift=shift, scale=scale)


# ---------------------------------------------------------------------------
# Doses
# ---------------------------------------------------------------------------

def _unit(gen, n):
    return torch.rand(n, generator=gen, dtype=F64).to(DEV)


def _blobs(shape, h, gen, at):
    """Sum of six Gaussian blobs (sigma 8-25 mm, amplitude 0.3-1) at the pixel
    positions moved by at = (dy, dx) mm, for each entry of `at`; scaled so
    that the first one's maximum is 1."""
    ny, nx = shape
    cy, cx = (0.2 + 0.6 * _unit(gen, 6)) * ny * h, (0.2 + 0.6 * _unit(gen, 6)) * nx * h
    sg, amp = 8.0 + 17.0 * _unit(gen, 6), 0.3 + 0.7 * _unit(gen, 6)
    y, x = torch.arange(ny, device=DEV, dtype=F64) * h, torch.arange(nx, device=DEV, dtype=F64) * h
    out = []
    for sy, sx in at:
        ey = torch.exp(-((y[None] - sy - cy[:, None]) ** 2) / (2 * sg[:, None] ** 2))
        ex = torch.exp(-((x[None] - sx - cx[:, None]) ** 2) / (2 * sg[:, None] ** 2))
        out.append(torch.einsum("k,ky,kx->yx", amp, ey, ex))
    top = out[0].max()
    return [o / top for o in out]


def _beam_weights(gen):
    return 0.2 + 0.8 * torch.rand((7, 10, 10), generator=gen, dtype=F64).to(DEV)


def _beams(z, y, x, box, weights):
    """Dose at the grid positions z, y, x (mm): seven coplanar beams about the
    z axis, exp(-0.005 depth) times a 10 x 10 beamlet fluence over 40 % of the
    box, blurred by a 3 mm Gaussian penumbra."""
    lo, hi = box
    cen = [(a + b) / 2 for a, b in zip(lo, hi)]
    w_u, w_z = 0.4 * max(hi[1] - lo[1], hi[2] - lo[2]), 0.4 * (hi[0] - lo[0])
    ue = torch.linspace(-w_u / 2, w_u / 2, 11, device=DEV, dtype=F64)
    ze = torch.linspace(-w_z / 2, w_z / 2, 11, device=DEV, dtype=F64)

    def bumps(t, e):
        c = torch.special.ndtr((t[..., None] - e) / 3.0)
        return c[..., :-1] - c[..., 1:]

    cz = bumps(z - cen[0], ze)                                         # (nz, 10)
    yy, xx = y[:, None].expand(-1, x.numel()), x[None, :].expand(y.numel(), -1)
    total = torch.zeros((z.numel(), y.numel() * x.numel()), device=DEV)
    for k in range(7):
        th = 2.0 * math.pi * k / 7
        dy, dx = math.sin(th), math.cos(th)
        depth = torch.full_like(yy, math.inf)
        if abs(dx) > 1e-12:
            depth = torch.minimum(depth, ((xx - lo[2]) if dx > 0 else (hi[2] - xx)) / abs(dx))
        if abs(dy) > 1e-12:
            depth = torch.minimum(depth, ((yy - lo[1]) if dy > 0 else (hi[1] - yy)) / abs(dy))
        u = (yy - cen[1]) * dx - (xx - cen[2]) * dy
        fl = torch.exp(-0.005 * depth.clamp_min(0.0))[..., None] * bumps(u, ue)     # (ny, nx, 10)
        total += (cz @ weights[k].T).float() @ fl.reshape(-1, 10).T.float()
    return total.reshape(z.numel(), y.numel(), x.numel())


def _smooth_noise(shape, h, gen, sigma_mm=10.0, sd=0.01):
    """White noise blurred by a Gaussian of sigma_mm, with standard deviation sd."""
    f = torch.randn(shape, generator=gen, device=DEV)
    for a in range(3):
        i = torch.arange(shape[a], device=DEV, dtype=torch.float32)
        w = torch.exp(-0.5 * ((i[:, None] - i[None, :]) * h / sigma_mm) ** 2)
        f = torch.movedim(torch.tensordot(w / w.sum(1, keepdim=True), f, dims=([1], [a])), 0, a)
    return f * (sd / f.std())


def _gens(seed):
    cpu, dev = torch.Generator(), torch.Generator(device=DEV)
    cpu.manual_seed(seed)
    dev.manual_seed(seed + 7919)
    return cpu, dev


def _axes(n, h, origin=0.0):
    return [torch.arange(k, device=DEV, dtype=F64) * h + origin for k in n]


def _pair(c, seed):
    """Reference and evaluation dose (float32, contiguous) of a map case."""
    cpu, dev = _gens(seed)
    shape, h = (c["nz"], c["ny"], c["nx"]), c["h"]
    if c["nz"] == 1:
        r, e = _blobs(shape[1:], h, cpu, [(0.0, 0.0), (0.0, c["shift"])])
        e = c["scale"] * e + 0.005 * torch.randn(shape[1:], generator=dev, device=DEV)
        return r.float().contiguous(), e.float().contiguous()
    box = ([-h / 2] * 3, [(k - 0.5) * h for k in shape])
    w = _beam_weights(cpu)
    z, y, x = _axes(shape, h)
    r = _beams(z, y, x, box, w)
    e = _beams(z, y, x - c["shift"], box, w)
    top = r.max()
    e = c["scale"] * (e / top) + _smooth_noise(shape, h, dev)
    return (r / top).contiguous(), e.contiguous()


def _grids_geometry(c):
    """Evaluation grid of a two-grid case: its shape, spacing and origin."""
    he = c["h"] / c["ratio"]
    shape = [max(2, int(round(n * c["ratio"]))) for n in (c["nz"], c["ny"], c["nx"])]
    return shape, float(np.float32(he)), float(np.float32(c["offset"]))


def _grids_pair(c, seed):
    """Reference dose on its grid and the evaluation dose on a finer one."""
    cpu, dev = _gens(seed)
    shape, h = (c["nz"], c["ny"], c["nx"]), c["h"]
    box = ([-h / 2] * 3, [(k - 0.5) * h for k in shape])
    w = _beam_weights(cpu)
    eshape, he, origin = _grids_geometry(c)
    r = _beams(*_axes(shape, h), box, w)
    z, y, x = _axes(eshape, he, origin)
    top = r.max()
    e = c["scale"] * (_beams(z, y, x - c["shift"], box, w) / top) + _smooth_noise(eshape, he, dev)
    return (r / top).contiguous(), e.contiguous()


def _batch_pairs(c):
    """The pairs of a batch case as map cases: 256 x 256 planes at 1 mm and
    volumes at 2 mm from 64^3 to 200 x 200 x 150."""
    rng = np.random.default_rng(3000 + c["pick"])
    out = []
    for i in range(c["planes"] + c["volumes"]):
        dd, dta = [(0.01, 1.0), (0.02, 2.0), (0.03, 3.0)][int(rng.integers(0, 3))]
        shift, scale = float(rng.uniform(0.0, 3.0)), float(rng.uniform(0.97, 1.05))
        t = float(rng.uniform(0.0, 1.0))
        shape = (1, 256, 256) if i < c["planes"] else tuple(
            int(round(math.exp(math.log(64) + t * math.log(b / 64)))) for b in (150, 200, 200))
        out.append(_map("map", shape, 1.0 if i < c["planes"] else 2.0, dd, dta, shift=shift, scale=scale))
    return out


def _crit(c):
    return g.criteria(c["dd"], c["dta"], c.get("local", False), 0.10, 0.0)


def _geom(c):
    nd = 2 if c["nz"] == 1 else 3
    return nd, (c["nz"], c["ny"], c["nx"]), (1.0 if nd == 2 else c["h"], c["h"], c["h"])


# ---------------------------------------------------------------------------
# Network rows
# ---------------------------------------------------------------------------

def _sampled(c, ref, ev, seed, rows):
    """Voxels whose network rows are taken: evaluated ones, three quarters of
    them with a dose difference worth a search."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 31)
    dd = np.float32(c["dd"]) * ref.max()
    act = ref >= np.float32(0.1) * ref.max()
    far = (act & ((ev - ref).abs() > dd * (c["h"] / c["dta"]))).flatten().nonzero()[:, 0]
    anyv = act.flatten().nonzero()[:, 0]
    n_far = min(far.numel(), rows * 3 // 4)
    pick = lambda v, n: v[torch.randint(0, v.numel(), (n,), generator=gen, device=DEV)]
    parts = ([pick(far, n_far)] if n_far else []) + [pick(anyv, rows - n_far)]
    return torch.cat(parts).to(torch.int32)


def _grad(d, hn):
    """Gradient magnitude of a dose in dose per normalised length: central
    differences inside, one-sided at the edges."""
    s = torch.zeros_like(d)
    for a in range(3):
        v = torch.movedim(d, a, 0)
        q = torch.empty_like(v)
        q[1:-1] = (v[2:] - v[:-2]) * 0.5
        q[0], q[-1] = v[1] - v[0], v[-1] - v[-2]
        s += (torch.movedim(q, 0, a) / hn) ** 2
    return s.sqrt()


def _features(c, ref, ev, vox):
    """The 375 features of the listed voxels of a 3D pair, in 64 bits, padded
    to 384 columns."""
    r, e = ref.double(), ev.double()
    dd = float(np.float32(c["dd"])) * float(ref.max())
    hn = c["h"] / c["dta"]
    ge, gr = (_grad(e, hn) / dd).clamp_max(32.0), (_grad(r, hn) / dd).clamp_max(32.0)
    nz, ny, nx = ref.shape
    v = vox.long()
    x, y, z = v % nx, (v // nx) % ny, v // (nx * ny)
    o = torch.arange(5, device=DEV) - 2
    oz, oy, ox = [t.flatten() for t in torch.meshgrid(o, o, o, indexing="ij")]
    X = torch.zeros((v.numel(), K_PAD), device=DEV, dtype=F64)
    for i in range(0, v.numel(), 65536):
        s = slice(i, i + 65536)
        px, py, pz = x[s, None] + ox, y[s, None] + oy, z[s, None] + oz
        ok = (px >= 0) & (px < nx) & (py >= 0) & (py < ny) & (pz >= 0) & (pz < nz)
        p = torch.where(ok, (pz * ny + py) * nx + px, 0)
        d0 = ((e.flatten()[p] - r.flatten()[v[s], None]) / dd).clamp(-16.0, 16.0)
        for k, f in enumerate((d0, ge.flatten()[p], gr.flatten()[p])):
            X[s, 125 * k:125 * k + 125] = torch.where(ok, f, 0.0)
    return X


def _network_rows(rows, seed):
    """Feature rows (bf16) as the training recipe meets them, from one 2 mm pair."""
    c = _map("map", (72, 96, 96), 2.0, 0.02, 2.0, shift=2.5, scale=1.03)
    ref, ev = _pair(c, seed)
    return _features(c, ref, ev, _sampled(c, ref, ev, seed, rows)).to(torch.bfloat16).contiguous()


def _targets(rows, seed):
    """Training targets: nearest-point offsets (normalised) and log(gamma + 1e-3)."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 57)
    off = 0.6 * torch.randn((rows, 3), generator=gen, device=DEV)
    gam = off.norm(dim=1, keepdim=True) * (1.0 + torch.rand((rows, 1), generator=gen, device=DEV))
    return torch.cat([off, torch.log(gam + 1e-3)], 1).contiguous()


def _split(p):
    """Parameter vector -> W1 [128][384], b1, W2 [128][128], b2, W3 [8][128], b3."""
    sizes = [(K_H, K_PAD), (K_H,), (K_H, K_H), (K_H,), (K_OUTPAD, K_H), (K_OUTPAD,)]
    out, at = [], 0
    for s in sizes:
        n = int(np.prod(s))
        out.append(p[at:at + n].reshape(s))
        at += n
    return out


def _start_params(seed):
    """He-normal weights, zero biases and padding (float32 numpy)."""
    rng = np.random.default_rng(seed)
    p = np.zeros(K_H * K_PAD + K_H + K_H * K_H + K_H + K_OUTPAD * K_H + K_OUTPAD, np.float32)
    W1, _, W2, _, W3, _ = _split(p)
    W1[:, :K_IN] = rng.normal(size=(K_H, K_IN)) * math.sqrt(2.0 / K_IN)
    W2[:] = rng.normal(size=(K_H, K_H)) * math.sqrt(2.0 / K_H)
    W3[:K_OUT] = rng.normal(size=(K_OUT, K_H)) * math.sqrt(1.0 / K_H)
    return p


def _file_params(path):
    with open(path, "rb") as f:
        data = f.read()
    n = K_H * K_PAD + K_H + K_H * K_H + K_H + K_OUTPAD * K_H + K_OUTPAD
    head = 8 + struct.calcsize("<6iqQ")
    return np.frombuffer(data, "<f4", n, head).copy()


# ---------------------------------------------------------------------------
# State, run
# ---------------------------------------------------------------------------

class State:
    def __init__(self, **kw):
        self.handle = self.model = None
        self.__dict__.update(kw)

    def __del__(self):
        g.gamma_destroy(self.handle)
        g.gamma_model_destroy(self.model)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        m = g.gamma_model_create(1)
        g.gamma_model_set_params(m, _start_params(seed))
        return State(kind=kind, model=m, X=_network_rows(c["rows"], seed), T=_targets(c["rows"], seed))
    if kind == "infer":
        m = g.gamma_model_create(1)
        g.gamma_model_load(m, MODEL)
        X = _network_rows(c["rows"], seed)
        return State(kind=kind, model=m, X=X, Y=torch.empty((c["rows"], K_OUT), device=DEV))
    if kind == "batch":
        cases = _batch_pairs(c)
        pairs = [_pair(p, seed + 101 * i) for i, p in enumerate(cases)]
        outs = [torch.empty_like(r) for r, _ in pairs]
        h = g.gamma_batch_create([(r, e, o, *_geom(p), _crit(p))
                                  for (r, e), o, p in zip(pairs, outs, cases)])
        return State(kind=kind, handle=h, pairs=pairs, outs=outs)
    if kind == "grids":
        ref, ev = _grids_pair(c, seed)
        eshape, he, origin = _grids_geometry(c)
        h = g.gamma_create_grids(ref, ev, 3, ref.shape, [c["h"]] * 3, [0.0] * 3, eshape, [he] * 3,
                                 [origin] * 3, _crit(c))
        return State(kind="map", handle=h, ref=ref, ev=ev, out=torch.empty_like(ref))
    ref, ev = _pair(c, seed)
    if kind == "host":
        pin = lambda t: t.cpu().pin_memory()
        h = g.gamma_create(None, None, *_geom(c), _crit(c))
        return State(kind=kind, handle=h, ref=pin(ref), ev=pin(ev),
                     out=torch.empty(ref.shape, pin_memory=True))
    out = torch.empty_like(ref)
    h = g.gamma_create(ref, ev, *_geom(c), _crit(c))
    st = State(kind="map", handle=h, ref=ref, ev=ev, out=out)
    if kind == "learned":
        g.gamma_load_model(h, MODEL)
    if kind == "rows":
        g.gamma_run(h, out)
        g.gamma_pass_rate(h)
        st.kind, st.vox = kind, _sampled(c, ref, ev, seed, c["rows"])
        st.X = torch.empty((c["rows"], K_PAD), dtype=torch.bfloat16, device=DEV)
        st.T = torch.empty((c["rows"], K_OUT), device=DEV)
    return st


def run(s):
    if s.kind == "map":
        g.gamma_run(s.handle, s.out)
        return s.out
    if s.kind == "batch":
        g.gamma_batch_run(s.handle)
        return s.outs
    if s.kind == "host":
        g.gamma_run_host(s.handle, s.ref, s.ev, s.out)
        return {"rate": g.gamma_pass_rate(s.handle)[0], "map": s.out}
    if s.kind == "rows":
        g.gamma_features(s.handle, s.vox, s.X)
        g.gamma_labels(s.handle, s.out, s.vox, s.T)
        return {"X": s.X, "T": s.T}
    if s.kind == "train":
        loss = g.gamma_model_train_step(s.model, s.X, s.T, 1e-3)
        return {"loss": loss, "params": g.gamma_model_get_params(s.model)}
    g.gamma_model_infer(s.model, s.X, s.Y)
    return s.Y


def work(c):
    """Doses read and the map written once (12 bytes per voxel); FLOPs of the
    faces through each evaluated voxel (about 40 % of the voxels pass the
    cutoff; 38 edges of 4 and 74 faces of 6 operations in 3D, 10 and 12 in
    2D).  Rows: inputs and outputs once, and the network's multiply-adds."""
    kind = c["kind"]
    net = 2.0 * (K_IN * K_H + K_H * K_H + K_H * K_OUT)
    if kind == "infer":
        return {"bytes": c["rows"] * (2.0 * K_PAD + 4.0 * K_OUT), "flops": c["rows"] * net}
    if kind == "train":
        return {"bytes": c["rows"] * (2.0 * K_PAD + 4.0 * K_OUT) + 4.0 * 7 * 66824,
                "flops": c["rows"] * (3.0 * net - 2.0 * K_IN * K_H)}
    if kind == "rows":
        return {"bytes": c["rows"] * (2.0 * 4 * 343 + 2.0 * K_PAD + 4.0 * K_OUT + 8.0),
                "flops": c["rows"] * (125.0 * 2 * 10 + 8.0 * 615)}
    if kind == "batch":
        ws = [work(p) for p in _batch_pairs(c)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    n = c["nz"] * c["ny"] * c["nx"]
    if kind == "grids":
        ne = int(np.prod(_grids_geometry(c)[0]))
        return {"bytes": 8.0 * n + 4.0 * ne, "flops": 0.4 * n * 8 * 615.0}
    per = 10 * 4 + 12 * 6 if c["nz"] == 1 else 38 * 4 + 74 * 6
    return {"bytes": 12.0 * n, "flops": 0.4 * n * per}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _chains(nd):
    """Faces owned by a cell: strictly nested axis sets u1 < ... < um."""
    full = range(1, 1 << nd)
    two = [(u, v) for u in full for v in full if u & v == u and u != v]
    three = [(u, v, w) for u, v in two for w in full if v & w == v and v != w]
    return [(u,) for u in full] + two + three


def _cell_d2(q, off, hn2, nd):
    """Smallest squared distance from the origin to the faces of each cell: q
    [n, 2^nd] relative doses of its vertices (NaN outside the grid), off
    [n, nd] its lower corner (x, y, z; cells)."""
    kap = {A: 1.0 / sum(hn2[a] for a in range(nd) if A >> a & 1) for A in range(1, 1 << nd)}
    lin = [hn2[a] * off[:, a] for a in range(nd)]
    sq = [lin[a] * off[:, a] for a in range(nd)]
    beta, rho = {}, {}
    for A in kap:
        ax = [a for a in range(nd) if A >> a & 1]
        beta[A] = -sum(lin[a] for a in ax) * kap[A]
        rho[A] = sum((hn2[a] * hn2[b] * kap[A]) * (off[:, a] - off[:, b]) ** 2
                     for a, b in itertools.combinations(ax, 2)) if len(ax) > 1 else 0.0
    rest = {M: sum((sq[a] for a in range(nd) if not M >> a & 1), torch.zeros_like(q[:, 0]))
            for M in range(1 << nd)}
    best = q[:, 0] ** 2 + rest[0]
    for ch in _chains(nd):
        node = (0,) + ch
        D, L, r2, d, sets = 1.0, q[:, 0], rest[ch[-1]], [], []
        for u, v in zip(node, node[1:]):
            A = u ^ v
            dl = q[:, v] - q[:, u]
            D = D + dl * dl * kap[A]
            L = L + dl * beta[A]
            r2 = r2 + rho[A]
            d.append(dl)
            sets.append(A)
        f = L / D
        mu = [1.0] + [beta[A] - f * dl * kap[A] for A, dl in zip(sets, d)] + [0.0]
        ok = torch.ones_like(q[:, 0], dtype=torch.bool)
        for a, b in zip(mu, mu[1:]):
            ok &= torch.as_tensor(a, device=DEV, dtype=F64) >= b
        best = torch.where(ok, torch.minimum(best, r2 + L * f), best)
    return best


def _exact_map(ref, ev, h_ref, o_ref, h_ev, o_ev, c):
    """Gamma of every reference voxel against the evaluation surface, in 64
    bits (3D, or 2D with a leading axis of 1); NaN below the cutoff."""
    f32 = np.float32
    nd = 2 if ref.shape[0] == 1 else 3
    dta, dd = float(f32(c["dta"])), float(f32(c["dd"]))
    norm = ref.max()
    act = (ref >= f32(0.1) * norm) & ((ref > 0) if c.get("local") else (ref == ref))
    vox = act.flatten().nonzero()[:, 0]
    hn = [float(f32(h_ev)) / dta] * nd
    n = [ev.shape[2 - a] for a in range(nd)]
    rn = [ref.shape[2 - a] for a in range(3)]
    ix = [vox % rn[0], (vox // rn[0]) % rn[1], vox // (rn[0] * rn[1])][:nd]
    same = h_ref == h_ev and o_ref == o_ev
    c0, fr = [], []
    for a in range(nd):
        u = ix[a].double() if same else (o_ref + ix[a].double() * h_ref - o_ev) / h_ev
        k = torch.floor(u).clamp(0, n[a] - 1 if same else n[a] - 2)
        c0.append(k.long())
        fr.append(u - k)
    dr = ref.flatten()[vox].double()
    inv = 1.0 / (dd * (dr if c.get("local") else norm.double()))
    best = torch.full_like(dr, math.inf)
    evf = ev.flatten()
    stride = [1, n[0], n[0] * n[1]]
    # cell offsets by a lower bound of their distance from any point of the voxel's cell
    reach = 2.0
    done = -1.0
    while True:
        lim = [min(int(math.ceil(reach / hn[a])) + 1, n[a]) for a in range(nd)]
        axes = [torch.arange(-l - 1, l + 1) for l in lim]
        grid = torch.stack([t.flatten() for t in torch.meshgrid(*axes, indexing="ij")], 1)
        gap = torch.clamp(torch.maximum(grid - (0 if same else 1), -grid - 1), min=0).double()
        key = (gap * torch.tensor(hn, dtype=F64)).pow(2).sum(1).sqrt()
        sel = ((key > done) & (key <= reach)).nonzero()[:, 0]
        order = sel[torch.argsort(key[sel])]
        offs, keys = grid[order].to(DEV), key[order]
        at = 0
        while at < offs.shape[0]:
            live = (best > float(keys[at]) ** 2).nonzero()[:, 0]
            if live.numel() == 0:
                break
            k = max(1, min(offs.shape[0] - at, 3000000 // live.numel()))
            for l0 in range(0, live.numel(), 3000000):
                lv = live[l0:l0 + 3000000].repeat_interleave(k)
                of = offs[at:at + k].repeat(live[l0:l0 + 3000000].numel(), 1)
                p = [c0[a][lv] + of[:, a] for a in range(nd)]
                d = [of[:, a].double() - fr[a][lv] for a in range(nd)]
                ok = torch.ones_like(lv, dtype=torch.bool)
                k2 = torch.zeros_like(dr[lv])
                for a in range(nd):
                    ok &= (p[a] >= 0) & (p[a] < n[a])
                    k2 += (torch.maximum(d[a], -d[a] - 1).clamp_min(0) * hn[a]) ** 2
                m = (ok & (k2 < best[lv])).nonzero()[:, 0]
                if m.numel() == 0:
                    continue
                lv, k2 = lv[m], k2[m]
                p, d = [t[m] for t in p], torch.stack([t[m] for t in d], 1)
                base = sum(p[a] * stride[a] for a in range(nd))
                q = torch.empty((m.numel(), 1 << nd), device=DEV, dtype=F64)
                for u in range(1 << nd):
                    o, inside = base, None
                    for a in range(nd):
                        if u >> a & 1:
                            o = o + stride[a]
                            t = p[a] + 1 < n[a]
                            inside = t if inside is None else inside & t
                    if inside is None:
                        q[:, u] = evf[o].double()
                    else:
                        q[:, u] = torch.where(inside, evf[torch.where(inside, o, base)].double(), math.nan)
                iv = inv[lv] if inv.dim() else inv
                q = (q - dr[lv, None]) * (iv[:, None] if inv.dim() else iv)
                lo = torch.nan_to_num(q, nan=math.inf).amin(1)
                hi = torch.nan_to_num(q, nan=-math.inf).amax(1)
                gp = torch.maximum(lo, -hi).clamp_min(0)
                m = (k2 + gp * gp < best[lv]).nonzero()[:, 0]
                if m.numel():
                    best.scatter_reduce_(0, lv[m], _cell_d2(q[m], d[m], [t * t for t in hn], nd), "amin")
            at += k
        if not bool((best > reach * reach).any()) or reach > sum(k * t for k, t in zip(n, hn)) + 1:
            break
        done, reach = reach, reach * 2
    out = torch.full((ref.numel(),), math.nan, device=DEV, dtype=F64)
    out[vox] = best.clamp_min(0).sqrt()
    return out.reshape(ref.shape)


def _exact_train(c, seed):
    X = _network_rows(c["rows"], seed).double()
    T = _targets(c["rows"], seed).double()
    p = torch.from_numpy(_start_params(seed)).to(DEV).double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = _split(p)
    y = torch.relu(torch.relu(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
    r = (y[:, :K_OUT] - T).abs()
    loss = torch.where(r <= 1, 0.5 * r * r, r - 0.5).sum() / c["rows"]
    loss.backward()
    gr = p.grad
    step = 1e-3 * gr / (gr.abs() + 1e-8)               # the first Adam step
    return {"loss": loss.detach(), "params": (p.detach() - step).cpu().numpy()}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        return _exact_train(c, seed)
    if kind == "infer":
        W1, b1, W2, b2, W3, b3 = [torch.from_numpy(a).to(DEV).double() for a in _split(_file_params(MODEL))]
        X = _network_rows(c["rows"], seed).double()
        y = torch.relu(torch.relu(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
        return y[:, :K_OUT].contiguous()
    if kind == "batch":
        cases = _batch_pairs(c)
        return [_exact_one(p, *_pair(p, seed + 101 * i)) for i, p in enumerate(cases)]
    if kind == "grids":
        ref, ev = _grids_pair(c, seed)
        _, he, origin = _grids_geometry(c)
        return _exact_map(ref, ev, c["h"], 0.0, he, origin, c)
    ref, ev = _pair(c, seed)
    if kind == "rows":
        return {"X": _features(c, ref, ev, _sampled(c, ref, ev, seed, c["rows"])), "T": None}
    m = _exact_one(c, ref, ev)
    if kind == "host":
        ok = m[torch.isfinite(m)]
        return {"rate": (ok <= 1).double().mean(), "map": m.cpu()}
    return m


def _exact_one(c, ref, ev):
    if ref.dim() == 2:
        return _exact_map(ref[None], ev[None], c["h"], 0.0, c["h"], 0.0, c)[0]
    return _exact_map(ref, ev, c["h"], 0.0, c["h"], 0.0, c)
