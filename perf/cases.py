"""Workloads whose run time is measured, with their inputs, the work they cannot
do without, and their exact results in 64 bits.

A case is a dict of plain values.  Every kind of call a program makes of the
library per frame or per training run is there, over the sizes of the
repository's own workloads (``paper_1404_3363_gb300.scenes``, the benchmark,
the tests): tiles of 64 x 64 pixels up to 3840 x 2160 frames, cubic and
quadratic volumes of one to 16 blocks, every scalar mode in use, FP32, mixed
and FP64 arithmetic, the error-controlled and the fixed-step integrators,
per-sample root finding, cutting planes, batches, host read-back, and the
training of the learned guess.

``exact`` is an independent 64-bit renderer in plain torch: Cox-de Boor
evaluation, ray/face intersections by Newton from small screen-space cells of
every boundary face, blockwise pairing, the preimage of every sample by
Newton, and the compositing of Alg. 1 with supersampling.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_1404_3363_gb300 import ivv, scenes

FP32, MIXED, FP64 = scenes.PRECISION_FP32, scenes.PRECISION_MIXED, scenes.PRECISION_FP64
SCENES = {
    "cube": scenes.twisted_cube,      # one cubic element, control-point scalar
    "bar": scenes.twisted_bar,        # one cubic block 8x8x32, Eq. 23
    "beam": scenes.bent_beam,         # 16 cubic blocks, control-point scalar
    "loaded": scenes.bent_beam,       # the same with a displacement: von Mises scalar
    "step": scenes.backstep,          # 3 quadratic blocks, sharp shear layer
}


def _case(name, call, scene, width, height, **more):
    c = {"call": call, "scene": scene, "width": width, "height": height, "precision": FP32, "method": 0, "guess": 0,
         "rk_method": 0, "rk_tol": 1e-5, "cuts": 0, "count": 1}
    c.update(more)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a plug-in host renders one tile of a picture into memory of its own pool
        _case("tile64_cube_fp32", "tile", "cube", 64, 64),
        # the small preview frame while the user turns the model
        _case("preview256_bar_fp32", "render", "bar", 256, 256),
        # the ordinary full-HD frame of one block (the benchmark's headline)
        _case("frame1080_bar_fp32", "render", "bar", 1920, 1080),
        # a full-HD frame of a multi-block model with accurate entry points
        _case("frame1080_beam_mixed", "render", "beam", 1920, 1080, precision=MIXED),
        # the large frame: a flow field at 4K with its tight tolerance
        _case("frame4k_step_fp32", "render", "step", 3840, 2160, rk_tol=7e-7),
        # root finding from the trained guess network, mixed precision
        _case("frame1080_beam_rf_learned", "render", "beam", 1920, 1080, precision=MIXED, method=1, guess=1),
        # root finding from the chord in a window of odd size, many elements
        _case("window1367_step_rf_chord", "render", "step", 1367, 769, method=1, guess=2),
        # structural analysis: von Mises value, the model cut open by a plane
        _case("frame720_loaded_cut", "render", "loaded", 1280, 720, cuts=1),
        # the reference-accuracy picture: everything in FP64 at a tight tolerance
        _case("image64_cube_fp64", "render", "cube", 64, 64, precision=FP64, rk_tol=1e-8),
        # a frame read back to host memory, the paper's midpoint integrator
        _case("host1080_bar_midpoint", "host", "bar", 1920, 1080, rk_method=2),
        # a render server: requests of several users and volumes in one graph
        _case("batch16_mixed_sizes", "batch", "all", 0, 0, count=16),
        # preparing the learned guess of a new model: 128 optimiser steps
        _case("train_guess_bar", "train", "bar", 0, 0, count=128),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: kinds of calls as above, sizes spread over
    their logarithm, aspect ratios from portrait to wide, odd sizes included."""
    kind = rng.choice(["tile", "ode", "ode", "ode", "rf", "rf", "fixed", "vm", "fp64", "host", "batch", "train"])
    if kind == "train":
        return _case(None, "train", rng.choice(["bar", "cube", "step"]), 0, 0, count=_spread(rng, 16, 160))
    if kind == "batch":
        return _case(None, "batch", "all", 0, 0, count=_spread(rng, 2, 20))
    if kind == "tile":
        return _case(None, "tile", rng.choice(["cube", "bar", "beam"]), rng.randint(16, 64), rng.randint(16, 64),
                     precision=rng.choice([FP32, MIXED]))
    if kind == "fp64":
        return _case(None, "render", "cube", rng.randint(24, 64), rng.randint(24, 64), precision=FP64,
                     rk_tol=10.0 ** rng.uniform(-8, -6))
    px = _spread(rng, 128 * 128, 3840 * 2160 if kind == "ode" else 1920 * 1080)
    w = max(64, int(math.sqrt(px * math.exp(rng.uniform(math.log(0.6), math.log(2.4))))))
    h = max(64, px // w)
    prec = rng.choice([FP32, MIXED])
    if kind == "ode":
        scene = rng.choice(["cube", "bar", "beam", "step"])
        if scene != "step" and w * h > 1920 * 1080:
            w, h = w // 2, h // 2
        return _case(None, "render", scene, w, h, precision=prec, rk_tol=7e-7 if scene == "step" else 1e-5,
                     cuts=rng.choice([0, 0, 0, 1]))
    if kind == "rf":
        scene, guess = rng.choice([("bar", 2), ("bar", 1), ("beam", 2), ("beam", 1), ("step", 2)])
        return _case(None, "render", scene, w, h, precision=prec, method=1, guess=guess)
    if kind == "vm":
        return _case(None, "render", "loaded", w, h, precision=prec, cuts=rng.choice([0, 1]))
    if kind == "fixed":
        return _case(None, "render", rng.choice(["bar", "beam"]), w, h, rk_method=rng.randint(2, 6))
    return _case(None, "host", rng.choice(["cube", "bar", "beam"]), w, h, rk_method=rng.choice([0, 2]))


# ------------------------------------------------------------------- inputs

def _transfer(rng, n, clear=0.0):
    """A colour map of n knots near even spacing, transparent below `clear`."""
    r = np.linspace(0.0, 1.0, n)
    r[1:-1] += rng.uniform(-0.25, 0.25, n - 2) / (n - 1)
    rgba = rng.uniform(0.0, 1.0, (n, 4))
    rgba[:, 3] = np.where(r <= clear, 0.0, 0.1 + 0.9 * rgba[:, 3])
    return scenes.TransferFunction(r.astype(np.float32), rgba.astype(np.float32), 4.0)


def _scene(case, seed):
    """The case's scene: geometry, camera and transfer function of this seed."""
    kw = {"displacement": True} if case["scene"] == "loaded" else {}
    s = SCENES[case["scene"]](seed=seed, width=max(case["width"], 1), height=max(case["height"], 1),
                              precision=case["precision"], **kw)
    rng = np.random.default_rng(seed + 77)
    tf = _transfer(rng, 32 if case["scene"] == "step" else 8, 0.25 if case["scene"] in ("beam", "loaded") else 0.0)
    lo, hi = s.cp_bbox()
    cuts = []
    for _ in range(case["cuts"]):
        n = rng.normal(size=3)
        n /= np.linalg.norm(n)
        cuts.append((n[0], n[1], n[2], float(-n @ (0.5 * (lo + hi)))))
    p = scenes.RenderParams(rk_tol=case["rk_tol"], ds=s.params.ds, precision=case["precision"], method=case["method"],
                            use_mlp_guess=case["guess"], rf_tol=1e-3, rk_method=case["rk_method"],
                            cut_planes=tuple(cuts))
    return dataclasses.replace(s, tf=tf, params=p)


def _requests(case, seed):
    """A batch's volumes and requests; the sizes (256 to 1024 pixels a side)
    belong to the case, what is shown and from where to the seed."""
    vols, reqs = scenes.batch_requests(seed=seed, n=case["count"])
    rng, sizes = np.random.default_rng(seed + 77), np.random.default_rng(case["count"])
    return vols, [dataclasses.replace(q, width=int(sizes.integers(256, 1025)), height=int(sizes.integers(256, 1025)),
                                      tf=_transfer(rng, 8)) for q in reqs]


def prepare(case, seed):
    if case["call"] == "batch":
        vols, reqs = _requests(case, seed)
        handles = [ivv.volume_for(s) for s in vols]
        batch = ivv.Batch([(handles[q.volume], q.camera, q.width, q.height, q.tf) for q in reqs])
        return {"call": "batch", "batch": batch, "volumes": handles}
    sc = _scene(case, seed)
    st = {"call": case["call"], "scene": sc, "volume": ivv.volume_for(sc)}
    if case["call"] == "train":
        st["steps"], st["seed"] = case["count"], seed
        return st
    h, w = sc.height, sc.width
    if case["call"] == "host":
        st["out"] = torch.empty((h, w, 4), dtype=torch.float32).pin_memory()
    else:
        st["out"] = torch.empty((h, w, 4), dtype=torch.float32, device="cuda")
    if case["guess"] == 1:
        st["volume"].train_guess(samples_per_block=1 << 15, epochs=4, batch=2048, seed=seed)
    return st


TRAIN_BATCH = 4096


def run(state):
    call = state["call"]
    if call == "batch":
        return state["batch"].render()
    sc, vol = state["scene"], state["volume"]
    if call == "train":
        per_epoch = min(32, state["steps"])
        loss = vol.train_guess(samples_per_block=per_epoch * TRAIN_BATCH, epochs=max(1, state["steps"] // per_epoch),
                               batch=TRAIN_BATCH, seed=state["seed"])
        return {"loss": np.array(loss, np.float32),
                "weights": np.stack([vol.get_guess_weights(b)[0] for b in range(len(loss))])}
    if call == "tile":
        return vol.render_noalloc(sc.camera, sc.params, sc.width, sc.height, state["out"])
    if call == "host":
        return vol.render_to_host(sc.camera, sc.params, sc.width, sc.height, state["out"])
    return vol.render(sc.camera, sc.params, sc.width, sc.height, out=state["out"])


# --------------------------------------------------------------------- work

# share of the pixels whose ray meets the volume and the mean number of
# samples on such a ray (the average over camera seeds)
COVER = {"cube": (0.14, 62.0), "bar": (0.07, 14.0), "beam": (0.065, 14.0), "loaded": (0.065, 14.0), "step": (0.15, 25.0)}
# evaluations of the map per sample: right-hand sides of the error-controlled
# pair, stages of the fixed-step family, Newton evaluations
FIXED_STAGES = {2: 2, 3: 3, 4: 4, 5: 4, 6: 6}


def _map_flops(degree):
    """One evaluation of phi, J and the 3x3 solve by sum factorisation."""
    n = degree + 1
    return 2 * (6 * n ** 3 + 9 * n ** 2 + 12 * n) + 131


def _volume_bytes(sc):
    return 4 * sum(b.geom_cp.size + b.geom_cp.size // 3 for b in sc.blocks)


def work(case):
    """The image written once and the control points read once; one map
    evaluation per right-hand side or Newton step, the scalar, and Alg. 1 with
    four sub-samples per sample."""
    if case["call"] == "train":
        # three products of the 3-64-64-3 network per sample, samples read once a step
        n = case["count"] * TRAIN_BATCH
        return {"bytes": 32.0 * n, "flops": 3.0 * 2 * (3 * 64 + 64 * 64 + 64 * 3) * n}
    if case["call"] == "batch":
        px = case["count"] * 640.0 ** 2
        return {"bytes": 16 * px, "flops": px * 0.12 * 23 * (1.5 * _map_flops(3) + 350)}
    sc = _scene(case, 1)
    px = float(case["width"] * case["height"])
    cover, per_ray = COVER[case["scene"]]
    rhs = _map_flops(max(sc.blocks[0].degree))
    if case["method"] == 1:
        evals = 2.0
    elif case["rk_method"]:
        evals = float(FIXED_STAGES[case["rk_method"]])
    else:
        evals = 1.2 if case["precision"] != FP64 else 12.0
    samples = px * cover * per_ray
    scalar = {"bar": 1220, "loaded": 2348}.get(case["scene"], 200)
    return {"bytes": 16 * px + _volume_bytes(sc), "flops": samples * (evals * rhs + scalar + 150)}


# -------------------------------------------------------------------- exact

def exact(case, seed):
    if case["call"] == "train":
        return None                     # the optimiser's path has no closed form
    with torch.no_grad():
        if case["call"] == "batch":
            vols, reqs = _requests(case, seed)
            images = []
            for q in reqs:
                sc = vols[q.volume]
                sc = dataclasses.replace(sc, tf=q.tf, camera=q.camera, width=q.width, height=q.height,
                                         params=scenes.RenderParams(ds=sc.cp_diag() / 128.0))
                images.append(_Exact(sc).image())
            return images
        return _Exact(_scene(case, seed)).image()


F8 = torch.float64


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=F8, device="cuda")


def _basis(knots, degree, x):
    """First control point, values and derivatives of the degree + 1 B-splines
    that do not vanish at x (Cox-de Boor, the end point taken from the left)."""
    n = len(knots) - degree - 1
    t = _dev((knots - knots[0]) / (knots[-1] - knots[0]))
    k = torch.searchsorted(t, x.contiguous(), right=True) - 1
    k = k.clamp(degree, n - 1)
    b = [torch.ones_like(x)]
    low = b
    for p in range(1, degree + 1):
        if p == degree:
            low = b
        new = [torch.zeros_like(x) for _ in range(p + 1)]
        for r in range(p):
            left, right = t[k + 1 + r - p], t[k + 1 + r]
            u = b[r] / (right - left)
            new[r] = new[r] + (right - x) * u
            new[r + 1] = new[r + 1] + (x - left) * u
        b = new
    d = [torch.zeros_like(x) for _ in range(degree + 1)]
    for r in range(degree):
        u = degree * low[r] / (t[k + 1 + r] - t[k + 1 + r - degree])
        d[r] = d[r] - u
        d[r + 1] = d[r + 1] + u
    return k - degree, torch.stack(b, -1), torch.stack(d, -1)


class _Exact:
    CHUNK = 1 << 17

    def __init__(self, sc):
        self.sc = sc
        self.fields = []                 # per block: control points [nw][nv][nu][C]
        for b in sc.blocks:
            parts = [np.asarray(b.geom_cp, np.float64)]
            if sc.scalar_mode == scenes.SCALAR_CP:
                parts.append(np.asarray(b.scalar_cp, np.float64)[..., None])
            elif sc.scalar_mode == scenes.SCALAR_VONMISES:
                parts.append(np.asarray(b.disp_cp, np.float64))
            self.fields.append(_dev(np.concatenate(parts, -1)))
        self.diag = sc.cp_diag()
        c = sc.camera
        eye, target, up = (np.asarray(v, np.float64) for v in (c.eye, c.target, c.up))
        f = (target - eye) / np.linalg.norm(target - eye)
        r = np.cross(f, up)
        r /= np.linalg.norm(r)
        u = np.cross(r, f)
        self.sy = 0.5 * c.ortho_height if c.ortho else math.tan(0.5 * math.radians(c.fovy_deg))
        self.sx = self.sy * sc.width / sc.height
        self.eye, self.f, self.r, self.u = (_dev(v) for v in (eye, f, r, u))

    # ---- camera
    def rays(self, pix):
        w, h = self.sc.width, self.sc.height
        nx = ((pix % w).to(F8) + 0.5) / w * 2 - 1
        ny = 1 - (torch.div(pix, w, rounding_mode="floor").to(F8) + 0.5) / h * 2
        off = nx[:, None] * self.sx * self.r + ny[:, None] * self.sy * self.u
        if self.sc.camera.ortho:
            return self.eye + off, self.f.expand(len(pix), 3)
        d = self.f + off
        return self.eye.expand(len(pix), 3), d / d.norm(dim=1, keepdim=True)

    def screen(self, g):
        """Pixel coordinates (centres at integers) of world points."""
        e = g - self.eye
        x, y = e @ self.r, e @ self.u
        if not self.sc.camera.ortho:
            z = e @ self.f
            x, y = x / z, y / z
        return (x / self.sx + 1) * 0.5 * self.sc.width - 0.5, (1 - y / self.sy) * 0.5 * self.sc.height - 0.5

    # ---- splines
    def evaluate(self, block, p):
        """Values [n][C] and partials [n][3][C] of a block's fields."""
        b, cp = self.sc.blocks[block], self.fields[block]
        nw, nv, nu, ch = cp.shape
        flat = cp.reshape(-1, ch)
        outs, ders = [], []
        for q in p.split(self.CHUNK):
            (iu, bu, du), (iv, bv, dv), (iw, bw, dw) = (_basis(np.asarray(b.knots[d], np.float64), b.degree[d],
                                                               q[:, d].clamp(0, 1)) for d in range(3))
            a = [torch.arange(b.degree[d] + 1, device="cuda") for d in range(3)]
            at = (((iw[:, None] + a[2])[:, :, None, None] * nv + (iv[:, None] + a[1])[:, None, :, None]) * nu
                  + (iu[:, None] + a[0])[:, None, None, :])
            g = flat[at]                                              # [n][w][v][u][C]
            gu, gdu = torch.einsum("nwvuc,nu->nwvc", g, bu), torch.einsum("nwvuc,nu->nwvc", g, du)
            gv, gdv = torch.einsum("nwvc,nv->nwc", gu, bv), torch.einsum("nwvc,nv->nwc", gu, dv)
            gud = torch.einsum("nwvc,nv->nwc", gdu, bv)
            outs.append(torch.einsum("nwc,nw->nc", gv, bw))
            ders.append(torch.stack([torch.einsum("nwc,nw->nc", gud, bw), torch.einsum("nwc,nw->nc", gdv, bw),
                                     torch.einsum("nwc,nw->nc", gv, dw)], 1))
        return torch.cat(outs), torch.cat(ders)

    def scalar(self, block, p):
        val, der = self.evaluate(block, p)
        if self.sc.scalar_mode == scenes.SCALAR_CP:
            return val[:, 3]
        J = der[:, :, :3].transpose(1, 2)                             # J[r][c] = d phi_r / d p_c
        if self.sc.scalar_mode == scenes.SCALAR_VONMISES:
            Ju = der[:, :, 3:6].transpose(1, 2)
            X = torch.linalg.solve(J.transpose(1, 2), Ju.transpose(1, 2)).transpose(1, 2)
            s = 0.5 * (X + X.transpose(1, 2))
            dev = ((s[:, 0, 0] - s[:, 1, 1]) ** 2 + (s[:, 1, 1] - s[:, 2, 2]) ** 2 + (s[:, 2, 2] - s[:, 0, 0]) ** 2
                   + 6 * (s[:, 0, 1] ** 2 + s[:, 1, 2] ** 2 + s[:, 2, 0] ** 2))
            return (0.5 * dev).sqrt()
        det = torch.linalg.det(J)
        return det if self.sc.scalar_mode == scenes.SCALAR_DETJ else det / (J * J).sum((1, 2)).sqrt()

    def scalar_range(self):
        if self.sc.scalar_mode == scenes.SCALAR_CP:
            return (min(float(b.scalar_cp.min()) for b in self.sc.blocks),
                    max(float(b.scalar_cp.max()) for b in self.sc.blocks))
        x = (torch.arange(64, dtype=F8, device="cuda") + 0.5) / 64
        grid = torch.stack(torch.meshgrid(x, x, x, indexing="ij"), -1).reshape(-1, 3)
        v = [self.scalar(b, grid) for b in range(len(self.sc.blocks))]
        return min(float(a.min()) for a in v), max(float(a.max()) for a in v)

    # ---- intersections with the boundary faces
    def face_hits(self, block, face):
        """(pixel, t, front, p) of every ray that meets one boundary face."""
        b = self.sc.blocks[block]
        nd, side = face >> 1, face & 1
        ad, bd = (nd + 1) % 3, (nd + 2) % 3

        def embed(a, c):
            p = torch.empty(len(a), 3, dtype=F8, device="cuda")
            p[:, nd], p[:, ad], p[:, bd] = float(side), a, c
            return p

        ga, gb = (self.cells(b, d) for d in (ad, bd))
        fine = [torch.cat([g, 0.5 * (g[1:] + g[:-1])]).sort()[0] for g in (ga, gb)]
        A, B = torch.meshgrid(fine[0], fine[1], indexing="ij")
        g, _ = self.evaluate(block, embed(A.reshape(-1), B.reshape(-1)))
        sx, sy = (v.reshape(A.shape) for v in self.screen(g[:, :3]))
        w, h = self.sc.width, self.sc.height
        box = []                         # screen box of each cell: its 3 x 3 points, and a margin for its curvature
        for s, most in ((sx, w), (sy, h)):
            pts = torch.stack([s[i:s.shape[0] - 2 + i:2, j:s.shape[1] - 2 + j:2] for i in range(3) for j in range(3)])
            lo, hi = pts.min(0)[0], pts.max(0)[0]
            pad = 0.25 * (hi - lo) + 0.05
            box += [(lo - pad).ceil().clamp(0, most).long().reshape(-1), ((hi + pad).floor().clamp(-1, most - 1)).long().reshape(-1)]
        nx, ny = (box[1] - box[0] + 1).clamp(min=0), (box[3] - box[2] + 1).clamp(min=0)
        count = nx * ny
        ca, cb = torch.meshgrid(0.5 * (ga[1:] + ga[:-1]), 0.5 * (gb[1:] + gb[:-1]), indexing="ij")
        wa, wb = torch.meshgrid(ga[1:] - ga[:-1], gb[1:] - gb[:-1], indexing="ij")
        got = []
        ends = count.cumsum(0)
        first = 0
        while first < len(count):                                     # cells, about 2^19 candidates at a time
            base = int(ends[first - 1]) if first else 0
            last = max(first + 1, int(torch.searchsorted(ends, base + (1 << 19))))
            sel = torch.arange(first, min(last, len(count)), device="cuda")
            first = min(last, len(count))
            n = count[sel]
            if int(n.sum()) == 0:
                continue
            cell = torch.repeat_interleave(sel, n)
            k = torch.arange(len(cell), device="cuda") - torch.repeat_interleave(n.cumsum(0) - n, n)
            px = box[0][cell] + k % nx[cell]
            py = box[2][cell] + torch.div(k, nx[cell], rounding_mode="floor")
            pix = py * w + px
            o, d = self.rays(pix)
            for da, db in ((0.0, 0.0), (-0.3, -0.3), (0.3, 0.3), (-0.3, 0.3), (0.3, -0.3)):
                hw, hb = wa.reshape(-1)[cell], wb.reshape(-1)[cell]
                a0, b0 = ca.reshape(-1)[cell], cb.reshape(-1)[cell]
                a, c = a0 + da * hw, b0 + db * hb
                ok = self.newton2(block, embed, ad, bd, o, d, a, c)
                a, c = ok[1], ok[2]
                keep = ok[0] & ((a - a0).abs() <= 1.5 * hw) & ((c - b0).abs() <= 1.5 * hb)
                keep &= (a >= -1e-12) & (a <= 1 + 1e-12) & (c >= -1e-12) & (c <= 1 + 1e-12)
                if not bool(keep.any()):
                    continue
                p = embed(a[keep].clamp(0, 1), c[keep].clamp(0, 1))
                g, der = self.evaluate(block, p)
                t = ((g[:, :3] - o[keep]) * d[keep]).sum(1)
                nrm = torch.linalg.cross(der[:, ad, :3], der[:, bd, :3])
                front = (nrm * d[keep]).sum(1) * (1.0 if side else -1.0) < 0
                got.append((pix[keep], t, front, p))
        return [torch.cat(v) for v in zip(*got)] if got else None

    def cells(self, b, direction):
        """Cell bounds along one face direction: about 4 cells a knot span,
        more where a span covers much of the model."""
        brk = np.unique(np.asarray(b.knots[direction], np.float64))
        brk = (brk - brk[0]) / (brk[-1] - brk[0])
        s = max(4, int(math.ceil(32.0 / (len(brk) - 1))))
        return _dev(np.concatenate([np.linspace(x, y, s, endpoint=False) for x, y in zip(brk[:-1], brk[1:])] + [[1.0]]))

    def newton2(self, block, embed, ad, bd, o, d, a, c):
        axis = torch.zeros_like(d)
        axis.scatter_(1, d.abs().argmin(1, keepdim=True), 1.0)
        e1 = torch.linalg.cross(d, axis)
        e1 = e1 / e1.norm(dim=1, keepdim=True)
        e2 = torch.linalg.cross(d, e1)
        a, c = a.clone(), c.clone()
        live = torch.arange(len(a), device="cuda")
        done = torch.zeros(len(a), dtype=torch.bool, device="cuda")
        for it in range(12):
            q = embed(a[live].clamp(0, 1), c[live].clamp(0, 1))
            g, der = self.evaluate(block, q)
            # beyond the face the patch is continued by its tangent plane
            over_a, over_c = a[live] - q[:, ad], c[live] - q[:, bd]
            g = g[:, :3] + over_a[:, None] * der[:, ad, :3] + over_c[:, None] * der[:, bd, :3]
            e = g - o[live]
            fx, fy = (e * e1[live]).sum(1), (e * e2[live]).sum(1)
            small = fx * fx + fy * fy <= (1e-13 * self.diag) ** 2
            done[live[small]] = True
            if it == 11:
                break
            xa, xc = (der[:, ad, :3] * e1[live]).sum(1), (der[:, bd, :3] * e1[live]).sum(1)
            ya, yc = (der[:, ad, :3] * e2[live]).sum(1), (der[:, bd, :3] * e2[live]).sum(1)
            det = xa * yc - xc * ya
            da, dc = (fy * xc - fx * yc) / det, (fx * ya - fy * xa) / det
            a[live], c[live] = a[live] + da.clamp(-0.2, 0.2), c[live] + dc.clamp(-0.2, 0.2)
            near = ~small & torch.isfinite(da) & torch.isfinite(dc) & (a[live] > -0.3) & (a[live] < 1.3) & \
                (c[live] > -0.3) & (c[live] < 1.3)
            live = live[near]
            if not len(live):
                break
        return done, a, c

    def pairs(self):
        """Entry/exit pairs of every pixel: (pixel, block, t0, t1, p0, p1)."""
        found = []
        for block in range(len(self.sc.blocks)):
            got = [x for x in (self.face_hits(block, f) for f in range(6)) if x is not None]
            if not got:
                continue
            pix, t, front, p = (torch.cat(v) for v in zip(*got))
            o = t.argsort(stable=True)
            o = o[pix[o].argsort(stable=True)]
            pix, t, front, p = pix[o], t[o], front[o], p[o]
            keep = torch.ones(len(pix), dtype=torch.bool, device="cuda")
            keep[1:] = (pix[1:] != pix[:-1]) | (t[1:] - t[:-1] > 1e-9 * self.diag) | (front[1:] != front[:-1])
            pix, t, front, p = pix[keep], t[keep], front[keep], p[keep]
            ok = (pix[1:] == pix[:-1]) & front[:-1] & ~front[1:]
            found.append((pix[:-1][ok], torch.full_like(pix[:-1][ok], block), t[:-1][ok], t[1:][ok], p[:-1][ok],
                          p[1:][ok]))
        return [torch.cat(v) for v in zip(*found)]

    # ---- samples
    def invert(self, block, g, p):
        tol = 1e-13 * self.diag
        p = p.clamp(0, 1)
        live = torch.arange(len(p), device="cuda")
        for _ in range(30):
            val, der = self.evaluate(block, p[live])
            F = val[:, :3] - g[live]
            nF = F.norm(dim=1)
            far = nF > tol
            live, F, nF, J = live[far], F[far], nF[far], der[far][:, :, :3].transpose(1, 2)
            if not len(live):
                break
            step = torch.linalg.solve_ex(J, -F[:, :, None])[0][:, :, 0]
            lam = torch.ones_like(nF)
            new = (p[live] + step).clamp(0, 1)
            for _ in range(6):
                worse = (self.evaluate(block, new)[0][:, :3] - g[live]).norm(dim=1) >= nF
                if not bool(worse.any()):
                    break
                lam = torch.where(worse, 0.5 * lam, lam)
                new = torch.where(worse[:, None], (p[live] + lam[:, None] * step).clamp(0, 1), new)
            moved = (new != p[live]).any(1)
            p[live] = new
            live = live[moved]
        return p

    def image(self):
        sc, w, h = self.sc, self.sc.width, self.sc.height
        out = torch.zeros(h * w, 4, dtype=F8, device="cuda")
        pix, block, t0, t1, p0, p1 = self.pairs()
        o, d = self.rays(pix)
        length = t1 - t0
        c0, c1 = t0.clone(), t1.clone()
        for n0, n1, n2, wp in sc.params.cut_planes:
            n = _dev([n0, n1, n2])
            fo, fd = o @ n + wp, d @ n
            tc = -fo / fd
            c1 = torch.where(fd > 0, torch.minimum(c1, tc), c1)
            c0 = torch.where(fd > 0, c0, torch.maximum(c0, tc))
        ok = c1 > c0
        p0, p1 = ((p0 + ((c - t0) / length)[:, None] * (p1 - p0))[ok] for c in (c0, c1))
        pix, block, t0, t1, o, d = pix[ok], block[ok], c0[ok], c1[ok], o[ok], d[ok]
        order = t0.argsort(stable=True)
        order = order[pix[order].argsort(stable=True)]
        pix, block, t0, t1, p0, p1, o, d = (v[order] for v in (pix, block, t0, t1, p0, p1, o, d))
        if not len(pix):
            return out.reshape(h, w, 4)
        # samples s_j = j ds, and the exit where it is not one of them
        ds, length = sc.params.ds, t1 - t0
        ns = (length / ds).floor()
        n = ns.long() + (length - ns * ds > 1e-12 * self.diag).long() + 1
        pair = torch.repeat_interleave(torch.arange(len(pix), device="cuda"), n)
        j = torch.arange(len(pair), device="cuda") - torch.repeat_interleave(n.cumsum(0) - n, n)
        s = torch.minimum(j.to(F8) * ds, length[pair])
        rho = torch.empty_like(s)
        for b in range(len(sc.blocks)):
            for at in (block[pair] == b).nonzero()[:, 0].split(8 * self.CHUNK):
                q = pair[at]
                g = o[q] + (t0[q] + s[at])[:, None] * d[q]
                p = p0[q] + (s[at] / length[q])[:, None] * (p1[q] - p0[q])
                rho[at] = self.scalar(b, self.invert(b, g, p))
        # intervals between consecutive samples of a pair, by rank along the pixel
        at = (j > 0).nonzero()[:, 0]
        ip = pix[pair[at]]
        new = torch.ones(len(ip), dtype=torch.bool, device="cuda")
        new[1:] = ip[1:] != ip[:-1]
        start = new.nonzero()[:, 0]
        many = torch.diff(torch.cat([start, torch.tensor([len(ip)], device="cuda")]))
        tf = sc.tf
        lo, hi = (tf.lo, tf.hi) if math.isfinite(tf.lo) and tf.hi > tf.lo else self.scalar_range()
        r, rgba = _dev(tf.r.astype(np.float64)), _dev(tf.rgba.astype(np.float64))
        K = sc.params.supersample_k
        acc = torch.zeros(len(start), 4, dtype=F8, device="cuda")
        live = torch.arange(len(start), device="cuda")
        for rank in range(int(many.max()) if len(many) else 0):
            live = live[(many[live] > rank) & (acc[live, 3] < sc.params.early_alpha)]
            if not len(live):
                break
            i = at[start[live] + rank]
            tau = tf.sigma * (s[i] - s[i - 1]) / K
            for k in range(K):
                x = ((rho[i - 1] + (k + 0.5) / K * (rho[i] - rho[i - 1]) - lo) / (hi - lo)).clamp(0, 1)
                m = (torch.searchsorted(r, x, right=True) - 1).clamp(0, len(r) - 2)
                f = ((x - r[m]) / (r[m + 1] - r[m]))[:, None]
                c = rgba[m] + f * (rgba[m + 1] - rgba[m])
                wgt = (1 - torch.exp(-tau * c[:, 3])) * (1 - acc[live, 3])
                acc[live] += wgt[:, None] * torch.cat([c[:, :3], torch.ones_like(c[:, :1])], 1)
        out[ip[start]] = acc
        return out.reshape(h, w, 4)
