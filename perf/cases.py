"""Timed cases of libnam: what a renderer and a trainer have the library do.

Evaluation of a frame's shading points in each arithmetic, of frames whose
material varies per pixel, importance sampling, and the training steps.
Sizes are those of the repository's workloads, tests and benchmark: frames of
1280x720 to 3840x2160 and small batches, latent pyramids of 256^2 to 2048^2
texels, the paper's decoder sizes, training batches of 50,000 to 262,144.
All inputs are seeded and synthetic, made on the GPU.
"""
import math

import numpy as np
import torch

import paper_2305_02678_gb300 as nam

DEV = "cuda"


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # a picker, a thumbnail or the last stragglers of a wavefront: one small batch, latency
        dict(name="shade_1k", kind="shade", prec="f16", n=1000, tex=256, tex_f16=True, frame="paper", H=32, NH=2,
             filt="trilinear", addr="wrap", out=3, cosine=False, warp=False),
        # a full-HD frame of one material in the library's main arithmetic
        dict(name="shade_1080p", kind="shade", prec="f16", n=1920 * 1080, tex=2048, tex_f16=True, frame="mlp", H=64,
             NH=2, filt="trilinear", addr="wrap", out=3, cosine=False, warp=True),
        # the paper's largest decoder on a 4K frame, one texel fetch per query picked at random
        dict(name="shade_4k_3x64", kind="shade", prec="f16", n=3840 * 2160, tex=2048, tex_f16=True, frame="paper",
             H=64, NH=3, filt="stochastic", addr="wrap", out=3, cosine=True, warp=True),
        # an offline bake or a preview of a model under training: FP32 texels, no frame, a 2x32 decoder
        dict(name="fp32_64k", kind="shade", prec="f32", n=65536, tex=256, tex_f16=False, frame="none", H=32, NH=2,
             filt="trilinear", addr="wrap", out=3, cosine=False, warp=False),
        # a 720p frame at full precision (the reference a reduced-precision material is compared with)
        dict(name="fp32_720p", kind="shade", prec="f32", n=1280 * 720, tex=2048, tex_f16=True, frame="mlp", H=64,
             NH=2, filt="trilinear", addr="wrap", out=3, cosine=False, warp=True),
        # the E4M3 form on a frame whose size is no multiple of anything
        dict(name="shade_fp8_odd", kind="shade", prec="fp8", n=1597 * 899, tex=1024, tex_f16=True, frame="mlp", H=64,
             NH=2, filt="trilinear", addr="clamp", out=3, cosine=False, warp=True),
        # a wavefront in no order: a material drawn per pixel
        dict(name="binned_1080p", kind="many", how="binned", ids="random", mats=16, n=1920 * 1080, tex=1024, H=64,
             NH=2, frame="mlp"),
        # a frame of 16 surfaces: materials in screen regions, a code path per tile
        dict(name="select_regions", kind="many", how="select", ids="regions", mats=16, n=1920 * 1080, tex=1024, H=64,
             NH=2, frame="mlp"),
        # one BSDF sample and its density for each pixel of a path-traced frame
        dict(name="sample_1080p", kind="sample", n=1920 * 1080, tex=2048),
        # one step of fitting the latent texture, the frame and the decoder
        dict(name="train_262k", kind="train", n=262144, tex=1024, H=64, frame="mlp", out=3),
        # one step of the first training phase: the latents come from the encoder
        dict(name="train_encoder_131k", kind="encoder", n=131072, tex=256, H=64, frame="mlp"),
        # torch owns the loss and the optimiser: forward and backward through autograd
        dict(name="autograd_50k", kind="autograd", n=49999, tex=256, H=32, frame="mlp"),
    ]


def draw(rng):
    def logn(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["shade", "shade", "shade", "shade", "many", "sample", "train", "encoder", "autograd"])
    c = dict(kind=kind)
    if kind == "shade":
        prec = rng.choice(["f16", "f16", "f32", "fp8"])
        H, NH = rng.choice([(16, 2), (32, 2), (64, 2), (64, 3)])
        if prec == "f32":
            n = logn(1000, 1500000)
        else:
            n = logn(1000, 6000000)
        c.update(prec=prec, n=n, tex=rng.choice([256, 512, 1000, 1024, 2048]), tex_f16=rng.random() < 0.75,
                 frame=rng.choice(["none", "mlp", "paper"]), H=H, NH=NH,
                 filt=rng.choice(["trilinear", "trilinear", "stochastic"]),
                 addr=rng.choice(["wrap", "wrap", "clamp"]), out=rng.choice([3, 3, 6]),
                 cosine=rng.random() < 0.5, warp=rng.random() < 0.7)
    elif kind == "many":
        c.update(how=rng.choice(["binned", "select"]), ids=rng.choice(["random", "regions"]),
                 mats=rng.choice([2, 5, 16, 40]), n=logn(20000, 2500000), tex=rng.choice([256, 512, 1024]),
                 H=rng.choice([32, 64]), NH=2, frame=rng.choice(["mlp", "paper"]))
    elif kind == "sample":
        c.update(n=logn(2000, 4000000), tex=rng.choice([512, 1024, 2048]))
    elif kind == "train":
        c.update(n=logn(20000, 400000), tex=rng.choice([256, 512, 1024]), H=rng.choice([32, 64]),
                 frame=rng.choice(["mlp", "mlp", "none"]), out=rng.choice([3, 3, 6]))
    elif kind == "encoder":
        c.update(n=logn(20000, 300000), tex=rng.choice([256, 512]), H=rng.choice([32, 64]), frame="mlp")
    else:
        c.update(n=logn(10000, 300000), tex=rng.choice([256, 512]), H=rng.choice([16, 32, 64]),
                 frame=rng.choice(["mlp", "none"]))
    return c


# ----------------------------------------------------------------------------
# seeded inputs
# ----------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _levels(tex):
    L = 1
    while tex >> L:
        L += 1
    return L


def _geometry(tex):
    L = _levels(tex)
    w = [max(1, tex >> l) for l in range(L)]
    off = np.concatenate([[0], np.cumsum([x * x for x in w])])
    return L, w, [int(o) for o in off[:-1]], int(off[-1])


def _pyramid(seed, salt, tex, f16):
    """[texels, 8] independent N(0, 0.5) latents, on the GPU."""
    _, _, _, n = _geometry(tex)
    z = torch.randn((n, 8), generator=_gen(seed, salt), device=DEV, dtype=torch.float32) * 0.5
    return z.half() if f16 else z


def _mlp(rng, widths):
    """Glorot-uniform weights, biases in +-0.1: [(W [out][in], b [out])] in FP32."""
    out = []
    for a, b in zip(widths[:-1], widths[1:]):
        lim = math.sqrt(6.0 / (a + b))
        out.append((rng.uniform(-lim, lim, (b, a)).astype(np.float32),
                    rng.uniform(-0.1, 0.1, b).astype(np.float32)))
    return out


def _model(seed, salt, frame, H, NH, out):
    rng = np.random.default_rng([int(seed), salt])
    f = None if frame == "none" else _mlp(rng, (8, 16, 6)) if frame == "mlp" else _mlp(rng, (8, 12))
    d = _mlp(rng, (20 if frame == "paper" else 14,) + (H,) * NH + (out,))
    return f, d


def _hemisphere(g, n):
    r, p = torch.rand((2, n), generator=g, device=DEV, dtype=torch.float64)
    s = r.sqrt()
    p = p * (2.0 * math.pi)
    return s * p.cos(), s * p.sin(), (1.0 - r).sqrt()


def _frame_size(n):
    """Width of a 16:9 frame of n pixels (the last row may be short)."""
    return max(1, int(round(math.sqrt(n * 16.0 / 9.0))))


def _queries(seed, salt, n, tex, warp):
    """n planar FP32 queries: uniform over the texture with any level, or a
    frame whose uv follow a smooth random warp (1 to 64 texels per pixel) with
    the level of its pixel footprint; cosine-weighted directions."""
    g = _gen(seed, salt)
    L = _levels(tex)
    if warp:
        rng = np.random.default_rng([int(seed), salt])
        width = _frame_size(n)
        zoom0 = width / tex
        k0 = rng.integers(1, 4, 2) * rng.choice([-1, 1], 2)
        ph0 = rng.uniform(0, 2 * math.pi)
        ks = rng.integers(1, 4, (4, 2)) * rng.choice([-1, 1], (4, 2))
        am, ph, an = rng.uniform(0, 0.02, 4), rng.uniform(0, 2 * math.pi, 4), rng.uniform(0, 2 * math.pi, 4)
        i = torch.arange(n, device=DEV, dtype=torch.float64)
        py = torch.floor(i / width)
        px = i - py * width + 0.5
        py = py + 0.5

        def at(x, y):
            p0, p1 = x / width, y / width
            s = 0.5 + 0.5 * torch.sin(2 * math.pi * (float(k0[0]) * p0 + float(k0[1]) * p1) + ph0)
            m = zoom0 * torch.exp2(6.0 * s)
            u, v = 0.5 + (p0 - 0.5) * m, 0.5 + (p1 - 0.5) * m
            for k, a, h, e in zip(ks, am, ph, an):
                w = a * torch.sin(2 * math.pi * (float(k[0]) * p0 + float(k[1]) * p1) + h)
                u, v = u + w * math.cos(e), v + w * math.sin(e)
            return u, v

        u, v = at(px, py)
        (ax, bx), (cx, dx) = at(px + 1, py), at(px - 1, py)
        (ay, by), (cy, dy) = at(px, py + 1), at(px, py - 1)
        det = ((ax - cx) * (by - dy) - (ay - cy) * (bx - dx)).abs() * 0.25
        lod = 0.5 * torch.log2(torch.clamp(det * float(tex) * float(tex), min=1e-30))
    else:
        u, v, lod = torch.rand((3, n), generator=g, device=DEV, dtype=torch.float64)
        lod = lod * (L - 1)
    wi, wo = _hemisphere(g, n), _hemisphere(g, n)
    xi = torch.rand(n, generator=g, device=DEV, dtype=torch.float32)
    q = dict(zip(("u", "v", "lod", "wix", "wiy", "wiz", "wox", "woy", "woz"), (u, v, lod) + wi + wo))
    q = {k: t.float().contiguous() for k, t in q.items()}
    q["xi"] = xi.clamp(max=1.0 - 2.0 ** -24)
    return q


def _ids(seed, salt, n, mats, how):
    g = _gen(seed, salt)
    if how == "random":
        return torch.randint(0, mats, (n,), generator=g, device=DEV, dtype=torch.int32)
    width = _frame_size(n)
    i = torch.arange(n, device=DEV)
    x, y = (i % width).float(), (i // width).float()
    site = torch.rand((mats, 2), generator=g, device=DEV)
    sx, sy = site[:, 0] * width, site[:, 1] * (n / width)
    best, ids = None, torch.zeros(n, device=DEV, dtype=torch.int32)
    for m in range(mats):
        d = (x - sx[m]) ** 2 + (y - sy[m]) ** 2
        if best is None:
            best = d
        else:
            ids = torch.where(d < best, torch.full_like(ids, m), ids)
            best = torch.minimum(best, d)
    return ids


def _targets(seed, salt, n):
    """Reflectances as a measured or procedural material gives them: mostly
    diffuse, some highlights."""
    g = _gen(seed, salt)
    a = torch.rand((n, 3), generator=g, device=DEV)
    spec = torch.rand((n, 1), generator=g, device=DEV)
    return (0.02 + 0.28 * a + 0.5 * spec ** 8).contiguous()


# ----------------------------------------------------------------------------
# what a program keeps, and one pass
# ----------------------------------------------------------------------------
class Owner:
    """A context, closed (its materials freed) once nothing refers to it: the
    state, or a tensor over memory that its materials own."""

    def __init__(self):
        self.ctx = nam.Context(0)

    def __del__(self):
        self.ctx.close()


class _View:
    """CUDA array interface over FP32 device memory of `owner`, which the tensor made from it keeps."""

    def __init__(self, owner, ptr, *shape):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (int(ptr), False), "version": 3}


class State:
    def __init__(self, **kw):
        self.__dict__.update(kw)


_PREC = {"f32": 0, "f16": 1, "fp8": 2}


def _geom_args(case):
    return case["tex"], case["tex"], _levels(case["tex"])


def _shade_material(ctx, case, seed, q):
    pyr = _pyramid(seed, 1, case["tex"], case["tex_f16"]).cpu().numpy()
    frame, dec = _model(seed, 2, case["frame"], case["H"], case["NH"], case["out"])
    kw = dict(filter=int(case["filt"] == "stochastic"), address=int(case["addr"] == "clamp"))
    if case["prec"] == "fp8":
        m32 = ctx.material(*_geom_args(case), pyr, frame, dec, precision=0, **kw)
        scale = nam.B.nam_fp8_calibrate(ctx.h, m32.h, q, min(case["n"], 65536), torch.cuda.current_stream())
        m32.destroy()
        kw["act_scale"] = scale[:len(dec)]
    return ctx.material(*_geom_args(case), pyr, frame, dec, precision=_PREC[case["prec"]], **kw)


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    owner = Owner()
    ctx = owner.ctx
    st = State(owner=owner, ctx=ctx, case=dict(case), step=0)
    if kind == "shade":
        st.q = _queries(seed, 3, n, case["tex"], case["warp"])
        st.mat = _shade_material(ctx, case, seed, st.q)
    elif kind == "many":
        st.q = _queries(seed, 3, n, case["tex"], True)
        st.ids = _ids(seed, 4, n, case["mats"], case["ids"])
        pyr = _pyramid(seed, 1, case["tex"], True).cpu().numpy()
        st.mats = []
        for k in range(case["mats"]):
            frame, dec = _model(seed, 100 + k, case["frame"], case["H"], case["NH"], 3)
            st.mats.append(ctx.material(*_geom_args(case), pyr, frame, dec, precision=1))
    elif kind == "sample":
        st.q = _queries(seed, 3, n, case["tex"], True)
        pyr = _pyramid(seed, 1, case["tex"], True).cpu().numpy()
        frame, dec = _model(seed, 2, "mlp", 64, 2, 3)
        smp = _mlp(np.random.default_rng([int(seed), 5]), (11, 32, 32, 32, 9))
        st.mat = ctx.material(*_geom_args(case), pyr, frame, dec, precision=1, sampler=smp)
        st.u = torch.rand((n, 3), generator=_gen(seed, 6), device=DEV).clamp(max=1.0 - 2.0 ** -24).contiguous()
    elif kind in ("train", "encoder"):
        st.q = _queries(seed, 3, n, case["tex"], False)
        pyr = _pyramid(seed, 1, case["tex"], False).cpu().numpy()
        frame, dec = _model(seed, 2, case["frame"], case["H"], 2, case.get("out", 3))
        enc = None
        if kind == "encoder":
            enc = _mlp(np.random.default_rng([int(seed), 7]), (4, 32, 32, 8))
            st.attrs = torch.rand((n, 4), generator=_gen(seed, 8), device=DEV)
        st.mat = ctx.material(*_geom_args(case), pyr, frame, dec, precision=0, trainable=True, encoder=enc)
        st.target = _targets(seed, 9, n)
        if case.get("out", 3) == 6:
            st.target_albedo = _targets(seed, 10, n)
        dev = torch.device(DEV, ctx.device)
        p, z = st.mat.params()
        st.params = torch.as_tensor(_View(owner, p, st.mat.info.n_params), device=dev)
        st.pyramid = torch.as_tensor(_View(owner, z, st.mat.info.texels, 8), device=dev)
        if kind == "encoder":
            e = nam.B.nam_material_encoder(ctx.h, st.mat.h)
            st.enc = torch.as_tensor(_View(owner, e, nam.B.encoder_param_count(4)), device=dev)
    else:
        from paper_2305_02678_gb300 import autograd
        st.q = _queries(seed, 3, n, case["tex"], False)
        pyr = _pyramid(seed, 1, case["tex"], False).cpu().numpy()
        frame, dec = _model(seed, 2, case["frame"], case["H"], 2, 3)
        st.model = autograd.NeuralMaterial(ctx, *_geom_args(case), pyr, frame, dec)
        st.loss = autograd.log_l1_loss
        st.target = _targets(seed, 9, n)
    return st


def run(st):
    case, B = st.case, nam.B
    kind, n = case["kind"], case["n"]
    stream = torch.cuda.current_stream()
    if kind == "shade":
        flags = B.NAM_OUT_COSINE if case["cosine"] else 0
        if case["out"] == 6:
            return st.mat.eval_albedo(st.q, flags=flags)
        return st.mat.eval(st.q, flags=flags)
    if kind == "many":
        out = torch.empty((n, 3), dtype=torch.float32, device=DEV)
        call = B.nam_eval_binned if case["how"] == "binned" else B.nam_eval_select
        call(st.ctx.h, [m.h for m in st.mats], st.q, st.ids, n, out, stream)
        return out
    if kind == "sample":
        wo = torch.empty((n, 3), dtype=torch.float32, device=DEV)
        pdf = torch.empty(n, dtype=torch.float32, device=DEV)
        B.nam_sample(st.ctx.h, st.mat.h, st.q, n, st.u, wo, pdf, stream)
        return wo, pdf
    if kind == "train":
        st.step += 1
        if case["out"] == 6:
            loss = B.nam_train_step_albedo(st.ctx.h, st.mat.h, st.q, st.target, st.target_albedo, n, step=st.step,
                                           stream=stream)
        else:
            loss = B.nam_train_step(st.ctx.h, st.mat.h, st.q, st.target, n, step=st.step, stream=stream)
        return loss, st.params, st.pyramid
    if kind == "encoder":
        st.step += 1
        loss = B.nam_train_step_encoded(st.ctx.h, st.mat.h, st.q, st.attrs, st.target, n, step=st.step, stream=stream)
        return loss, st.params, st.enc
    st.model.params.grad = st.model.pyramid.grad = None
    rgb = st.model(st.q)
    loss = st.loss(rgb, st.target)
    loss.backward()
    return loss.detach(), rgb.detach(), st.model.params.grad, st.model.pyramid.grad


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def _macs(case):
    frame, H, NH, out = case.get("frame", "mlp"), case.get("H", 64), case.get("NH", 2), case.get("out", 3)
    f = {"none": 0, "mlp": 8 * 16 + 16 * 6, "paper": 8 * 12}[frame]
    return f + (20 if frame == "paper" else 14) * H + (NH - 1) * H * H + out * H


def _texels(case, warp):
    """Distinct texels that the queries read: about 0.42 per query of a warped
    frame (counted at 1920x1080), or the expectation for uniform queries."""
    L, w, _, total = _geometry(case["tex"])
    n = case["n"]
    if warp:
        return min(total, 0.42 * n)
    got = 0.0
    for l in range(L):
        reads = 4.0 * n / (L - 1) * (1 if l in (0, L - 1) else 2)
        got += w[l] ** 2 * (1.0 - math.exp(-reads / w[l] ** 2))
    return got


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "shade":
        fields = 10 if case["filt"] == "stochastic" else 9
        tex = _texels(case, case["warp"]) * (16 if case["tex_f16"] else 32)
        return {"bytes": n * (4 * fields + 4 * case["out"]) + tex, "flops": 2.0 * n * _macs(case)}
    if kind == "many":
        return {"bytes": n * (36 + 4 + 12) + _texels(case, True) * 16, "flops": 2.0 * n * _macs(case)}
    if kind == "sample":
        return {"bytes": n * (24 + 12 + 16) + _texels(case, True) * 16,
                "flops": 2.0 * n * (11 * 32 + 2 * 32 * 32 + 32 * 9)}
    macs = _macs(case)
    texels = _geometry(case["tex"])[3]
    if kind == "train":
        # forward, deltas and weight gradients; Adam reads and writes value and two moments of each texel
        return {"bytes": n * (36 + 4 * case["out"]) + texels * 32 * 6, "flops": 6.0 * n * macs}
    if kind == "encoder":
        enc = 4 * 32 + 32 * 32 + 32 * 8
        return {"bytes": n * (24 + 16 + 12), "flops": 6.0 * n * (macs + enc)}
    # each query field, the target, rgb and its gradient; the texels read, the pyramid's gradient written
    return {"bytes": n * (36 + 12 + 24) + _texels(case, False) * 32 + texels * 32, "flops": 8.0 * n * macs}


# ----------------------------------------------------------------------------
# the same results in 64 bits, by plain torch
# ----------------------------------------------------------------------------
def _latent(pyr, tex, q, stochastic, clamp):
    """pyr [texels, 8] FP64; queries FP64."""
    L, w, off, _ = _geometry(tex)
    dev = pyr.device
    W = torch.tensor(w, device=dev)
    O = torch.tensor(off, device=dev)
    lod = q["lod"].clamp(0, L - 1)
    l0 = torch.floor(lod).long()
    l1 = (l0 + 1).clamp(max=L - 1)
    t = lod - l0
    if stochastic:
        parts = [(torch.where(q["xi"] < t, l1, l0), torch.ones_like(t))]
    else:
        parts = [(l0, 1.0 - t), (l1, t)]
    z = 0.0
    for l, wt in parts:
        Wl = W[l]

        def axis(x):
            x = x * Wl - 0.5
            x0 = torch.floor(x)
            f = x - x0
            i0 = x0.long()
            if clamp:
                hi = Wl - 1
                return torch.minimum(i0.clamp(min=0), hi), torch.minimum((i0 + 1).clamp(min=0), hi), f
            return i0 % Wl, (i0 + 1) % Wl, f

        x0, x1, fx = axis(q["u"])
        y0, y1, fy = axis(q["v"])
        o = O[l]
        for y, x, c in ((y0, x0, (1 - fx) * (1 - fy)), (y0, x1, fx * (1 - fy)),
                        (y1, x0, (1 - fx) * fy), (y1, x1, fx * fy)):
            z = z + (wt * c)[:, None] * pyr[o + y * Wl + x]
    return z


def _cross(a, b):
    return torch.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1], a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],
                        a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], 1)


def _unit(a):
    return a / a.norm(dim=1, keepdim=True)


def _forward(z, wi, wo, frame, kind, dec):
    """RGB (and albedo) from latents and directions, all FP64 torch."""
    if kind == "mlp":
        h = torch.relu(z @ frame[0][0].T + frame[0][1])
        r = h @ frame[1][0].T + frame[1][1]
        pairs = [(r[:, :3], r[:, 3:], True)]
    elif kind == "paper":
        r = z @ frame[0][0].T + frame[0][1]
        pairs = [(r[:, :3], r[:, 3:6], False), (r[:, 6:9], r[:, 9:], False)]
    else:
        pairs = None
    if pairs is None:
        x = torch.cat([z, wi, wo], 1)
    else:
        rows = []
        for nr, tr, gs in pairs:
            nn = _unit(nr)
            tt = _unit(tr - (tr * nn).sum(1, keepdim=True) * nn) if gs else _unit(tr)
            bb = _unit(_cross(nn, tt))
            rows += [tt, bb, nn]
        loc = [torch.stack([(r_ * d).sum(1) for r_ in rows], 1) for d in (wi, wo)]
        x = torch.cat([z] + loc, 1)
    for k, (W, b) in enumerate(dec):
        x = x @ W.T + b
        if k + 1 < len(dec):
            x = torch.relu(x)
    return x


def _t64(layers, prec="f32"):
    out = []
    for k, (W, b) in enumerate(layers or []):
        W, b = torch.from_numpy(W).to(DEV), torch.from_numpy(b).to(DEV)
        if prec != "f32":
            b = b.half()
            if prec == "fp8" and 0 < k < len(layers) - 1:
                s = 1.0
                top = float(W.abs().max())
                while top / s > 448.0:
                    s *= 2.0
                while top / (s * 0.5) <= 448.0:
                    s *= 0.5
                W = (W.double() / s).float().to(torch.float8_e4m3fn).double() * s
            else:
                W = W.half()
        out.append((W.double(), b.double()))
    return out


def _dirs(q, s):
    return torch.stack([q[s + "x"], q[s + "y"], q[s + "z"]], 1)


def _q64(q, a, b):
    return {k: t[a:b].double() for k, t in q.items()}


_CHUNK = 1 << 19


def _exact_shade(case, seed, q, pyr, frame, dec, kind, pick=None):
    rgb = []
    for a in range(0, case["n"], _CHUNK):
        c = _q64(q, a, a + _CHUNK)
        z = _latent(pyr, case["tex"], c, case.get("filt") == "stochastic", case.get("addr") == "clamp")
        y = _forward(z, _dirs(c, "wi"), _dirs(c, "wo"), frame, kind, dec)
        if case.get("cosine"):
            y = torch.cat([y[:, :3] * c["wiz"].clamp(min=0)[:, None], y[:, 3:]], 1)
        rgb.append(y)
    return torch.cat(rgb)


def _loss(y, case, target, target_albedo=None):
    g = y[:, :3]
    d = torch.log1p(torch.relu(g)) - torch.log1p(target)
    loss = (d.abs() + 0.01 * torch.relu(-g)).mean()
    if target_albedo is not None:
        loss = loss + ((y[:, 3:] - target_albedo) ** 2).mean()
    return loss


def _flat(layers):
    return torch.cat([t.reshape(-1) for W, b in layers for t in (W, b)])


def _grad_layers(layers):
    return [(W.requires_grad_(True), b.requires_grad_(True)) for W, b in layers]


def _flat_grad(layers):
    return torch.cat([t.grad.reshape(-1) for W, b in layers for t in (W, b)])


def _adam1(p, g, lr, eps=1e-8):
    """The first Adam step: both moments' bias corrections cancel."""
    return p - lr * g / (g.abs() + eps)


def _exact_many(case, seed):
    q = _queries(seed, 3, case["n"], case["tex"], True)
    ids = _ids(seed, 4, case["n"], case["mats"], case["ids"])
    pyr = _pyramid(seed, 1, case["tex"], True).double()
    out = torch.zeros((case["n"], 3), device=DEV, dtype=torch.float64)
    for k in range(case["mats"]):
        frame, dec = _model(seed, 100 + k, case["frame"], case["H"], case["NH"], 3)
        frame, dec = _t64(frame, "f16"), _t64(dec, "f16")
        at = torch.nonzero(ids == k)[:, 0]
        for a in range(0, at.numel(), _CHUNK):
            i = at[a:a + _CHUNK]
            c = {f: t[i].double() for f, t in q.items()}
            z = _latent(pyr, case["tex"], c, False, False)
            out[i] = _forward(z, _dirs(c, "wi"), _dirs(c, "wo"), frame, case["frame"], dec)
    return out


def _exact_sample(case, seed):
    """The directions.  Their densities have no such value: at grazing half
    vectors a density follows the last bits of its own direction."""
    q = _queries(seed, 3, case["n"], case["tex"], True)
    pyr = _pyramid(seed, 1, case["tex"], True).double()
    smp = _t64(_mlp(np.random.default_rng([int(seed), 5]), (11, 32, 32, 32, 9)))
    u = torch.rand((case["n"], 3), generator=_gen(seed, 6), device=DEV).clamp(max=1.0 - 2.0 ** -24).double()
    wos = []
    for a in range(0, case["n"], _CHUNK):
        c = _q64(q, a, a + _CHUNK)
        uu = u[a:a + _CHUNK]
        wi = _dirs(c, "wi")
        o = torch.cat([_latent(pyr, case["tex"], c, False, False), wi], 1)
        for k, (W, b) in enumerate(smp):
            o = o @ W.T + b
            if k < 3:
                o = torch.relu(o)
        w = torch.softmax(o[:, [0, 3]], 1)
        qt = torch.where(o.abs() < 2, o * (1 - o.abs() / 4), torch.sign(o))
        qs = o * (1 + o.abs() / 2)
        al = 1e-3 + (1 - 1e-3) * 0.5 * (qt + 1)
        wd, mdx, mdy = w[:, 0], qs[:, 1], qs[:, 2]
        ax, ay, rho, msx, msy = al[:, 4], al[:, 5], 0.99 * qt[:, 6], qs[:, 7], qs[:, 8]
        s = (1 - rho * rho).sqrt()
        r, ph = uu[:, 0].sqrt(), 2 * math.pi * uu[:, 1]
        lx, ly, lz = r * ph.cos(), r * ph.sin(), (1 - uu[:, 0]).clamp(min=0).sqrt()
        nd = _unit(torch.stack([-mdx, -mdy, torch.ones_like(mdx)], 1))
        aa = -1.0 / (1.0 + nd[:, 2])
        bb = nd[:, 0] * nd[:, 1] * aa
        t = torch.stack([1 + nd[:, 0] ** 2 * aa, bb, -nd[:, 0]], 1)
        dif = t * lx[:, None] + _cross(nd, t) * ly[:, None] + nd * lz[:, None]
        h = _unit(torch.stack([ax * lx - msx * lz, ay * rho * lx + ay * s * ly - msy * lz, lz], 1))
        spec = 2 * (wi * h).sum(1, keepdim=True) * h - wi
        wo = torch.where((uu[:, 2] < wd)[:, None], dif, spec)
        wos.append(wo)
    return torch.cat(wos), None


def _exact_train(case, seed):
    kind, n = case["kind"], case["n"]
    q = _queries(seed, 3, n, case["tex"], False)
    pyr = _pyramid(seed, 1, case["tex"], False).double()
    frame, dec = _model(seed, 2, case["frame"], case["H"], 2, case.get("out", 3))
    frame, dec = _grad_layers(_t64(frame)), _grad_layers(_t64(dec))
    target = _targets(seed, 9, n).double()
    talb = _targets(seed, 10, n).double() if case.get("out", 3) == 6 else None
    enc = None
    if kind == "encoder":
        enc = _grad_layers(_t64(_mlp(np.random.default_rng([int(seed), 7]), (4, 32, 32, 8))))
        attrs = torch.rand((n, 4), generator=_gen(seed, 8), device=DEV).double()
    else:
        pyr.requires_grad_(True)
    loss, ys = 0.0, []
    step = _CHUNK // 4
    for a in range(0, n, step):
        c = _q64(q, a, a + step)
        if enc is None:
            z = _latent(pyr, case["tex"], c, False, False)
        else:
            z = attrs[a:a + step]
            for k, (W, b) in enumerate(enc):
                z = z @ W.T + b
                if k < 2:
                    z = torch.relu(z)
        y = _forward(z, _dirs(c, "wi"), _dirs(c, "wo"), frame, case["frame"], dec)
        share = c["u"].numel() / n
        part = _loss(y, case, target[a:a + step], None if talb is None else talb[a:a + step]) * share
        part.backward()
        loss += float(part.detach())
        ys.append(y.detach())
    with torch.no_grad():
        gp = torch.cat([_flat_grad(frame), _flat_grad(dec)]) if frame else _flat_grad(dec)
        p = torch.cat([_flat(frame), _flat(dec)]) if frame else _flat(dec)
        if kind == "autograd":
            return torch.tensor(loss, dtype=torch.float64), torch.cat(ys), gp, pyr.grad
        p = _adam1(p, gp, 1e-3)
        if kind == "encoder":
            return loss, p, _adam1(_flat(enc), _flat_grad(enc), 1e-3)
        return loss, p, _adam1(pyr.detach(), pyr.grad, 1e-2)


def exact(case, seed):
    kind = case["kind"]
    if kind == "shade":
        q = _queries(seed, 3, case["n"], case["tex"], case["warp"])
        pyr = _pyramid(seed, 1, case["tex"], case["tex_f16"]).double()
        frame, dec = _model(seed, 2, case["frame"], case["H"], case["NH"], case["out"])
        prec = case["prec"]
        fw = _t64(frame, "f16" if prec == "fp8" else prec)
        y = _exact_shade(case, seed, q, pyr, fw, _t64(dec, prec), case["frame"])
        return (y[:, :3].contiguous(), y[:, 3:].contiguous()) if case["out"] == 6 else y
    if kind == "many":
        return _exact_many(case, seed)
    if kind == "sample":
        return _exact_sample(case, seed)
    return _exact_train(case, seed)
