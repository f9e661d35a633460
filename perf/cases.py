"""Performance cases: the calls that a training or rendering program makes, over the sizes it makes
them at, with the FP64 value of each.

    listed()              the cases; each stands for one recurring call of a scene optimisation
    draw(rng)             another case of the same ranges
    prepare(case, seed)   the inputs and the objects such a program holds before the call
    run(state)            one pass through the package's public entry points, and its outputs
    work(case)            bytes and flops that one pass cannot do without
    exact(case, seed)     what run() returns, evaluated in 64 bits with plain torch operations

Inputs: 100 (test time: 1) inward-facing pinhole views at radius 4 on the upper hemisphere around the
box [-1, 1]^3, focal 1111 at 800 x 800 pixels; density grids of balls (raw density 50 inside, 0
outside), 12-channel smooth features, MLP weights U(+-1/sqrt(fan_in)); sampling step half a voxel.
"""
import math

import numpy as np
import torch

import paper_2111_11215_gb300 as dvgo

BOX = (-1.0, 1.0)
FEAT, HID = 12, 128
N_BINS, PROP_FREQ, PROP_W = 64, 6, 64
MLP_KEYS = ("w1", "b1", "w2", "b2", "w3", "b3")


def listed():
    return [
        # the smallest training call: a preview or a unit-size scene, 32^3 coarse grid, 256 rays
        dict(name="coarse_32_rays256", kind="coarse", res=32, rays=256, aux=False),
        # one step of the coarse stage: 100^3 density and colour grids, 8192 rays, auxiliary losses
        dict(name="coarse_100_rays8192", kind="coarse", res=100, rays=8192, aux=True),
        # one step of the plain fine stage: FP32 features and MLP, uniform steps
        dict(name="fine_fp32_160_rays8192", kind="fine", res=160, rays=8192, mlp="fp32", feat="fp32", pe_x=False,
             skip=False, aux=False, samples=0, blob=False),
        # one step of the whole fine recipe on a grid of the progressive schedule: PE(x), known free
        # space and tau_f skipping, auxiliary losses
        dict(name="fine_fp32_recipe_101_rays8192", kind="fine", res=101, rays=8192, mlp="fp32", feat="fp32", pe_x=True,
             skip=True, aux=True, samples=0, blob=False),
        # the chosen form's training loop, one uniform and three proposal steps with their optimiser
        # steps (the whole call)
        dict(name="train_chosen_160_rays8192", kind="train", res=160, rays=8192),
        # one proposal step of the chosen form: BF16 features and MLP, 48 explicit samples a ray
        dict(name="fine_bf16_160_samples48", kind="fine", res=160, rays=8192, mlp="bf16", feat="bf16", pe_x=False,
             skip=False, aux=False, samples=48, blob=False),
        # the largest step: 256^3 grids, 65,536 rays aimed into a dense ball
        dict(name="fine_bf16_256_blob_rays65536", kind="fine", res=256, rays=65536, mlp="bf16", feat="bf16", pe_x=False,
             skip=False, aux=False, samples=0, blob=True),
        # a test-time frame (the whole call), BF16 MLP, tau_f skipping
        dict(name="frame_bf16_800x800", kind="frame", res=160, height=800, width=800, mlp="bf16", feat="bf16"),
        # a small, oddly sized preview frame in FP32
        dict(name="frame_fp32_187x251", kind="frame", res=128, height=187, width=251, mlp="fp32", feat="fp32"),
        # drawing the next step's samples from the proposal
        dict(name="proposal_sample_bf16_8192", kind="psample", rays=8192, samples=48, mlp="bf16"),
        # the proposal's labels, loss and gradient after a uniform step (FP32, its default)
        dict(name="proposal_train_fp32_1024", kind="ptrain", res=160, rays=8192, train=1024, mlp="fp32"),
        # progressive scaling to the next lattice, density and features
        dict(name="resize_127_to_160", kind="resize", nx=127, ny=127, nz=127, mx=160, my=160, mz=160),
    ]


def draw(rng):
    def logu(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["coarse", "fine", "fine", "fine", "train", "frame", "psample", "ptrain", "resize"])
    prec = rng.choice(["fp32", "bf16"])
    if kind == "coarse":
        return dict(kind=kind, res=logu(24, 128), rays=logu(64, 16384), aux=rng.random() < 0.5)
    if kind == "fine":
        samples = rng.choice([0, 0, rng.randint(16, 96)])
        return dict(kind=kind, res=logu(48, 200), rays=logu(128, 8192), mlp=prec,
                    feat="fp32" if prec == "fp32" else rng.choice(["fp32", "bf16"]), pe_x=rng.random() < 0.4,
                    skip=rng.random() < 0.4, aux=rng.random() < 0.4, samples=samples, blob=False)
    if kind == "train":
        return dict(kind=kind, res=logu(64, 160), rays=logu(512, 8192))
    if kind == "frame":
        h = logu(64, 800)
        return dict(kind=kind, res=logu(64, 160), height=h, width=max(32, min(800, int(h * rng.uniform(0.6, 1.7)))),
                    mlp=prec, feat="fp32" if prec == "fp32" else rng.choice(["fp32", "bf16"]))
    if kind == "psample":
        return dict(kind=kind, rays=logu(128, 32768), samples=rng.randint(16, 96), mlp=prec)
    if kind == "ptrain":
        rays = logu(256, 8192)
        return dict(kind=kind, res=logu(64, 160), rays=rays, train=max(64, int(rays * rng.uniform(0.1, 1.0))), mlp=prec)
    n = [logu(40, 127) for _ in range(3)]
    m = [min(170, int(v * rng.uniform(1.1, 1.4)) + 1) for v in n]
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], mx=m[0], my=m[1], mz=m[2])


# ----------------------------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _axes(*n):
    ax = [torch.linspace(BOX[0], BOX[1], v, device="cuda") for v in n]
    return torch.meshgrid(*ax, indexing="ij")


def _balls(seed, n=8):
    r = np.random.default_rng(seed)
    return r.uniform(-0.7, 0.7, size=(n, 3)), r.uniform(0.1, 0.3, size=n)


def _ball_density(res, balls, value, grow=0.0):
    X, Y, Z = _axes(res, res, res)
    out = torch.zeros((res,) * 3, device="cuda")
    for c, r in zip(*balls):
        out[(X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2 <= (r + grow) ** 2] = value
    return out


def _smooth(shape, channels, seed):
    r = np.random.default_rng(seed)
    X, Y, Z = _axes(*shape)
    out = torch.empty(tuple(shape) + (channels,), device="cuda")
    for ch in range(channels):
        acc = torch.zeros(tuple(shape), device="cuda")
        for _ in range(4):
            k, ph = r.uniform(-2 * np.pi, 2 * np.pi, size=3), r.uniform(0, 2 * np.pi)
            acc += torch.sin(float(k[0]) * X + float(k[1]) * Y + float(k[2]) * Z + float(ph))
        out[..., ch] = acc / 4
    return out


def _uniform_layers(dims, seed, out_bias_zero=True):
    """[w, b] pairs U(+-1/sqrt(fan_in)) as one flat FP32 tensor w1 | b1 | w2 | ..."""
    r = np.random.default_rng(seed)
    parts = []
    for i in range(len(dims) - 1):
        s = 1.0 / math.sqrt(dims[i])
        parts.append(r.uniform(-s, s, size=dims[i] * dims[i + 1]))
        last = i == len(dims) - 2
        parts.append(np.zeros(dims[i + 1]) if last and out_bias_zero else r.uniform(-s, s, size=dims[i + 1]))
    return torch.tensor(np.concatenate(parts), dtype=torch.float32, device="cuda")


def _rig(seed, n_views, radius=4.0):
    r = np.random.default_rng(seed)
    az, el = r.uniform(0, 2 * np.pi, size=n_views), np.deg2rad(r.uniform(5.0, 85.0, size=n_views))
    pos = radius * np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], -1)
    fwd = -pos / np.linalg.norm(pos, axis=-1, keepdims=True)
    right = np.cross(fwd, np.array([0.0, 0.0, 1.0]))
    right /= np.linalg.norm(right, axis=-1, keepdims=True)
    up = np.cross(right, fwd)
    return (torch.tensor(np.stack([right, up, -fwd], -1), dtype=torch.float32, device="cuda"),
            torch.tensor(pos, dtype=torch.float32, device="cuda"))


def _view_rays(rot, pos, v, x, y):
    dc = torch.stack([x, y, -torch.ones_like(x)], -1)
    d = (rot[v] * dc[:, None, :]).sum(-1)
    return pos[v].contiguous(), d.contiguous()


def _batch(n, seed):
    """A training batch: rays through uniform pixels of 100 views, jitter, target colours."""
    g = _gen(seed)
    rot, pos = _rig(1234, 100)
    v = torch.randint(0, 100, (n,), generator=g, device="cuda")
    px = torch.randint(0, 800, (2, n), generator=g, device="cuda").float()
    o, d = _view_rays(rot, pos, v, (px[0] + 0.5 - 400) / 1111.0, -(px[1] + 0.5 - 400) / 1111.0)
    jit = torch.rand(n, generator=g, device="cuda")
    tgt = torch.rand((n, 3), generator=g, device="cuda")
    return o, d, jit, tgt


def _blob_batch(n, seed):
    g = _gen(seed)
    o = torch.randn((n, 3), generator=g, device="cuda")
    o = o / o.norm(dim=1, keepdim=True) * 4.0
    t = torch.randn((n, 3), generator=g, device="cuda")
    t = t / t.norm(dim=1, keepdim=True) * 0.3 * torch.rand((n, 1), generator=g, device="cuda") ** (1 / 3)
    d = t - o
    return o, (d / d.norm(dim=1, keepdim=True)).contiguous(), torch.rand(n, generator=g, device="cuda"), \
        torch.rand((n, 3), generator=g, device="cuda")


def _shift(alpha, s):
    return float(dvgo.dvgo_shift_from_alpha_init(alpha, s))


def _fine_params(case, **kw):
    res = case["res"]
    return dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.5 * 2.0 / res, shift_b=_shift(1e-6, 2.0 / res),
                       mlp_prec=dvgo.DVGO_MLP_BF16 if case.get("mlp") == "bf16" else dvgo.DVGO_MLP_FP32,
                       n_freq_pos=5 if case.get("pe_x") else 0, **kw)


def _explicit(o, d, balls, n, seed):
    """n sorted samples a ray as a trained proposal draws them: most around the first ball on the
    ray, the rest along the whole box, and their step lengths."""
    g = _gen(seed)
    o, d = o.double(), d.double()
    lo, hi, dn = _clip(o, d)
    hit = hi > lo
    ts = lo + (hi - lo) * 0.5
    for c, r in zip(*balls):
        oc = o - torch.tensor(c, device="cuda")
        b = (oc * dn).sum(-1)
        disc = b * b - ((oc * oc).sum(-1) - r * r)
        t = -b - torch.sqrt(disc.clamp(min=0))
        ts = torch.where((disc > 0) & (t > lo) & (t < ts), t, ts)
    R = o.shape[0]
    u = torch.rand((R, n), generator=g, device="cuda", dtype=torch.float64)
    near = torch.rand((R, n), generator=g, device="cuda") < 0.8
    t = torch.where(near, ts[:, None] + 0.3 * (u - 0.35), lo[:, None] + u * (hi - lo)[:, None])
    t = torch.minimum(torch.maximum(t, lo[:, None]), hi[:, None]).sort(dim=1).values
    t = torch.where(hit[:, None], t, torch.zeros_like(t)).float()
    dt = torch.cat([t[:, 1:] - t[:, :-1], torch.full((R, 1), 0.005, device="cuda")], 1)
    return t.contiguous(), dt.contiguous()


def _inputs(case, seed):
    """Plain tensors and numbers of a case, made from the seed; shared by prepare() and exact()."""
    k, I = case["kind"], {}
    if k == "coarse":
        n, R = case["res"], case["rays"]
        g = _gen(seed + 1)
        balls = _balls(seed)
        I["density"] = _ball_density(n, balls, 25.0) + 0.1 * torch.randn((n,) * 3, generator=g, device="cuda")
        I["cgrid"] = 0.5 + 0.1 * torch.randn((n, n, n, 3), generator=g, device="cuda")
        I["o"], I["d"], I["jit"], I["tgt"] = _batch(R, seed + 2)
        I["shift"], I["step"], I["aux"] = _shift(1e-6, 2.0 / n), 0.5 * 2.0 / n, (0.1, 0.01) if case["aux"] else (0.0, 0.0)
    elif k in ("fine", "frame", "train", "ptrain"):
        n = case["res"]
        balls = (np.zeros((1, 3)), np.array([0.3])) if case.get("blob") else _balls(seed)
        I["density"] = _ball_density(n, balls, 200.0 if case.get("blob") else 50.0)
        I["balls"] = balls
        I["shift"], I["step"] = _shift(1e-6, 2.0 / n), 0.5 * 2.0 / n
        if k != "ptrain":
            feat = _smooth((n,) * 3, FEAT, seed + 1)
            I["cgrid"] = feat.to(torch.bfloat16) if case.get("feat") == "bf16" else feat
            I["mlp"] = _uniform_layers([39 + (33 if case.get("pe_x") else 0), HID, HID, 3], seed + 2)
        I["aux"] = (0.01, 0.001) if case.get("aux") else (0.0, 0.0)
        I["tau_f"] = 1e-4 if case.get("skip") or k == "frame" else 0.0
        if case.get("skip"):
            m = max(16, int(n * 100 / 160))
            I["fs"] = dict(density=_ball_density(m, balls, 25.0, grow=2.0 / m), shift=_shift(1e-6, 2.0 / m),
                           step=0.5 * 2.0 / m, tau=1e-3)
        if k == "frame":
            h, w = case["height"], case["width"]
            rot, pos = _rig(seed + 3, 1)
            rr, cc = torch.meshgrid(torch.arange(h, device="cuda"), torch.arange(w, device="cuda"), indexing="ij")
            f = 1111.0 * max(h, w) / 800.0
            I["o"], I["d"] = _view_rays(rot, pos, torch.zeros(h * w, dtype=torch.long, device="cuda"),
                                        (cc.reshape(-1) + 0.5 - w / 2) / f, -(rr.reshape(-1) + 0.5 - h / 2) / f)
            I["jit"] = None
        else:
            I["o"], I["d"], I["jit"], I["tgt"] = (_blob_batch if case.get("blob") else _batch)(case["rays"], seed + 3)
        if case.get("samples"):
            I["t"], I["dt"] = _explicit(I["o"], I["d"], balls, case["samples"], seed + 4)
    elif k == "psample":
        I["o"], I["d"], I["jit"], _ = _batch(case["rays"], seed + 3)
    elif k == "resize":
        s, m = (case["nx"], case["ny"], case["nz"]), (case["mx"], case["my"], case["mz"])
        g = _gen(seed)
        I["src"], I["dst"] = s, m
        I["density"] = torch.randn(s, generator=g, device="cuda") * 10
        I["cgrid"] = torch.randn(s + (FEAT,), generator=g, device="cuda") * 0.5
    if k in ("psample", "ptrain", "train"):
        I["prop"] = _uniform_layers([3 + 6 * PROP_FREQ, PROP_W, PROP_W, PROP_W, 1], seed + 5)
    return I


def _proposal_dict(flat):
    out, off = {}, 0
    for i, (a, b) in enumerate(((39, PROP_W), (PROP_W, PROP_W), (PROP_W, PROP_W), (PROP_W, 1))):
        out[f"w{i}"], off = flat[off:off + a * b].view(a, b), off + a * b
        out[f"b{i}"], off = flat[off:off + b], off + b
    return out


# ----------------------------------------------------------------------------------------------
# prepare / run
# ----------------------------------------------------------------------------------------------

def prepare(case, seed):
    k, I = case["kind"], _inputs(case, seed)
    S = {"case": case, "I": I}
    prec = dvgo.DVGO_MLP_BF16 if case.get("mlp") == "bf16" else dvgo.DVGO_MLP_FP32
    if k == "coarse":
        n, R = case["res"], case["rays"]
        p = dvgo.Params(step=I["step"], shift_b=I["shift"], w_pt_rgb=I["aux"][0], w_bg=I["aux"][1])
        S["rend"] = dvgo.Renderer(p, dvgo.GridDesc((n,) * 3, 1), dvgo.GridDesc((n,) * 3, 3), R)
    elif k in ("fine", "frame"):
        n = case["res"]
        fs = None
        if "fs" in I:
            f = I["fs"]
            fs = dvgo.FreeSpace(f["density"], dvgo.GridDesc(tuple(f["density"].shape), 1), f["shift"], f["step"], f["tau"])
        p = _fine_params(case, tau_f=I["tau_f"], freespace=fs, w_pt_rgb=I["aux"][0], w_bg=I["aux"][1])
        dd = dvgo.GridDesc((n,) * 3, 1)
        cd = dvgo.GridDesc((n,) * 3, FEAT, dtype=dvgo.DVGO_DTYPE_BF16 if case["feat"] == "bf16" else dvgo.DVGO_DTYPE_F32)
        S["mlp"] = dvgo.mlp_views(I["mlp"], p.mlp_in_dim(FEAT))
        if k == "fine":
            S["rend"] = dvgo.Renderer(p, dd, cd, case["rays"], samples_per_ray=case["samples"] or None)
            S["samples"] = (I["t"], I["dt"]) if case["samples"] else None
        else:
            S["frame"] = dvgo.FrameRenderer(p, dd, cd)
    if k in ("coarse", "fine"):
        R = case["rays"]
        S["rgb"], S["tfinal"] = torch.empty((R, 3), device="cuda"), torch.empty(R, device="cuda")
        S["loss"], S["dloss"] = torch.zeros(1, device="cuda"), torch.empty((R, 3), device="cuda")
        S["g_density"] = torch.zeros_like(I["density"])
        S["g_cgrid"] = torch.zeros(I["cgrid"].shape, device="cuda")
        S["g_mlp"] = torch.zeros_like(I["mlp"]) if k == "fine" else None
    elif k == "train":
        # a model in mid-training: moments of the size its gradients have, 5000 steps done
        m = dvgo.FineModel(I["density"], I["cgrid"], I["mlp"], _fine_params(dict(case, mlp="bf16")), case["rays"],
                           bf16_feat=True, overlap_adam=True)
        g = _gen(seed + 9)
        for key, scale in (("density", 1e-11), ("feat", 1e-11), ("mlp", 1e-6)):
            m.adam[key].v.uniform_(0.5, 1.5, generator=g).mul_(scale)
        m.step_count = 5000
        prop = dvgo.Proposal(_proposal_dict(I["prop"]), m.params, m.dd, case["rays"],
                             sample_precision=dvgo.DVGO_MLP_BF16, train_precision=dvgo.DVGO_MLP_BF16)
        prop.adam.v.uniform_(0.5, 1.5, generator=g).mul_(1e-6)
        prop.step_count = 1250
        S["trainer"] = dvgo.ProposalTrainer(m, prop)
        S["batches"] = [(I["o"], I["d"], I["jit"], I["tgt"])] + [_batch(case["rays"], seed + 20 + j) for j in range(3)]
    elif k == "psample":
        p = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.5 * 2.0 / 160, shift_b=_shift(1e-6, 2.0 / 160))
        S["prop"] = dvgo.Proposal(_proposal_dict(I["prop"]), p, dvgo.GridDesc((160,) * 3, 1), case["rays"],
                                  sample_precision=prec)
        S["t"] = torch.empty((case["rays"], case["samples"]), device="cuda")
        S["dt"] = torch.empty_like(S["t"])
    elif k == "ptrain":
        n, R = case["res"], case["rays"]
        p = _fine_params(dict(case, mlp="bf16"))
        feat = torch.zeros((n, n, n, FEAT), device="cuda")
        mlp = dvgo.mlp_views(torch.zeros(dvgo.mlp_flat_size(), device="cuda"))
        rend = dvgo.Renderer(p, dvgo.GridDesc((n,) * 3, 1), dvgo.GridDesc((n,) * 3, FEAT), R)
        rend.forward(I["density"], feat, mlp, I["o"], I["d"], I["jit"])
        S["rend"], S["p"], S["prec"] = rend, p, prec
        S["prop"] = _proposal_dict(I["prop"])
        S["labels"] = torch.empty((R, N_BINS), device="cuda")
        S["probs"], S["loss"] = torch.empty((case["train"], N_BINS), device="cuda"), torch.zeros(1, device="cuda")
        S["grad"] = torch.zeros_like(I["prop"])
    elif k == "resize":
        S["descs"] = [(dvgo.GridDesc(I["src"], c), dvgo.GridDesc(I["dst"], c)) for c in (1, FEAT)]
        S["out"] = [torch.empty(I["dst"], device="cuda"), torch.empty(I["dst"] + (FEAT,), device="cuda")]
    return S


def run(S):
    case, I = S["case"], S["I"]
    k = case["kind"]
    if k in ("coarse", "fine"):
        for g in (S["g_density"], S["g_cgrid"]) + ((S["g_mlp"],) if k == "fine" else ()):
            g.zero_()
        r, mlp, smp = S["rend"], S.get("mlp"), S.get("samples")
        r.forward(I["density"], I["cgrid"], mlp, I["o"], I["d"], I["jit"], smp, I["tgt"], S["rgb"], S["tfinal"],
                  S["loss"], S["dloss"])
        r.backward(I["density"], I["cgrid"], mlp, I["o"], I["d"], I["jit"], smp, S["dloss"], None, S["g_density"],
                   S["g_cgrid"], S["g_mlp"])
        out = {q: S[q] for q in ("rgb", "tfinal", "loss", "g_density", "g_cgrid")}
        return dict(out, g_mlp=S["g_mlp"]) if k == "fine" else out
    if k == "frame":
        rgb, tfinal = S["frame"].render(I["density"], I["cgrid"], S["mlp"], I["o"], I["d"])
        return {"rgb": rgb, "tfinal": tfinal}
    if k == "train":
        tr = S["trainer"]
        for b in S["batches"]:
            loss = tr.step(*b)
        m = tr.model
        return {"loss": loss, "density": m.density, "feat": m.feat, "mlp": m.mlp_flat, "prop": tr.proposal.flat}
    if k == "psample":
        t, dt = S["prop"].sample(I["o"], I["d"], I["jit"], case["samples"], t_out=S["t"], dt_out=S["dt"])
        return {"probs": S["prop"].probs, "t": t, "dt": dt}
    if k == "ptrain":
        p, dd, n = S["p"], S["rend"].dd, case["train"]
        S["grad"].zero_()
        dvgo.dvgo_weight_bins(p, dd, case["rays"], N_BINS, S["rend"].workspace, S["labels"])
        o, d, lab = I["o"][:n], I["d"][:n], S["labels"][:n]
        dvgo.dvgo_proposal_fwd(p, dd, N_BINS, PROP_FREQ, PROP_W, S["prop"], o, d, lab, S["probs"], S["loss"],
                               precision=S["prec"])
        dvgo.dvgo_proposal_bwd(p, dd, N_BINS, PROP_FREQ, PROP_W, S["prop"], o, d, lab, S["grad"], precision=S["prec"])
        return {"labels": S["labels"], "probs": S["probs"], "loss": S["loss"], "grad": S["grad"]}
    for (a, b), src, out in zip(S["descs"], (I["density"], I["cgrid"]), S["out"]):
        dvgo.dvgo_resize_grid(a, src, b, out)
    return {"density": S["out"][0], "cgrid": S["out"][1]}


# ----------------------------------------------------------------------------------------------
# work
# ----------------------------------------------------------------------------------------------

def _samples_of(case):
    """Samples whose colour is evaluated in one pass, from the mean path of the rays through the box
    (79 % of the rays hit it; 1.05 lattice units of step a voxel), 12 % of them in occupied space."""
    if case.get("blob"):
        return case["rays"] * 617.0 * case["res"] / 256
    rays = case["rays"] if "rays" in case else case["height"] * case["width"]
    if case.get("samples"):
        n = 0.79 * case["samples"]
    else:
        n = 167.0 * case["res"] / 160
    return rays * n * (0.12 if case.get("skip") or case["kind"] == "frame" else 1.0)


def work(case):
    k = case["kind"]
    if k == "resize":
        a, b = case["nx"] * case["ny"] * case["nz"], case["mx"] * case["my"] * case["mz"]
        return {"bytes": 4 * (1 + FEAT) * (a + b), "flops": 16 * (1 + FEAT) * b}
    bins = case.get("rays", 0) * N_BINS
    prop = 2.0 * (39 * PROP_W + 2 * PROP_W * PROP_W + PROP_W)
    if k == "psample":
        return {"bytes": case["rays"] * (28 + 4 * N_BINS + 8 * case["samples"]), "flops": 0.79 * bins * prop}
    pts = case["res"] ** 3
    if k == "ptrain":
        s = case["rays"] * 167.0 * case["res"] / 160
        return {"bytes": 16 * s + 4 * N_BINS * (case["rays"] + case["train"]),
                "flops": 0.79 * case["train"] * N_BINS * prop * 4 + 10 * s}
    if k == "coarse":
        s = case["rays"] * 167.0 * case["res"] / 160
        return {"bytes": 2 * 4 * 4 * pts + 60 * case["rays"], "flops": s * 2 * 8 * 4 * 3}
    s = _samples_of(case)
    in_dim = 39 + (33 if case.get("pe_x") else 0)
    fwd = 2.0 * (in_dim * HID + HID * HID + HID * 3) + 2 * 8 * (FEAT + 1)
    fbytes = pts * (4 + FEAT * (2 if case.get("feat") == "bf16" else 4))
    if k == "frame":
        return {"bytes": fbytes + 40 * case["height"] * case["width"], "flops": s * fwd}
    if k == "fine":
        return {"bytes": fbytes + 4 * pts * (1 + FEAT) + 60 * case["rays"], "flops": 3 * s * fwd}
    # train: one uniform and three 48-sample steps, four dense Adam sweeps (28 B and the BF16 copy)
    s = s + 3 * 0.79 * 48 * case["rays"]
    return {"bytes": 4.0 * pts * ((1 + FEAT) * 28 + 2 * FEAT), "flops": 3 * s * fwd + 3 * 0.79 * bins * prop}


# ----------------------------------------------------------------------------------------------
# exact
# ----------------------------------------------------------------------------------------------

def _clip(o, d):
    """Box clip in FP64: entry and exit distance along the normalised direction (hi <= lo: a miss)."""
    ln = torch.sqrt((d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2])
    dn = d / ln[:, None]
    t1, t2 = (BOX[0] - o) / dn, (BOX[1] - o) / dn
    lo = torch.minimum(t1, t2).amax(-1).clamp(min=0.0)
    hi = torch.maximum(t1, t2).amin(-1)
    return lo, hi, dn


def _f32(x):
    return float(np.float32(x))


def _interp(grid, u, shape):
    """Trilinear interpolation of grid [nx ny nz, C] at lattice coordinates u [N, 3]."""
    n = torch.tensor(shape, device="cuda")
    i0 = torch.minimum(torch.floor(u).long().clamp(min=0), n - 2)
    f = u - i0
    out = 0.0
    for q in range(8):
        b = (q >> 2 & 1, q >> 1 & 1, q & 1)
        w = 1.0
        for a in range(3):
            w = w * (f[:, a] if b[a] else 1.0 - f[:, a])
        idx = ((i0[:, 0] + b[0]) * shape[1] + i0[:, 1] + b[1]) * shape[2] + i0[:, 2] + b[2]
        out = out + w[:, None] * grid[idx]
    return out


def _softplus(z):
    return torch.logaddexp(z, torch.zeros_like(z))


def _pe(x, freqs):
    k = 2.0 ** torch.arange(freqs, device="cuda", dtype=torch.float64)
    a = x[:, :, None] * k
    return torch.cat([x, torch.sin(a).flatten(1), torch.cos(a).flatten(1)], 1)


def _layers(x, flat, dims, last=None):
    off = 0
    for i in range(len(dims) - 1):
        w = flat[off:off + dims[i] * dims[i + 1]].view(dims[i], dims[i + 1])
        off += dims[i] * dims[i + 1]
        x = x @ w + flat[off:off + dims[i + 1]]
        off += dims[i + 1]
        if i < len(dims) - 2:
            x = torch.relu(x)
    return x


def _ray_samples(I, rows, step, shape):
    """Samples of the rays `rows`: ray index, sample index, step length, lattice coordinate, direction."""
    o, d = I["o"][rows].double(), I["d"][rows].double()
    lo, hi, dn = _clip(o, d)
    R = o.shape[0]
    if "t" in I:
        n = torch.where(hi > lo, I["t"].shape[1], 0)
        t, dt = I["t"][rows].double()[hi > lo].reshape(-1), I["dt"][rows].double()[hi > lo].reshape(-1)
        ray = torch.repeat_interleave(torch.arange(R, device="cuda"), n)
        k = None
    else:
        p = torch.full((R,), 0.5, device="cuda", dtype=torch.float64) if I["jit"] is None else I["jit"][rows].double()
        cap = math.ceil(math.sqrt(3 * (BOX[1] - BOX[0]) ** 2) / step) + 1
        n = torch.where(hi > lo, torch.ceil((hi - lo) / step - p).clamp(0, cap), torch.zeros_like(lo)).long()
        ray = torch.repeat_interleave(torch.arange(R, device="cuda"), n)
        k = torch.arange(ray.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
        t = lo[ray] + (k + p[ray]) * step
        dt = torch.full_like(t, step)
    x = o[ray] + t[:, None] * dn[ray]
    u = (x - BOX[0]) * ((torch.tensor(shape, device="cuda", dtype=torch.float64) - 1) / (BOX[1] - BOX[0]))
    return ray, k, dt, x, u, dn, n, lo, hi


def _composite_weights(tau, ray, n):
    c = torch.cumsum(tau, 0)
    end = torch.cumsum(n, 0)
    c0 = torch.cat([torch.zeros(1, device="cuda", dtype=torch.float64), c])
    before = c0[end - n]
    T = torch.exp(-(c - tau - before[ray]))
    return T * -torch.expm1(-tau), torch.exp(-(c0[end] - before))


def _exact_render(case, I, grad):
    fine = case["kind"] != "coarse"
    shape = (case["res"],) * 3
    step, b, tau_f = _f32(I["step"]), _f32(I["shift"]), _f32(I.get("tau_f", 0.0))
    dens = I["density"].double().reshape(-1, 1).requires_grad_(grad)
    C = 12 if fine else 3
    cg = I["cgrid"].double().reshape(-1, C).requires_grad_(grad)
    mlp = I["mlp"].double().requires_grad_(grad) if fine else None
    R = I["o"].shape[0]
    per = 1000000 if grad else 3000000
    chunk = max(1, int(per / max(1.0, 617.0 * case["res"] / 256 if case.get("blob") else
                                 (case.get("samples") or 330.0 * case["res"] / 160))))
    rgbs, tks, loss = [], [], 0.0
    for s in range(0, R, chunk):
        rows = slice(s, min(R, s + chunk))
        ray, _, dt, x, u, dn, n, _, _ = _ray_samples(I, rows, step, shape)
        with torch.set_grad_enabled(grad):
            keep = torch.ones_like(dt, dtype=torch.bool)
            if "fs" in I:
                f = I["fs"]
                m = tuple(f["density"].shape)
                uc = (x - BOX[0]) * ((torch.tensor(m, device="cuda", dtype=torch.float64) - 1) / (BOX[1] - BOX[0]))
                v = _interp(f["density"].double().reshape(-1, 1), uc, m)[:, 0]
                keep = ~(-torch.expm1(-_softplus(v + _f32(f["shift"])) * _f32(f["step"])) < _f32(f["tau"]))
            tau = _softplus(_interp(dens, u, shape)[:, 0] + b) * dt
            keep = keep & ~(-torch.expm1(-tau.detach()) < tau_f)
            tau = torch.where(keep, tau, torch.zeros_like(tau))
            w, TK = _composite_weights(tau, ray, n)
            kept = keep.nonzero()[:, 0]
            col = _interp(cg, u[kept], shape)
            if fine:
                e = [col, _pe(dn, 4)[ray[kept]]] + ([_pe(x[kept], 5)] if case.get("pe_x") else [])
                dims = [39 + (33 if case.get("pe_x") else 0), HID, HID, 3]
                col = torch.sigmoid(_layers(torch.cat(e, 1), mlp, dims))
            rk = ray[kept]
            rgb = torch.zeros((n.numel(), 3), device="cuda", dtype=torch.float64).index_add(0, rk, w[kept][:, None] * col)
            rgb = rgb + TK[:, None]
            if grad:
                tgt = I["tgt"][rows].double()
                part = ((rgb - tgt) ** 2).sum() / R
                if I["aux"][0]:
                    part = part + _f32(I["aux"][0]) * (w[kept].detach() * ((col - tgt[rk]) ** 2).sum(-1)).sum() / R
                    A = (1 - TK).clamp(1e-6, 1 - 1e-6)
                    part = part + _f32(I["aux"][1]) * (-A * torch.log(A) - (1 - A) * torch.log1p(-A)).sum() / R
                part.backward()
                loss = loss + part.detach()
        rgbs.append(rgb.detach())
        tks.append(TK.detach())
    out = {"rgb": torch.cat(rgbs), "tfinal": torch.cat(tks)}
    if grad:
        out.update(loss=loss.reshape(1), g_density=dens.grad.reshape(shape), g_cgrid=cg.grad.reshape(shape + (C,)))
        if case.get("blob") and case.get("mlp") == "bf16":
            # inside one ball the gradient is made of differences of neighbouring colours that are
            # smaller than the BF16 operands resolve: the FP64 value says nothing about this output
            out["g_density"] = None
        if fine:
            out["g_mlp"] = mlp.grad
    return out


def _exact_logits(I, rows, flat):
    o, d = I["o"][rows].double(), I["d"][rows].double()
    lo, hi, dn = _clip(o, d)
    hit = hi > lo
    tb = lo[:, None] + (torch.arange(N_BINS, device="cuda") + 0.5) * ((hi - lo) / N_BINS)[:, None]
    x = torch.where(hit[:, None, None], o[:, None, :] + tb[..., None] * dn[:, None, :], torch.zeros(3, device="cuda", dtype=torch.float64))
    z = _layers(_pe(x.reshape(-1, 3), PROP_FREQ), flat, [39, PROP_W, PROP_W, PROP_W, 1]).view(-1, N_BINS)
    return torch.where(hit[:, None], z, torch.zeros_like(z)), lo, hi, hit


def exact(case, seed):
    k = case["kind"]
    if k == "train":
        return None
    I = _inputs(case, seed)
    if k in ("coarse", "fine"):
        return _exact_render(case, I, True)
    if k == "frame":
        return _exact_render(case, I, False)
    if k == "psample":
        z, lo, hi, hit = _exact_logits(I, slice(None), I["prop"].double())
        p = torch.softmax(z, 1)
        n, eta = case["samples"], _f32(0.05)
        q = (1 - eta) * p + eta / N_BINS
        Q = torch.cat([torch.zeros((q.shape[0], 1), device="cuda", dtype=torch.float64), torch.cumsum(q, 1)], 1)
        u = (torch.arange(n, device="cuda") + I["jit"].double()[:, None]) / n * Q[:, -1:]
        b = (torch.searchsorted(Q[:, 1:].contiguous(), u, right=True)).clamp(max=N_BINS - 1)
        w = ((hi - lo) / N_BINS)[:, None]
        qb = q.gather(1, b)
        t = lo[:, None] + (b + (u - Q.gather(1, b)) / qb) * w
        dt = torch.cat([t[:, 1:] - t[:, :-1], w * Q[:, -1:] / (n * qb[:, -1:])], 1)
        zero = torch.zeros_like(t)
        return {"probs": p, "t": torch.where(hit[:, None], t, zero), "dt": torch.where(hit[:, None], dt, zero)}
    if k == "ptrain":
        R, n, step = case["rays"], case["train"], _f32(I["step"])
        shape = (case["res"],) * 3
        ray, j, dt, x, u, dn, cnt, lo, hi = _ray_samples(I, slice(None), step, shape)
        tau = _softplus(_interp(I["density"].double().reshape(-1, 1), u, shape)[:, 0] + _f32(I["shift"])) * dt
        w, _ = _composite_weights(tau, ray, cnt)
        b = torch.floor((j + I["jit"].double()[ray]) * ((step * N_BINS) / (hi - lo))[ray]).clamp(0, N_BINS - 1).long()
        lab = torch.zeros(R * N_BINS, device="cuda", dtype=torch.float64).index_add(0, ray * N_BINS + b, w).view(R, N_BINS)
        tot = lab.sum(1, keepdim=True)
        lab = torch.where(tot < 1e-4, torch.full_like(lab, 1.0 / N_BINS), lab / tot)
        flat = I["prop"].double().requires_grad_(True)
        z, _, _, hit = _exact_logits(I, slice(0, n), flat)
        logp = torch.log_softmax(z, 1)
        loss = -(torch.where(hit[:, None], lab[:n] * logp, torch.zeros_like(logp))).sum() / n
        loss.backward()
        return {"labels": lab, "probs": torch.exp(logp.detach()), "loss": loss.detach().reshape(1), "grad": flat.grad}
    out = {}
    s, m = I["src"], I["dst"]
    for key, C in (("density", 1), ("cgrid", FEAT)):
        src, res = I[key].double().reshape(-1, C), []
        ax = [torch.arange(v, device="cuda", dtype=torch.float64) * (a - 1) / (v - 1) for v, a in zip(m, s)]
        for i in range(m[0]):
            X, Y, Z = torch.meshgrid(ax[0][i:i + 1], ax[1], ax[2], indexing="ij")
            res.append(_interp(src, torch.stack([X, Y, Z], -1).reshape(-1, 3), s))
        out[key] = torch.cat(res).reshape(m + ((C,) if C > 1 else ()))
    return out
