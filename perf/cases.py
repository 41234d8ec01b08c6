"""Performance cases of the library: the calls a reconstruction makes, from one
small face to the paper's image size, through the public entry points.

A case is a dict of plain values; `kind` selects the call and the rest its
sizes.  The sizes are those of the repository's own workloads (the small C1
face, the paper-scale C2 face, the large C5 face, the serving mix) and the
ranges around them.  Scenes and library contexts are what a program keeps for
every face it reconstructs; the parameters, targets and adjoint images come
from the seed.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2101_05356_gb300 import autograd, facert, optim, synth


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the smallest fused step (render + loss + all gradients): launches and latency
        dict(name="step_small", kind="step", mesh="c1", width=64, height=64, spp=4, lights=8, stage="", tex=128),
        # the paper-scale face's step, the benchmark's headline
        dict(name="step_paper", kind="step", mesh="c2", width=256, height=256, spp=16, lights=40, stage="", tex=512),
        # the paper's image size under its 20-light icosahedral stage, light geometry optimised too
        dict(name="step_stage_512", kind="step", mesh="c2", width=512, height=512, spp=16, lights=20, stage="ico",
             tex=512),
        # a large image: hit records exceed their buffer, textures of 2048^2
        dict(name="step_large", kind="step", mesh="c5", width=1024, height=1024, spp=64, lights=80, stage="",
             tex=2048),
        # an evaluation render of a ragged image, no gradients
        dict(name="forward_ragged", kind="forward", mesh="c2", width=203, height=155, spp=8, lights=40, tex=512),
        # the autograd function under an environment map: forward, then the re-tracing backward
        dict(name="autograd_env", kind="autograd", mesh="c2", width=128, height=128, spp=8, env=32, block=4, tex=512),
        # one step of the server: faces of mixed size, sample count and stage, BF16 morph
        dict(name="serving_batch", kind="batch", mesh="c2", faces=8, largest=384, spp=32, lights=40, tex=512),
        # statistical albedo of a batch on the tensor cores (the served Stage I)
        dict(name="albedo_batch", kind="albedo", faces=8, tex=512, columns=80, bf16=True),
        # its transpose, texture gradients of a batch to coefficients
        dict(name="albedo_adjoint_batch", kind="albedo_adjoint", faces=8, tex=512, columns=80),
        # one face's FP32 albedo and its transpose (the plain Stage I)
        dict(name="albedo_one", kind="albedo_both", faces=1, tex=512, columns=80),
        # the Stage II optimiser step over the three textures
        dict(name="adam_textures", kind="adam", tex=512),
        # the photometric loss alone at the paper's image size
        dict(name="loss_512", kind="loss", width=512, height=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "forward", "autograd", "batch", "batch", "albedo",
                       "albedo_adjoint", "albedo_both", "adam", "loss"])
    if kind == "step":
        mesh = rng.choice(["c1", "c2", "c2"])
        stage = rng.choice(["", "", "ico"])
        return dict(kind=kind, mesh=mesh, width=_log(rng, 48, 512), height=_log(rng, 48, 512),
                    spp=rng.choice([4, 8, 16, 32]), lights=20 if stage else rng.choice([8, 20, 40, 80]), stage=stage,
                    tex=rng.choice([128, 256, 512]) if mesh == "c1" else 512)
    if kind == "forward":
        return dict(kind=kind, mesh=rng.choice(["c1", "c2"]), width=_log(rng, 48, 512), height=_log(rng, 48, 512),
                    spp=rng.choice([1, 4, 8, 16]), lights=rng.choice([8, 40, 80]), tex=512)
    if kind == "autograd":
        return dict(kind=kind, mesh=rng.choice(["c1", "c2"]), width=_log(rng, 48, 256), height=_log(rng, 48, 256),
                    spp=rng.choice([4, 8, 16]), env=32, block=rng.choice([4, 8]), tex=512)
    if kind == "batch":
        return dict(kind=kind, mesh=rng.choice(["c1", "c2"]), faces=rng.randint(2, 12), largest=_log(rng, 96, 448),
                    spp=rng.choice([8, 16, 32]), lights=40, tex=512)
    if kind == "albedo":
        return dict(kind=kind, faces=rng.randint(1, 12), tex=_log(rng, 96, 512), columns=rng.randint(20, 80),
                    bf16=rng.random() < 0.6)
    if kind in ("albedo_adjoint", "albedo_both"):
        return dict(kind=kind, faces=rng.randint(1, 12), tex=_log(rng, 96, 512), columns=rng.randint(20, 80))
    if kind == "adam":
        return dict(kind=kind, tex=_log(rng, 96, 1024))
    return dict(kind="loss", width=_log(rng, 48, 1024), height=_log(rng, 48, 1024))


# --------------------------------------------------------------------------
# scenes and contexts (kept by a program across faces)
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _mesh(config):
    return synth.make_scene(config, tex_size=4, n_lights=1)


def _scene(mesh, width, height, spp, tex, lights=0, stage="", env=0, block=0):
    base = _mesh(mesh)
    geo = None
    if env:
        records, d, a = synth.env_blocks(env, block)
    elif stage:
        records, d, a = synth.polyhedral_stage(stage, 3.0, 0.25)
        geo = synth.polyhedral_stage_geometry(stage)
    else:
        records = synth.light_stage(lights, 3.0, 0.5, mesh == "c1")
        d, a = np.full(lights, 3.0, np.float32), np.ones(lights, np.float32)
    return dataclasses.replace(base, width=width, height=height, spp=spp, tex_size=tex, lights=records, light_d=d,
                               light_a=a, stage=geo, env_size=env)


@functools.lru_cache(maxsize=6)
def _renderer(mesh, width, height, spp, tex, lights, stage, env, block, flags, max_batch):
    sc = _scene(mesh, width, height, spp, tex, lights, stage, env, block)
    return facert.Renderer(sc, edge_spp=1, flags=flags, seed=0, max_batch=max_batch)


@functools.lru_cache(maxsize=2)
def _albedo_model(tex, columns):
    """Smooth columns (white noise at a 24th of the resolution, interpolated)
    of RMS 0.08 / (1 + k) and 0.01 / (1 + k), the scales of synth.albedo_model."""
    g = torch.Generator().manual_seed(31)
    out = []
    for lo, hi, rms in ((0.35, 0.65, 0.08), (0.05, 0.05, 0.01)):
        mean = lo + (hi - lo) * _field(g, 3, tex, tex, 16)
        cols = torch.randn(columns, 3, 24, 24, generator=g) * (rms / (1.0 + torch.arange(columns))).view(-1, 1, 1, 1)
        cols = torch.nn.functional.interpolate(cols, size=(tex, tex), mode="bilinear", align_corners=True)
        out += [mean.permute(1, 2, 0).contiguous().numpy(), cols.permute(0, 2, 3, 1).contiguous().numpy()]
    return synth.AlbedoModel(*[np.ascontiguousarray(x, np.float32) for x in out])


@functools.lru_cache(maxsize=2)
def _albedo_renderer(tex, columns, bf16, max_batch):
    sc = dataclasses.replace(_scene("c1", 64, 64, 4, tex, lights=8), albedo=_albedo_model(tex, columns))
    return facert.Renderer(sc, flags=facert.FLAG_MORPH_BF16 if bf16 else 0, max_batch=max_batch)


# --------------------------------------------------------------------------
# inputs from the seed
# --------------------------------------------------------------------------
def _field(g, channels, height, width, cells):
    """Smooth field in [0, 1] [channels, height, width]."""
    x = torch.rand(1, channels, cells, cells, generator=g)
    return torch.nn.functional.interpolate(x, size=(height, width), mode="bilinear", align_corners=True)[0]


def _picture(g, height, width):
    """A photograph-like target [height, width, 3]: a shaded ellipse on black with N(0, 0.01) pixel noise."""
    y = (torch.arange(height) + 0.5) / height * 2.0 - 1.0
    x = (torch.arange(width) + 0.5) / width * 2.0 - 1.0
    inside = ((x[None, :] / 0.65) ** 2 + (y[:, None] / 0.85) ** 2 < 1.0).float()
    img = (0.05 + 0.5 * _field(g, 3, height, width, 9)) * inside
    return (img.permute(1, 2, 0) + 0.01 * torch.randn(height, width, 3, generator=g)).contiguous()


def _params(scene, seed):
    """Ground-truth-like parameters (synth.random_params' distributions, textures made on a coarse grid)."""
    rng = np.random.default_rng(seed + 7)
    g = torch.Generator().manual_seed(seed + 11)
    m = scene.tex_size
    coef = np.concatenate([rng.normal(size=scene.n_shape), rng.uniform(0.0, 0.5, size=scene.n_expr)])
    p = synth.Params(coef=np.float32(coef), rot=np.float32(rng.uniform(-0.04, 0.04, 3)),
                     trans=np.float32(np.array([0.0, 0.0, 4.5]) + rng.normal(0.0, 0.03, 3)),
                     focal=np.float32([scene.focal_px()]),
                     light_i=np.float32(rng.uniform(0.2, 1.5, (scene.n_lights, 3))),
                     diffuse=(0.2 + 0.6 * _field(g, 3, m, m, 16)).permute(1, 2, 0).contiguous().numpy(),
                     specular=np.full((m, m, 3), 0.05, np.float32),
                     roughness=(0.3 + 0.3 * torch.rand(m, m, generator=g)).numpy(),
                     env=synth.env_map(rng, scene.env_size) if scene.env_size else None)
    return synth.with_stage_geometry(scene, p, seed) if scene.stage is not None else p


def _step_context(case):
    return (case["mesh"], case["width"], case["height"], case["spp"], case["tex"], case.get("lights", 0),
            case.get("stage", ""), case.get("env", 0), case.get("block", 0))


def _albedo_inputs(case, seed):
    """Coefficients and texture gradients of the batch's faces (CPU)."""
    g = torch.Generator().manual_seed(seed)
    n, k, m = case["faces"], case["columns"], case["tex"]
    coef = torch.randn(2, n, k, generator=g)
    grad = torch.zeros(2, n, m, m, 3)
    if case["kind"] != "albedo":
        small = torch.randn(2 * n, 3, 32, 32, generator=g) * 1e-2
        grad = torch.nn.functional.interpolate(small, size=(m, m), mode="bilinear").permute(0, 2, 3, 1)
        grad = grad.reshape(2, n, m, m, 3).contiguous()
    return coef, grad


def _adam_inputs(case, seed):
    """Stage II textures, their references, gradients and moments part way through the stage (CPU)."""
    g = torch.Generator().manual_seed(seed)
    m = case["tex"]
    out = {}
    for name, c in (("diffuse", 3), ("specular", 3), ("roughness", 1)):
        shape = (m, m, c) if c > 1 else (m, m)
        ref = (0.2 + 0.6 * _field(g, c, m, m, 16)).permute(1, 2, 0).reshape(shape).contiguous()
        out[name] = dict(ref=ref, x=ref + 0.02 * torch.randn(shape, generator=g),
                         g=0.02 * torch.randn(shape, generator=g), m=0.01 * torch.randn(shape, generator=g),
                         v=1e-4 * torch.rand(shape, generator=g))
    return out


ADAM_STEP = 40


def prepare(case, seed):
    kind = case["kind"]
    g = torch.Generator().manual_seed(seed)
    st = dict(kind=kind)
    if kind in ("step", "forward", "autograd"):
        r = _renderer(*_step_context(case), 0, 1)
        p = r.device_params(_params(r.scene, seed))
        st.update(r=r, p=p, iteration=seed % 100)
        if kind == "step":
            st["target"] = _picture(g, case["height"], case["width"]).cuda()
        if kind == "autograd":
            st["adj"] = torch.sign(torch.randn(case["height"], case["width"], 3, generator=g)).cuda()
            for t in p.values():
                t.requires_grad_(True)
    elif kind == "batch":
        n, top = case["faces"], case["largest"]
        r = _renderer(case["mesh"], top, top, case["spp"], case["tex"], case["lights"], "", 0, 0,
                      facert.FLAG_MORPH_BF16, n)
        rng = np.random.default_rng(seed)
        items = []
        for k in range(n):
            # sizes and sample counts of the mix follow the face, not the seed, so the work is fixed
            w, spp = (top, max(64, top // 2), max(64, 3 * top // 4 + 1), max(64, top // 3))[k % 4], case["spp"] >> (k % 3)
            sc = dataclasses.replace(r.scene, width=w, height=w)
            p = r.device_params(_params(sc, 97 * seed + k))
            items.append(dict(width=w, height=w, spp=spp, edge_spp=1,
                              flags=optim.STAGE2_FLAGS if k % 2 else 0, iteration=int(rng.integers(100)), face_id=k,
                              params=p, target=_picture(g, w, w).cuda(),
                              image=torch.zeros(w, w, 3, device="cuda"),
                              loss=torch.zeros(1, dtype=torch.float64, device="cuda"), grads=r.zero_grads(p)))
        st.update(r=r, items=items)
    elif kind in ("albedo", "albedo_adjoint", "albedo_both"):
        n = case["faces"]
        st["r"] = _albedo_renderer(case["tex"], case["columns"], bool(case.get("bf16", False)), n)
        coef, grad = _albedo_inputs(case, seed)
        st["coef"] = [list(coef[q].cuda()) for q in range(2)]
        st["grad"] = [list(grad[q].cuda()) for q in range(2)]
        st["tex"] = [[torch.empty(case["tex"], case["tex"], 3, device="cuda") for _ in range(n)] for _ in range(2)]
        st["g_coef"] = [torch.zeros(n, case["columns"], device="cuda") for _ in range(2)]
    elif kind == "adam":
        st["t"] = {n: {q: x.cuda() for q, x in d.items()} for n, d in _adam_inputs(case, seed).items()}
        st["reg"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    else:
        r = _renderer("c1", case["width"], case["height"], 1, 4, 8, "", 0, 0, 0, 1)
        st.update(r=r, target=_picture(g, case["height"], case["width"]).cuda(),
                  image=_picture(g, case["height"], case["width"]).cuda())
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(state):
    kind, r = state["kind"], state.get("r")
    if kind == "step":
        image, loss, grads = r.render(state["p"], state["target"], state["iteration"])
        return dict(image=image, loss=loss, grads=dict(grads))
    if kind == "forward":
        return dict(image=r.forward(state["p"], state["iteration"]))
    if kind == "autograd":
        image = autograd.render(r, state["p"], state["iteration"])
        names = list(state["p"])
        grads = torch.autograd.grad(image, [state["p"][n] for n in names], state["adj"])
        return dict(image=image.detach(), grads=dict(zip(names, grads)))
    if kind == "batch":
        for it in state["items"]:
            it["grads"].zero_()
        facert.fr_render_batch(r.ctx, state["items"])
        # every gradient of a face is a view of its one flat buffer
        return [dict(image=it["image"], loss=it["loss"], grads=it["grads"].flat) for it in state["items"]]
    if kind in ("albedo", "albedo_adjoint", "albedo_both"):
        out = {}
        if kind != "albedo_adjoint":
            facert.fr_albedo_morph(r.ctx, *state["coef"], *state["tex"])
            out.update(diffuse=state["tex"][0], specular=state["tex"][1])
        if kind != "albedo":
            for t in state["g_coef"]:
                t.zero_()
            facert.fr_albedo_adjoint(r.ctx, *state["grad"], list(state["g_coef"][0]), list(state["g_coef"][1]))
            out.update(g_beta=state["g_coef"][0], g_gamma=state["g_coef"][1])
        return out
    if kind == "adam":
        W, lr = optim.W, optim.LR["texture"]
        rgb = dict(kind=facert.GROUP_TEX_RGB, lr=lr, w_sym=W["w2"], w_chroma=W["w3"], w_smooth=W["w4"])
        d, s, q = (state["t"][n] for n in ("diffuse", "specular", "roughness"))
        M = d["x"].shape[0]
        groups = [facert.opt_group(d["x"], d["m"], d["v"], d["g"], aux=d["ref"], width=M, step=ADAM_STEP, **rgb),
                  facert.opt_group(s["x"], s["m"], s["v"], s["g"], aux=s["ref"], width=M, step=ADAM_STEP,
                                   w_box=W["box"], **rgb),
                  facert.opt_group(q["x"], q["m"], q["v"], q["g"], kind=facert.GROUP_TEX_MONO, width=M, lr=lr,
                                   w_smooth=W["w4"], w_box=W["box"], clamp=(0.02, 1.5), step=ADAM_STEP)]
        facert.fr_adam(groups, reg_energy=state["reg"])
        return dict({n: {k: t[k] for k in ("x", "m", "v")} for n, t in state["t"].items()}, reg=state["reg"])
    loss, adj, blurred = r.loss(state["image"], state["target"])
    return dict(loss=loss, adj=adj, blurred=blurred)


# --------------------------------------------------------------------------
# the work a pass cannot do without
# --------------------------------------------------------------------------
MESHES = {"c1": (2562, 5120, 20), "c2": (35709, 70789, 144), "c5": (50002, 100000, 20)}
FACE_SHARE = 0.42       # of the camera samples hit the face in every one of these scenes
FACING = 0.45           # of the lights are in front of a shading point


def _render_work(mesh, px, spp, lights, tex, grads, basis_bytes=4):
    """Inputs read and outputs written once; 300 flops per traced ray (one root-to-leaf path of a
    balanced tree and a triangle test) and 100 per shaded light, twice that for its reverse."""
    n, t, k = MESHES[mesh]
    model = 3 * n * (k + 1) * basis_bytes + 12 * t + 8 * n
    params = 4 * (7 * tex * tex + 3 * lights + k)
    hits = FACE_SHARE * px * spp
    rays = px * spp + FACING * lights * hits
    bytes_, flops = model + params + 12 * px, 2 * 3 * n * k + 300 * rays + 100 * FACING * lights * hits
    if grads:
        bytes_ += 12 * px + params + 4 * 3 * n * k
        flops += 2 * 3 * n * k + 200 * FACING * lights * hits + 2 * px * 300 * (1 + FACING * lights)
    return bytes_, flops


def work(case):
    kind = case["kind"]
    if kind in ("step", "forward", "autograd"):
        px = case["width"] * case["height"]
        lights = case.get("lights", 0) or (case["env"] // case["block"]) ** 2
        b, f = _render_work(case["mesh"], px, case["spp"], lights, case["tex"], kind != "forward")
    elif kind == "batch":
        n, top = case["faces"], case["largest"]
        nv, _, k = MESHES[case["mesh"]]
        b = f = 0
        for i in range(n):
            w, spp = (top, max(64, top // 2), max(64, 3 * top // 4 + 1), max(64, top // 3))[i % 4], case["spp"] >> (i % 3)
            bi, fi = _render_work(case["mesh"], w * w, spp, case["lights"], case["tex"], True)
            b, f = b + bi, f + fi
        b -= 2 * 4 * 3 * nv * k * (n - 1)            # the basis and its transpose's are read once for the batch
    elif kind in ("albedo", "albedo_adjoint", "albedo_both"):
        rows, k, n = 3 * case["tex"] ** 2, case["columns"], case["faces"]
        morph = 2 * (rows * k * (2 if case.get("bf16") else 4) + 4 * rows * (n + 1))
        adj = 2 * (4 * rows * k + 4 * rows * n)
        b = (morph if kind != "albedo_adjoint" else 0) + (adj if kind != "albedo" else 0)
        f = 2 * 2 * rows * k * n * (2 if kind == "albedo_both" else 1)
    elif kind == "adam":
        m2 = case["tex"] ** 2
        b, f = 4 * (7 * 7 + 6) * m2, 60 * 7 * m2      # x, m, v read and written, g read; two references
    else:
        px3 = 3 * case["width"] * case["height"]
        b, f = 4 * 4 * px3, 60 * px3                  # image, target in; adjoint, blurred out
    return {"bytes": float(b), "flops": float(f)}


# --------------------------------------------------------------------------
# the same outputs in 64 bits
# --------------------------------------------------------------------------
EXACT_TESTS = 6e9       # ray-triangle tests a brute-force 64-bit render may take


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "forward"):
        return _exact_render(case, seed)
    if kind in ("albedo", "albedo_adjoint", "albedo_both"):
        return _exact_albedo(case, seed)
    if kind == "adam":
        return _exact_adam(case, seed)
    if kind == "loss":
        g = torch.Generator().manual_seed(seed)
        target, image = (_picture(g, case["height"], case["width"]).double() for _ in range(2))
        loss, adj, blurred = _loss64(image, target)
        return dict(loss=loss.reshape(1), adj=adj, blurred=blurred)
    return None


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _loss64(image, target):
    """Sum |G * image - target| (3 x 3 Gaussian of sigma 1, replicated border), its gradient and the blurred image."""
    image = image.detach().requires_grad_(True)
    w = torch.exp(-0.5 * torch.tensor([1.0, 0.0, 1.0], dtype=torch.float64, device=image.device))
    w = torch.outer(w, w)
    w = (w / w.sum()).expand(3, 1, 3, 3)
    pad = torch.nn.functional.pad(image.permute(2, 0, 1)[None], (1, 1, 1, 1), mode="replicate")
    blurred = torch.nn.functional.conv2d(pad, w, groups=3)[0].permute(1, 2, 0)
    loss = (blurred - target).abs().sum()
    adj, = torch.autograd.grad(loss, image)
    return loss.detach(), adj, blurred.detach()


def _exact_albedo(case, seed):
    am, dev = _albedo_model(case["tex"], case["columns"]), _device()
    coef, grad = _albedo_inputs(case, seed)
    tex, g_coef = [], []
    for q, (mean, basis) in enumerate(((am.mean_diffuse, am.basis_diffuse), (am.mean_specular, am.basis_specular))):
        b = torch.as_tensor(basis, device=dev).reshape(case["columns"], -1)
        y = torch.as_tensor(mean, device=dev).double().reshape(1, -1).repeat(case["faces"], 1)
        gc = torch.zeros(case["faces"], case["columns"], dtype=torch.float64, device=dev)
        c, gr = coef[q].to(dev).double(), grad[q].to(dev).double().reshape(case["faces"], -1)
        for k in range(case["columns"]):
            row = b[k].double()
            y += c[:, k:k + 1] * row
            gc[:, k] = gr @ row
        tex.append([x.reshape(case["tex"], case["tex"], 3) for x in y])
        g_coef.append(gc)
    out = {}
    if case["kind"] != "albedo_adjoint":
        out.update(diffuse=tex[0], specular=tex[1])
    if case["kind"] != "albedo":
        out.update(g_beta=g_coef[0], g_gamma=g_coef[1])
    return out


def _exact_adam(case, seed):
    """Adam on E_ph + symmetry + chromaticity + smoothness + box terms of the textures."""
    W = dict(sym=0.3, chroma=0.3, smooth=0.0002, box=1.0)
    out, reg = {}, 0.0
    for name, d in _adam_inputs(case, seed).items():
        ref, x, g, m, v = (d[q].double() for q in ("ref", "x", "g", "m", "v"))
        X = x.reshape(x.shape[0], x.shape[1], -1).clone().requires_grad_(True)
        e = 2.0 * W["smooth"] * (((X[:, 1:] - X[:, :-1]) ** 2).sum() + ((X[1:] - X[:-1]) ** 2).sum())
        if name != "roughness":
            R = ref.reshape(X.shape)
            e = e + W["sym"] * (X - X.flip(1)).abs().sum()
            e = e + W["chroma"] * (X / (X.sum(-1, True) + 1e-6) - R / (R.sum(-1, True) + 1e-6)).abs().sum()
        if name != "diffuse":
            e = e + W["box"] * (X.clamp(max=0.0) ** 2 + (X - 1.0).clamp(min=0.0) ** 2).sum()
        ge, = torch.autograd.grad(e, X)
        g = g + ge.reshape(x.shape)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        x = x - 5e-3 * (m / (1.0 - 0.9 ** ADAM_STEP)) / ((v / (1.0 - 0.999 ** ADAM_STEP)).sqrt() + 1e-8)
        if name == "roughness":
            x = x.clamp(0.02, 1.5)
        out[name], reg = dict(x=x, m=m, v=v), reg + float(e.detach())
    return dict(out, reg=torch.tensor([reg], dtype=torch.float64))


def _philox(key, counter):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    k0, k1 = key
    c = [x.clone() for x in counter]
    for r in range(10):
        a, b = _mul32(0xD2511F53, c[0]), _mul32(0xCD9E8D57, c[2])
        c = [b[0] ^ c[1] ^ k0, b[1], a[0] ^ c[3] ^ k1, a[1]]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _mul32(m, x):
    """High and low 32 bits of m * x without overflowing 63 bits."""
    lo, hi = m * (x & 0xFFFF), m * (x >> 16)
    t = lo + ((hi & 0xFFFF) << 16)
    return (hi >> 16) + (t >> 32), t & 0xFFFFFFFF


def _first_hit(org, d, tri, skip=None, bounded=False):
    """Brute force (Moller-Trumbore): index of the nearest triangle hit (-1: none) and its (t, b1, b2);
    bounded: whether any triangle but `skip` is hit with 1e-4 < t < 1 - 1e-4."""
    if org.shape[0] == 0:
        return torch.zeros(0, dtype=torch.bool if bounded else torch.long, device=org.device)
    e1, e2, v0 = tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0], tri[:, 0]
    step = max(1, int(4e7) // tri.shape[0])
    best, val = [], []
    for i in range(0, org.shape[0], step):
        o, r = org[i:i + step, None], d[i:i + step, None]
        p = torch.linalg.cross(r, e2[None])
        det = (p * e1).sum(-1)
        s = o - v0
        b1 = (s * p).sum(-1) / det
        q = torch.linalg.cross(s, e1[None].expand_as(s))
        b2, t = (q * r).sum(-1) / det, (q * e2).sum(-1) / det
        ok = (det != 0) & (b1 >= 0) & (b2 >= 0) & (b1 + b2 <= 1)
        if bounded:
            ok &= (t > 1e-4) & (t < 1.0 - 1e-4)
            ok[torch.arange(o.shape[0]), skip[i:i + step]] = False
            best.append(ok.any(1))
            continue
        t = torch.where(ok & (t > 0), t, torch.inf)
        tm, k = t.min(1)
        best.append(torch.where(tm < torch.inf, k, -1))
        val.append(torch.stack([tm, b1.gather(1, k[:, None])[:, 0], b2.gather(1, k[:, None])[:, 0]], 1))
    return torch.cat(best) if bounded else (torch.cat(best), torch.cat(val))


def _g1(nv, r):
    s2 = (1.0 - nv * nv).clamp(min=1e-300)
    a = nv / (r * s2.sqrt())
    g = (3.535 * a + 2.181 * a * a) / (1.0 + 2.276 * a + 2.577 * a * a)
    return torch.where(a >= 1.6, torch.ones_like(a), g)


def _exact_render(case, seed):
    """Image, and for a step the loss and the gradients that no boundary term reaches (light intensities,
    textures), by brute force in 64 bits.  Area lights given by records only."""
    W, H, spp, NL, M = case["width"], case["height"], case["spp"], case["lights"], case["tex"]
    tests = W * H * spp * MESHES[case["mesh"]][1] * (1.0 + FACE_SHARE * FACING * NL)
    if case.get("stage") or tests > EXACT_TESTS:
        return None
    sc = _scene(case["mesh"], W, H, spp, M, NL)
    P = _params(sc, seed)
    dev = _device()

    def f64(x):
        return torch.as_tensor(np.asarray(x, np.float64), device=dev)

    # geometry: morph, pose, normals
    v = f64(sc.mean) + torch.tensordot(f64(P.coef), f64(sc.basis), 1)
    (sx, sy, sz), (cx, cy, cz) = (f(f64(P.rot)).tolist() for f in (torch.sin, torch.cos))
    Rx = f64([[1, 0, 0], [0, cx, -sx], [0, sx, cx]])
    Ry = f64([[cy, 0, sy], [0, 1, 0], [-sy, 0, cy]])
    Rz = f64([[cz, -sz, 0], [sz, cz, 0], [0, 0, 1]])
    v = (v - f64(P.trans)) @ (Rz @ Ry @ Rx)
    faces = torch.as_tensor(sc.faces, device=dev).long()
    tri = v[faces]
    nf = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    vn = torch.zeros_like(v)
    for k in range(3):
        vn.index_add_(0, faces[:, k], nf)
    vn = vn / vn.norm(dim=1, keepdim=True).clamp(min=1e-300)
    # camera samples
    n = W * H * spp
    q = torch.arange(n, device=dev)
    pixel, sample = q // spp, q % spp
    z = torch.zeros_like(pixel)

    def dims(d):
        w = _philox((0, 0), [pixel, (sample << 16) | (d >> 2), z + seed % 100, z])
        u = [((x >> 8).double() / 16777216.0) for x in w]
        return (u[2], u[3]) if d & 2 else (u[0], u[1])

    jx, jy = dims(0)
    f = float(P.focal[0])
    d = torch.stack([(pixel % W + jx - 0.5 * W) / f, -(pixel // W + jy - 0.5 * H) / f, torch.full_like(jx, -1.0)], 1)
    hit, tb = _first_hit(torch.zeros_like(d), d, tri)
    on = (hit >= 0).nonzero()[:, 0]
    h, b = hit[on], torch.stack([1.0 - tb[on, 1] - tb[on, 2], tb[on, 1], tb[on, 2]], 1)
    y = (tri[h] * b[..., None]).sum(1)
    ns = (vn[faces[h]] * b[..., None]).sum(1)
    ns = ns / ns.norm(dim=1, keepdim=True)
    o = -d[on] / d[on].norm(dim=1, keepdim=True)
    lit = (nf[h] * o).sum(1) > 0
    uv = (f64(sc.uv)[faces[h]] * b[..., None]).sum(1)
    # bilinear material, texel centres at u M - 1/2, clamp to edge
    leaf = {k: f64(getattr(P, k)).requires_grad_(True) for k in ("diffuse", "specular", "roughness", "light_i")}
    xy = uv * M - 0.5
    i0, fr = xy.floor().long(), xy - xy.floor()
    x0, x1 = i0[:, 0].clamp(0, M - 1), (i0[:, 0] + 1).clamp(0, M - 1)
    y0, y1 = i0[:, 1].clamp(0, M - 1), (i0[:, 1] + 1).clamp(0, M - 1)

    def texel(t):
        t = t.reshape(M, M, -1)
        fx, fy = fr[:, :1], fr[:, 1:]
        return (1 - fy) * ((1 - fx) * t[y0, x0] + fx * t[y0, x1]) + fy * ((1 - fx) * t[y1, x0] + fx * t[y1, x1])

    c, s, r = texel(leaf["diffuse"]), texel(leaf["specular"]), texel(leaf["roughness"])
    Lo = torch.zeros(on.shape[0], 3, dtype=torch.float64, device=dev)
    no = (ns * o).sum(1, keepdim=True)
    for j in range(NL):
        rec = f64(sc.lights[j])
        lc, e1, e2 = rec[1:4], rec[4:7], rec[7:10]
        nl_ = torch.linalg.cross(e1, e2)
        area, nl_ = nl_.norm(), nl_ / nl_.norm()
        u0, u1 = (x[on, None] for x in dims(2 + 2 * j))
        p = lc + e1 * (u0 - 0.5) + e2 * (u1 - 0.5)
        lv = p - y
        d2 = (lv * lv).sum(1, keepdim=True)
        l = lv / d2.sqrt()
        cs, cl = (ns * l).sum(1, keepdim=True), -(l @ nl_)[:, None]
        need = ((cs > 0) & (cl > 0))[:, 0] & lit
        idx = need.nonzero()[:, 0]
        idx = idx[~_first_hit(y[idx], lv[idx], tri, h[idx], bounded=True)]
        if idx.numel() == 0:
            continue
        l, cs, cl, d2, ok = l[idx], cs[idx], cl[idx], d2[idx], no[idx] > 0
        hv = l + o[idx]
        hv = hv / hv.norm(dim=1, keepdim=True)
        nh, oh = (ns[idx] * hv).sum(1, keepdim=True), (o[idx] * hv).sum(1, keepdim=True)
        rr, nv = r[idx], no[idx].clamp(min=1e-12)
        D = nh.clamp(min=1e-300) ** (2.0 / rr - 2.0) / (math.pi * rr)
        F = s[idx] + (1.0 - s[idx]) * (1.0 - oh) ** 5
        spec = torch.where(ok, D * _g1(nv, rr) * _g1(cs, rr) / (4.0 * nv * cs), torch.zeros_like(cs)) * F
        scale = float(sc.light_d[j]) ** 2 / float(sc.light_a[j]) * area
        Lo = Lo.index_add(0, idx, (c[idx] / math.pi + spec) * (cs * cl / d2) * leaf["light_i"][j] * scale)
    image = torch.zeros(W * H, 3, dtype=torch.float64, device=dev).index_add(0, pixel[on], Lo / spp).reshape(H, W, 3)
    if case["kind"] == "forward":
        return dict(image=image.detach())
    target = _picture(torch.Generator().manual_seed(seed), H, W).double().to(dev)
    loss, adj, _ = _loss64(image, target)
    got = dict(zip(leaf, torch.autograd.grad(image, list(leaf.values()), adj)))
    return dict(image=image.detach(), loss=loss.reshape(1), grads={k: got.get(k) for k in facert.PARAM_NAMES})
