"""Performance cases: the work that programs built on this library have it do,
through its public entry points, over the sizes they use.

A case is a dict of plain values.  ``prepare`` makes its inputs on the GPU
from a seed, with the buffers and workspaces that a program keeps between
calls; ``run`` is one pass; ``work`` states what one pass cannot do without;
``exact`` gives the same outputs from plain torch arithmetic in 64 bits.

The kinds of work:

* ``forward``   acoustic or elastic modelling of a survey (``sweep_forward``)
* ``gradient``  FWI gradient and misfit (``sweep_gradient``), with or without
                the illumination, by a direct call or a recorded graph
* ``autograd``  modelling and ``backward()`` through ``acoustic_modelling``,
                which also runs ``sweep_adjoint`` for the wavelets
* ``batch``     gradients of many models of uneven size (``batch.run``)
* ``train``     one training step of the learned preconditioner
* ``infer``     the preconditioner applied to gradients
* ``layer``     one 3 x 3 convolution layer forward and backward
"""
import math
import random

import torch
import torch.nn.functional as F

from paper_2604_14189_gb300 import autograd, batch, sweep, unet

V_MAX = 4500.0    # acoustic models lie in [1500, 4500] m/s; also the CPML reference velocity
VP_MAX = 5000.0   # elastic models: Vp in [1800, 5000] m/s
DT_AC, DX_AC, F_AC = 1e-3, 10.0, 10.0
DT_EL, DX_EL, F_EL = 5e-4, 5.0, 15.0

# channels of the preconditioner's 17 convolutions, in parameter order
UNET_LAYERS = [(32, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 256),
               (256, 256), (256, 128), (256, 128), (128, 128), (128, 64), (128, 64), (64, 64),
               (64, 32), (64, 32), (32, 32)]


def _survey(kind, name=None, physics="acoustic", nz=0, nx=0, pml=40, nt=0, shots=1, rec_step=1,
            illum=False, graph=False, deterministic=False):
    case = dict(kind=kind, physics=physics, nz=nz, nx=nx, pml=pml, nt=nt, shots=shots,
                rec_step=rec_step, illum=illum, graph=graph, deterministic=deterministic)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest modelling job: one shot over a three-layer-sized grid;
        # its steps are too small to fill the GPU, so latency counts
        _survey("forward", "forward_one_shot", nz=200, nx=200, nt=1000),
        # modelling a whole survey, as a line-search trial or to make data
        _survey("forward", "forward_survey", nz=301, nx=901, nt=1000, shots=20, rec_step=3),
        # a small inversion's gradient on an odd grid
        _survey("gradient", "gradient_small", nz=141, nx=187, pml=23, nt=900, shots=3),
        # one FWI iteration's gradient with illumination, replayed as the FWI loop does
        _survey("gradient", "gradient_fwi", nz=256, nx=256, nt=1500, shots=16, illum=True,
                graph=True),
        # the survey-sized gradient, the largest acoustic call
        _survey("gradient", "gradient_survey", nz=301, nx=901, nt=3000, shots=20, rec_step=3),
        # differentiable modelling inside a torch program, odd grid
        _survey("autograd", "autograd_step", nz=173, nx=305, pml=30, nt=1000, shots=4, rec_step=2),
        # elastic modelling of a 64-shot survey (records cut)
        _survey("forward", "elastic_forward", physics="elastic", nz=500, nx=1500, nt=250, shots=64,
                rec_step=2),
        # elastic gradient (vp, vs, rho) of 8 shots (records cut)
        _survey("gradient", "elastic_gradient", physics="elastic", nz=500, nx=1500, nt=500,
                shots=8, rec_step=2),
        # many models of uneven size, border, record length and shot count
        dict(name="batch_models", kind="batch", count=24, lo=128, hi=512, nt_lo=800, nt_hi=3000,
             pick=1003),
        # one training step of the preconditioner: batch of 8 gradients
        dict(name="train_step", kind="train", batch=8, height=256, width=256, channels=2),
        # the trained preconditioner inside the FWI loop: one gradient
        dict(name="infer_one", kind="infer", batch=1, height=256, width=256, channels=2),
        # a decoder layer on its own: forward, data gradient, weight gradient
        dict(name="conv_layer", kind="layer", batch=8, height=64, width=64, cin=256, cout=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "gradient", "gradient", "gradient", "autograd",
                       "elastic", "elastic", "batch", "train", "infer", "layer"])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 24), lo=rng.randint(96, 160),
                    hi=rng.randint(256, 512), nt_lo=800, nt_hi=rng.randint(1000, 2500),
                    pick=rng.randint(1, 10 ** 6))
    if kind in ("train", "infer"):
        return dict(kind=kind, batch=rng.randint(1, 8), height=128 * rng.randint(1, 2),
                    width=rng.choice([128, 256]), channels=rng.randint(1, 4))
    if kind == "layer":
        w = rng.choice([16, 32, 64, 128, 256])
        step = max(1, 128 // w)  # rows per 128-pixel tile
        h = step * max(1, _log(rng, 16, 256) // step)
        return dict(kind="layer", batch=rng.randint(1, 8), height=h, width=w,
                    cin=rng.choice([32, 64, 128, 192, 256]),
                    cout=rng.choice([32, 64, 128, 192, 256]))
    if kind == "elastic":
        mode = rng.choice(["forward", "gradient"])
        nz, nx, shots = _log(rng, 60, 500), _log(rng, 80, 1500), _log(rng, 1, 8)
        pml, nt = rng.randint(10, 40), _log(rng, 150, 1000)
        cells = (nz + 2 * pml) * (nx + 2 * pml) * shots
        nt = max(50, min(nt, int(2.5e9 / cells)))
        return _survey(mode, physics="elastic", nz=nz, nx=nx, pml=pml, nt=nt, shots=shots,
                       rec_step=rng.randint(1, 3))
    nz, nx, shots = _log(rng, 64, 512), _log(rng, 64, 1024), _log(rng, 1, 24)
    pml, nt = rng.randint(16, 40), _log(rng, 300, 3000)
    cells = (nz + 2 * pml) * (nx + 2 * pml) * shots
    nt = max(100, min(nt, int(8e9 / cells)))
    opt = rng.random()
    return _survey(kind, nz=nz, nx=nx, pml=pml, nt=nt, shots=shots, rec_step=rng.randint(1, 4),
                   illum=kind == "gradient" and opt < 0.3,
                   deterministic=kind != "autograd" and 0.3 <= opt < 0.45)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _layered(g, nz, nx, vmin, vmax):
    """Velocity rising with depth, undulating interfaces and smooth anomalies."""
    z = torch.arange(nz, device="cuda", dtype=torch.float64)[:, None]
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
    v = (vmin + (vmax - vmin) * z / max(nz - 1, 1)).expand(nz, nx)
    for depth, jump, k, ph in _uniform(g, (8, 4), 0.0, 1.0).tolist():
        surf = (0.1 + 0.8 * depth) * nz + 5.0 * torch.sin((1 + 2 * k) * 2 * math.pi * x / nx + 6 * ph)
        v = v + (300.0 * jump - 150.0) * (z >= surf)
    for cz, cx, amp in _uniform(g, (5, 3), 0.0, 1.0).tolist():
        r2 = (z - (0.2 + 0.6 * cz) * nz) ** 2 + (x - (0.2 + 0.6 * cx) * nx) ** 2
        v = v * (1.0 + (0.2 * amp - 0.1) * torch.exp(-r2 / 450.0))
    return v.clamp(vmin, vmax)


def _ricker(t, f0):
    a = (math.pi * f0 * t) ** 2
    return (1.0 - 2.0 * a) * torch.exp(-a)


def _wavelets(g, shots, nt, dt, f0):
    """Ricker wavelets whose strength varies a little from shot to shot."""
    t = torch.arange(nt, device="cuda", dtype=torch.float64) * dt - 1.5 / f0
    amp = _uniform(g, (shots, 1), 0.8, 1.2)
    return (amp * _ricker(t, f0)[None]).to(torch.float32).contiguous()


def _acquisition(nx, shots, rec_step):
    """Sources evenly spaced at the surface, receivers every rec_step cells."""
    sx = torch.linspace(0, nx - 1, shots, device="cuda").round().to(torch.int32)
    src = torch.stack([torch.full_like(sx, 2), sx], dim=-1).contiguous()
    rx = torch.arange(0, nx, rec_step, device="cuda", dtype=torch.int32)
    rec = torch.stack([torch.full_like(rx, 2), rx], dim=-1)
    return src, rec[None].expand(shots, -1, -1).contiguous()


def _records(g, src, rec, nt, dt, dx, f0, ncomp, level, vmin, vmax):
    """Observed data: a direct wave and reflections along their travel-time
    curves, falling off with time."""
    shots, nrec = rec.shape[:2]
    t = torch.arange(nt, device="cuda", dtype=torch.float32) * dt
    off = (rec[:, :, 1] - src[:, None, 1]).to(torch.float32) * dx
    d = torch.zeros(shots, ncomp, nrec, nt, device="cuda", dtype=torch.float32)
    for k, (a, b, c) in enumerate(_uniform(g, (4, 3), 0.0, 1.0).tolist()):
        t0 = 0.0 if k == 0 else (0.1 + 0.8 * a) * nt * dt
        v = vmin if k == 0 else vmin + (0.2 + 0.6 * b) * (vmax - vmin)
        amp = (1.0 if k == 0 else 0.6 * c - 0.3) * level
        tau = torch.sqrt(t0 * t0 + (off / v) ** 2)[:, :, None]
        wave = amp * _ricker(t - tau - 1.5 / f0, f0) / torch.sqrt(tau + 0.1)
        for comp in range(ncomp):
            d[:, comp] += wave if comp == 0 else 0.7 * wave
    return d


def _physical(case):
    if case["physics"] == "elastic":
        return sweep.ELASTIC, 2, DT_EL, DX_EL, F_EL
    return sweep.ACOUSTIC, 1, DT_AC, DX_AC, F_AC


def _survey_inputs(case, seed):
    g = _gen(seed)
    _, ncomp, dt, dx, f0 = _physical(case)
    nz, nx = case["nz"], case["nx"]
    if case["physics"] == "elastic":
        vp = _layered(g, nz, nx, 1800.0, VP_MAX)
        model = torch.stack([vp, vp / 1.73, 310.0 * vp ** 0.25])
        vmin, vmax, level = 1800.0, VP_MAX, 1e-7
    else:
        model = _layered(g, nz, nx, 1500.0, V_MAX)
        vmin, vmax, level = 1500.0, V_MAX, 0.03
    src, rec = _acquisition(nx, case["shots"], case["rec_step"])
    wav = _wavelets(g, case["shots"], case["nt"], dt, f0)
    d_obs = None
    if case["kind"] != "forward":
        d_obs = _records(g, src, rec, case["nt"], dt, dx, f0, ncomp, level, vmin, vmax)
    return dict(model=model.to(torch.float32).contiguous(), wav=wav, src=src, rec=rec, d_obs=d_obs)


def _problem(case, nrec):
    physics, _, dt, dx, f0 = _physical(case)
    return sweep.problem(physics, nz=case["nz"], nx=case["nx"], pml=case["pml"], dx=dx, dt=dt,
                         nt=case["nt"], nshot=case["shots"], nrec=nrec, f_ref=f0,
                         v_pml=VP_MAX if physics == sweep.ELASTIC else V_MAX,
                         flags=sweep.F_DETERMINISTIC if case["deterministic"] else 0)


def _batch_cases(case):
    """The batch's problems: sizes from `pick` alone."""
    r = random.Random(case["pick"])
    return [dict(kind="gradient", physics="acoustic", nz=r.randint(case["lo"], case["hi"]),
                 nx=r.randint(case["lo"], case["hi"]), pml=r.randint(20, 40),
                 nt=r.randint(case["nt_lo"], case["nt_hi"]), shots=r.randint(1, 8), rec_step=1,
                 illum=False, graph=False, deterministic=False) for _ in range(case["count"])]


def _unet_theta(g):
    """He-normal weights and small biases, as a network in training has."""
    parts = []
    for ci, co in UNET_LAYERS:
        parts.append(torch.randn(co * 9 * ci, generator=g, device="cuda") * math.sqrt(2 / (9 * ci)))
        parts.append(torch.randn(co, generator=g, device="cuda") * 0.01)
    parts.append(torch.randn(32, generator=g, device="cuda") * math.sqrt(1 / 32))
    parts.append(torch.zeros(1, device="cuda"))
    return torch.cat(parts)


def _images(g, n, h, w, c):
    """Smooth images with max |value| 1, like normalised FWI gradients."""
    x = torch.randn(n, c, h // 8, w // 8, generator=g, device="cuda")
    x = F.interpolate(x, size=(h, w), mode="bilinear", align_corners=False)
    x = x + 0.1 * torch.randn(n, c, h, w, generator=g, device="cuda")
    return (x / x.abs().amax(dim=(2, 3), keepdim=True)).permute(0, 2, 3, 1).contiguous()


def _unet_inputs(case, seed):
    g = _gen(seed)
    b, h, w, c = case["batch"], case["height"], case["width"], case["channels"]
    s = dict(theta=_unet_theta(g), x=_images(g, b, h, w, c))
    s["target"] = _images(g, b, h, w, 1)[..., 0].contiguous()
    s["m"] = 1e-4 * torch.randn(unet.PARAMS, generator=g, device="cuda")
    s["v"] = 1e-7 * (0.1 + torch.rand(unet.PARAMS, generator=g, device="cuda"))
    return s


def _layer_inputs(case, seed):
    g = _gen(seed)
    b, h, w, ci, co = (case[k] for k in ("batch", "height", "width", "cin", "cout"))

    def normal(*shape, scale=1.0):
        return (scale * torch.randn(*shape, generator=g, device="cuda")).to(torch.bfloat16)

    wgt = normal(co, 9, ci, scale=math.sqrt(2 / (9 * ci)))
    return dict(x=normal(b, h, w, ci).relu(), w=wgt,
                wt=wgt.flip(1).permute(2, 1, 0).contiguous(),  # transposed, taps mirrored
                bias=0.1 * torch.randn(co, generator=g, device="cuda"),
                dy=normal(b, h, w, co, scale=0.1))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "layer":
        s = _layer_inputs(case, seed)
        s["out"] = torch.empty_like(s["dy"])
        s["dx"] = torch.empty_like(s["x"])
        s["dw"] = torch.empty(case["cout"], 9, case["cin"], device="cuda")
    elif kind in ("train", "infer"):
        s = _unet_inputs(case, seed)
        s["shape"] = unet.shape(case["batch"], case["height"], case["width"], case["channels"])
        s["ws"] = unet.alloc_workspace(s["shape"], kind == "train")
        s["out"] = torch.empty_like(s["target"])
        if kind == "train":
            s["grad"] = torch.empty_like(s["theta"])
            s["loss"] = torch.empty((), dtype=torch.float64, device="cuda")
            s["step"] = 1000
    elif kind == "batch":
        items = []
        for k, c in enumerate(_batch_cases(case)):
            i = _survey_inputs(c, seed * 100003 + k)
            items.append(batch.Item(_problem(c, i["rec"].shape[1]), i["model"], i["wav"],
                                    i["src"], i["rec"], i["d_obs"]))
        s = dict(items=items)
    else:
        s = _survey_inputs(case, seed)
        p = s["problem"] = _problem(case, s["rec"].shape[1])
        if kind == "autograd":
            s["model"].requires_grad_(True)
            s["wav"].requires_grad_(True)
        else:
            mode = sweep.MODE_GRADIENT if kind == "gradient" else sweep.MODE_FORWARD
            s["ws"] = sweep.alloc_workspace(p, mode)
            g_shape, d_shape = batch.out_shapes(p)
            if kind == "forward":
                s["data"] = torch.empty(d_shape, device="cuda")
            else:
                s["grad"] = torch.empty(g_shape, device="cuda")
                s["misfit"] = torch.empty((), dtype=torch.float64, device="cuda")
                s["illum"] = torch.empty(g_shape, device="cuda") if case["illum"] else None
                if case["graph"]:
                    side = torch.cuda.Stream()
                    with sweep.capture(side) as c:
                        sweep.sweep_gradient(p, s["model"], s["wav"], s["src"], s["rec"],
                                             s["d_obs"], grad=s["grad"], misfit=s["misfit"],
                                             illum=s["illum"], ws=s["ws"], stream=side)
                    s["graph"] = c.graph
    s["kind"] = kind
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "forward":
        return sweep.sweep_forward(s["problem"], s["model"], s["wav"], s["src"], s["rec"],
                                   data=s["data"], ws=s["ws"])
    if kind == "gradient":
        if "graph" in s:
            s["graph"].launch()
        else:
            sweep.sweep_gradient(s["problem"], s["model"], s["wav"], s["src"], s["rec"], s["d_obs"],
                                 grad=s["grad"], misfit=s["misfit"], illum=s["illum"], ws=s["ws"])
        return dict(grad=s["grad"], misfit=s["misfit"], illum=s["illum"])
    if kind == "autograd":
        data = autograd.acoustic_modelling(s["model"], s["wav"], s["problem"], s["src"], s["rec"])
        loss = 0.5 * ((data - s["d_obs"]) ** 2).sum()
        gv, gw = torch.autograd.grad(loss, (s["model"], s["wav"]))
        return dict(data=data.detach(), grad_v=gv, grad_w=gw)
    if kind == "batch":
        codes = batch.run(s["items"], streams=2)
        return dict(codes=codes, grads=[it.grad for it in s["items"]],
                    misfits=torch.stack([it.misfit for it in s["items"]]))
    if kind == "train":
        unet.gradient(s["shape"], s["theta"], s["x"], s["target"], grad=s["grad"], out=s["out"],
                      loss=s["loss"], ws=s["ws"], sync=False)
        s["step"] += 1
        unet.adam(s["theta"], s["grad"], s["m"], s["v"], s["step"], 5e-4)
        return dict(loss=s["loss"], out=s["out"], grad=s["grad"], theta=s["theta"], m=s["m"],
                    v=s["v"])
    if kind == "infer":
        return unet.forward(s["shape"], s["theta"], s["x"], out=s["out"], ws=s["ws"], sync=False)
    unet.conv3x3(s["x"], s["w"], s["bias"], unet.OP_RELU, out=s["out"])
    unet.conv3x3(s["dy"], s["wt"], None, unet.OP_MASK, mask=s["x"], out=s["dx"])
    unet.conv3x3_wgrad(s["x"], s["dy"], dw=s["dw"])
    return dict(out=s["out"], dx=s["dx"], dw=s["dw"])


# -------------------------------------------------------------------- work

def _step_bytes(case):
    """(forward, backward) bytes of one time step of all shots: a step reads
    and writes the wave state once (acoustic: u twice read, once written, K;
    the border's memory variables read and written); a backward step also
    reconstructs u on the interior and adds to the image."""
    P, nz, nx, S = case["pml"], case["nz"], case["nx"], case["shots"]
    NZ, NX = nz + 2 * P, nx + 2 * P
    n, strips = NZ * NX, 2 * P * (NZ + NX)
    if case["physics"] == "elastic":
        fwd = S * (40 * n + 32 * strips) + 20 * n
        return fwd, S * (60 * n + 32 * strips) + 40 * n
    fwd = S * (12 * n + 16 * strips) + 4 * n
    return fwd, fwd + S * (20 * nz * nx)


def _survey_work(case, passes):
    """passes: (forward, backward) time loops of one call."""
    P, nz, nx = case["pml"], case["nz"], case["nx"]
    n = (nz + 2 * P) * (nx + 2 * P)
    fwd, bwd = _step_bytes(case)
    el = case["physics"] == "elastic"
    nrec = -(-nx // case["rec_step"])
    records = 4 * case["shots"] * nrec * case["nt"] * (2 if el else 1)
    nb = passes[0] * fwd * case["nt"] + passes[1] * bwd * case["nt"] + sum(passes) * records
    per = (60, 120) if el else (30, 65)
    return nb, (passes[0] * per[0] + passes[1] * per[1]) * n * case["nt"] * case["shots"]


def _unet_flops(case):
    px = case["batch"] * case["height"] * case["width"]
    level = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 2, 1, 1, 1, 0, 0, 0]
    return [2 * 9 * ci * co * px // 4 ** lv for (ci, co), lv in zip(UNET_LAYERS, level)]


def work(case):
    kind = case["kind"]
    if kind == "layer":
        px = case["batch"] * case["height"] * case["width"]
        ci, co = case["cin"], case["cout"]
        # forward x -> out, data gradient dy, x (mask) -> dx, weight gradient x, dy -> dw
        return dict(bytes=2 * px * (4 * ci + 3 * co) + 9 * ci * co * 8, flops=3 * 18 * px * ci * co)
    if kind in ("train", "infer"):
        px = case["batch"] * case["height"] * case["width"]
        fl = _unet_flops(case)
        if kind == "infer":
            return dict(bytes=4 * px * (case["channels"] + 1) + 4 * unet.PARAMS, flops=sum(fl))
        return dict(bytes=4 * px * (case["channels"] + 2) + 4 * unet.PARAMS * 8,
                    flops=3 * sum(fl) - fl[0])
    if kind == "batch":
        both = [_survey_work(c, (1, 1)) for c in _batch_cases(case)]
        return dict(bytes=sum(b for b, _ in both), flops=sum(f for _, f in both))
    # autograd: forward for the data; forward + backward for v; backward for the wavelets
    passes = {"forward": (1, 0), "gradient": (1, 1), "autograd": (2, 2)}[kind]
    nb, fl = _survey_work(case, passes)
    return dict(bytes=nb, flops=fl)


# ------------------------------------------------- 64-bit values of the outputs

C2 = (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)
C1 = (0.0, 4 / 5, -1 / 5, 4 / 105, -1 / 280)
LIMIT_S = 18.0  # exact() gives None for a case that would take longer


def _f32(x):
    return float(torch.tensor(x, dtype=torch.float32))


def _shift(fp, h, ax, k, n):
    return fp.narrow(ax, h + k, n)


def _centred(f, ax):
    """(second, first) 8th-order derivatives along axis ax (1: z, 2: x)."""
    fp = F.pad(f, (4, 4) if ax == 2 else (0, 0, 4, 4))
    n = f.shape[ax]
    d2, d1 = C2[0] * f, None
    for k in range(1, 5):
        a, b = _shift(fp, 4, ax, k, n), _shift(fp, 4, ax, -k, n)
        d2 = d2.add(a, alpha=C2[k]).add(b, alpha=C2[k])
        d1 = C1[1] * a if d1 is None else d1.add(a, alpha=C1[k])
        d1 = d1.add(b, alpha=-C1[k])
    return d2, d1


def _staggered(f, ax, plus):
    """4th-order staggered difference along ax at +1/2 (plus) or -1/2."""
    fp = F.pad(f, (2, 2) if ax == 2 else (0, 0, 2, 2))
    n, o = f.shape[ax], 1 if plus else 0
    r = (9 / 8) * _shift(fp, 2, ax, o, n)
    r = r.add(_shift(fp, 2, ax, o - 1, n), alpha=-9 / 8)
    r = r.add(_shift(fp, 2, ax, o + 1, n), alpha=-1 / 24)
    return r.add(_shift(fp, 2, ax, o - 2, n), alpha=1 / 24)


def _profile(n, P, dx, dt, vref, f_ref, half=False):
    x = torch.arange(n + 2 * P, device="cuda", dtype=torch.float64) + (0.5 if half else 0.0)
    d = torch.maximum(P - x, x - (P + n - 1)).clamp(min=0.0)
    rho = (d / max(P, 1)).clamp(max=1.0)
    sigma = 3 * vref * math.log(1000.0) / (2 * max(P, 1) * dx) * rho ** 2
    alpha = math.pi * f_ref * (1 - rho)
    a = torch.exp(-(sigma + alpha) * dt)
    b = sigma / (sigma + alpha).clamp(min=1e-300) * (a - 1)
    on = d > 0
    return torch.where(on, a, 0 * a), torch.where(on, b, 0 * b), on.double()


class _Acoustic:
    def __init__(self, case, i):
        P, self.S, self.nt = case["pml"], case["shots"], case["nt"]
        dt, dx = _f32(DT_AC), _f32(DX_AC)
        v = F.pad(i["model"].double()[None, None], (P, P, P, P), mode="replicate")[0, 0]
        self.leaf, self.scale, self.P = v, (dt / dx) ** 2, P
        prof = [_profile(n, P, dx, dt, V_MAX, _f32(F_AC)) for n in (case["nz"], case["nx"])]
        self.az, self.bz, self.mz = (t[None, :, None] for t in prof[0])
        self.ax, self.bx, self.mx = (t[None, None, :] for t in prof[1])
        self._positions(i, P)
        self.w = i["wav"].detach().double()

    def _positions(self, i, P):
        self.sidx = torch.arange(self.S, device="cuda")
        self.src = (self.sidx, i["src"][:, 0].long() + P, i["src"][:, 1].long() + P)
        self.rec = (self.sidx[:, None], i["rec"][..., 0].long() + P, i["rec"][..., 1].long() + P)

    def start(self):
        z = torch.zeros(self.S, *self.leaf.shape[-2:], device="cuda", dtype=torch.float64)
        return tuple(z for _ in range(6))

    def coefficients(self, leaf):
        return leaf * leaf * self.scale

    def step(self, s, K, w, n):
        u, up, px, pz, zx, zz = s
        d2x, d1x = _centred(u, 2)
        d2z, d1z = _centred(u, 1)
        wx = d2x + self.mx * _centred(px, 2)[1]
        wz = d2z + self.mz * _centred(pz, 1)[1]
        zx, zz = self.ax * zx + self.bx * wx, self.az * zz + self.bz * wz
        px, pz = self.ax * px + self.bx * d1x, self.az * pz + self.bz * d1z
        un = 2 * u - up + K * (wx + zx + wz + zz)
        un = un.index_put(self.src, K[self.src[1], self.src[2]] * w[:, n], accumulate=True)
        return (un, u, px, pz, zx, zz), un[self.rec][:, None]

    def illum(self, s):
        P = self.P
        u = _interior(s[0], P)
        return (u * u).sum(0)

    kernels, fields = 110, 60


def _interior(f, P):
    return f[..., P:f.shape[-2] - P, P:f.shape[-1] - P]


class _Elastic(_Acoustic):
    def __init__(self, case, i):
        P, self.S, self.nt = case["pml"], case["shots"], case["nt"]
        self.dt, self.dx, self.P = _f32(DT_EL), _f32(DX_EL), P
        self.leaf = F.pad(i["model"].double()[None], (P, P, P, P), mode="replicate")[0]
        f = _f32(F_EL)
        for ax, n in (("z", case["nz"]), ("x", case["nx"])):
            for half in (False, True):
                a, b, _ = _profile(n, P, self.dx, self.dt, VP_MAX, f, half)
                shape = (1, -1, 1) if ax == "z" else (1, 1, -1)
                setattr(self, ax + ("h" if half else "i"), (a.view(shape), b.view(shape)))
        self._positions(i, P)
        self.w = i["wav"].detach().double()

    def start(self):
        z = torch.zeros(self.S, *self.leaf.shape[-2:], device="cuda", dtype=torch.float64)
        return tuple(z for _ in range(13))

    def coefficients(self, leaf):
        vp, vs, rho = leaf
        mu = rho * vs * vs

        def right(t):
            return torch.cat([t[:, 1:], t[:, -1:]], 1)

        def down(t):
            return torch.cat([t[1:], t[-1:]], 0)

        r = 1 / mu
        dt = self.dt
        return (dt * 2 / (rho + right(rho)), dt * 2 / (rho + down(rho)), dt * rho * vp * vp,
                dt * rho * (vp * vp - 2 * vs * vs),
                dt * 4 / (r + right(r) + down(r) + right(down(r))))

    def step(self, s, c, w, n):
        vx, vz, txx, tzz, txz, *p = s
        bx, bz, l2m, lam, mu = c

        def d(f, ax, plus, k, prof):
            g = _staggered(f, ax, plus) / self.dx
            p[k] = prof[0] * p[k] + prof[1] * g
            return g + p[k]

        vx = vx + bx * (d(txx, 2, True, 0, self.xh) + d(txz, 1, False, 1, self.zi))
        vz = vz + bz * (d(txz, 2, False, 2, self.xi) + d(tzz, 1, True, 3, self.zh))
        out = torch.stack([vx[self.rec], vz[self.rec]], 1)
        ex, ez = d(vx, 2, False, 4, self.xi), d(vz, 1, False, 5, self.zi)
        txx, tzz = txx + l2m * ex + lam * ez, tzz + lam * ex + l2m * ez
        txz = txz + mu * (d(vx, 1, True, 6, self.zh) + d(vz, 2, True, 7, self.xh))
        amp = self.dt * w[:, n] / self.dx ** 2
        txx = txx.index_put(self.src, amp, accumulate=True)
        tzz = tzz.index_put(self.src, amp, accumulate=True)
        return (vx, vz, txx, tzz, txz, *p), out

    kernels, fields = 110, 130


def _exact_survey(case, i, residual_of, want_grad):
    """Data, and with want_grad the gradients of the misfit whose data
    gradient is residual_of(data), with respect to the model and wavelets:
    reverse-mode differentiation over checkpointed segments."""
    e = (_Elastic if case["physics"] == "elastic" else _Acoustic)(case, i)
    nt, C = e.nt, max(1, int(math.sqrt(e.nt)))
    cells = e.S * e.leaf.shape[-2] * e.leaf.shape[-1]
    step_s = max(e.kernels * 6e-6, e.fields * cells * 24 / 4e12)
    if nt * step_s * (5.0 if want_grad else 1.0) > LIMIT_S:
        return None
    state, ck, tr, illum = e.start(), [], [], 0.0
    with torch.no_grad():
        c = e.coefficients(e.leaf)
        for n in range(nt):
            if want_grad and n % C == 0:
                ck.append(state)
            if case["illum"]:
                illum = illum + e.illum(state)
            state, d = e.step(state, c, e.w, n)
            tr.append(d)
    data = torch.stack(tr, -1)
    if not want_grad:
        return dict(data=data)
    r = residual_of(data)
    leaf, w = e.leaf.clone().requires_grad_(True), e.w.clone().requires_grad_(True)
    adj = [torch.zeros_like(t) for t in state]
    g_leaf, g_w = torch.zeros_like(leaf), torch.zeros_like(w)
    for k in reversed(range(len(ck))):
        s0 = tuple(t.clone().requires_grad_(True) for t in ck[k])
        ck[k] = None
        s, c, traces = s0, e.coefficients(leaf), []
        for n in range(k * C, min(nt, (k + 1) * C)):
            s, d = e.step(s, c, w, n)
            traces.append(d)
        seg = torch.stack(traces, -1)
        got = torch.autograd.grad([seg, *s], [leaf, w, *s0],
                                  [r[..., k * C:k * C + seg.shape[-1]], *adj], allow_unused=True)
        g_leaf, g_w = g_leaf + got[0], g_w + got[1]
        adj = [torch.zeros_like(t) if a is None else a for a, t in zip(got[2:], s0)]
    return dict(data=data, grad=_interior(g_leaf, e.P), grad_w=g_w,
                illum=illum if case["illum"] else None, misfit=0.5 * (r * r).sum())


def _exact_unet(case, i, train):
    theta = i["theta"].double().requires_grad_(train)
    parts, k = [], 0
    for ci, co in UNET_LAYERS:
        wgt = theta[k:k + co * 9 * ci].view(co, 3, 3, ci).permute(0, 3, 1, 2)
        k += co * 9 * ci
        parts.append((wgt, theta[k:k + co]))
        k += co
    head_w, head_b = theta[k:k + 32], theta[k + 32]

    def conv(x, n):
        return F.conv2d(x, parts[n][0], parts[n][1], padding=1).relu()

    def up(x):
        return F.interpolate(x, scale_factor=2, mode="nearest")

    x = F.pad(i["x"].double(), (0, 32 - case["channels"])).permute(0, 3, 1, 2)
    skips = []
    for n in (0, 2, 4):
        x = conv(conv(x, n), n + 1)
        skips.append(x)
        x = F.avg_pool2d(x, 2)
    x = conv(conv(x, 6), 7)
    for n in (8, 11, 14):
        x = torch.cat([conv(up(x), n), skips.pop()], 1)
        x = conv(conv(x, n + 1), n + 2)
    out = (x * head_w[None, :, None, None]).sum(1) + head_b
    if not train:
        return out
    loss = ((out - i["target"].double()) ** 2).mean()
    g, = torch.autograd.grad(loss, theta)
    step = 1001
    m = 0.9 * i["m"].double() + 0.1 * g
    v = 0.999 * i["v"].double() + 0.001 * g * g
    th = theta - 5e-4 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    return dict(loss=loss.detach(), out=out.detach(), grad=g, theta=th.detach(), m=m, v=v)


def _exact_layer(case, i):
    x, dy, wgt = (i[k].double() for k in ("x", "dy", "w"))
    co, ci = case["cout"], case["cin"]
    w4 = wgt.view(co, 3, 3, ci).permute(0, 3, 1, 2)
    xn, dyn = x.permute(0, 3, 1, 2), dy.permute(0, 3, 1, 2)
    out = F.conv2d(xn, w4, i["bias"].double(), padding=1).relu()
    dx = F.conv2d(dyn, w4.flip(2, 3).transpose(0, 1), padding=1) * (xn > 0)
    xp = F.pad(x, (0, 0, 1, 1, 1, 1))
    h, w = case["height"], case["width"]
    flat = dy.reshape(-1, co).t()
    dw = torch.stack([flat @ xp[:, ky:ky + h, kx:kx + w].reshape(-1, ci)
                      for ky in range(3) for kx in range(3)], 1)
    return dict(out=out.permute(0, 2, 3, 1), dx=dx.permute(0, 2, 3, 1), dw=dw)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":  # the problems are the gradient cases' own; together they take too long
        return None
    if kind == "layer":
        return _exact_layer(case, _layer_inputs(case, seed))
    if kind in ("train", "infer"):
        return _exact_unet(case, _unet_inputs(case, seed), kind == "train")
    i = _survey_inputs(case, seed)
    got = _exact_survey(case, i, lambda d: d - i["d_obs"].double(), kind != "forward")
    if got is None:
        return None
    if kind == "forward":
        return got["data"]
    if kind == "autograd":
        return dict(data=got["data"], grad_v=got["grad"], grad_w=got["grad_w"])
    return dict(grad=got["grad"], misfit=got["misfit"], illum=got["illum"])
