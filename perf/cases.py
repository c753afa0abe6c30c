"""Performance cases: what a user of the library has it compute, with plain 64-bit references.

Two kinds of work carry the library.  A design evaluation (``Solver.evaluate``:
set the design and the damping, forward run, adjoint run, gradient) is what
every optimization loop repeats; it comes in the three solver modes (2D with E
out of plane, 2D with E in plane, 3D), two precisions and several ways to
keep the forward record.  The surrogate network (``UNet``) is trained on what
the evaluations give and predicts sensitivity maps between them.

Grids, boxes, absorbing layers, filters and checkpoint settings are those of
the workloads in ``inputs`` and of the tests.  Runs are shorter than an
optimization's; the pulse is shortened with them, so that every run sees the
wave reach the gap and the adjoint has a source.
"""
import math

import numpy as np
import torch

from paper_2203_01462_gb300 import inputs as I
from paper_2203_01462_gb300.binding import Solver
from paper_2203_01462_gb300.surrogate import UNet

DAMPING = (5e5, 3.0)  # sigma_max of the paper's sweep, a middle level of the damping continuation
LR = 1e-3

_EZ = dict(kind="ez", npml=10, gap=3, material="gold", filter=0, snap=0, snap_dtype="f32")
_IP = dict(kind="inplane", npml=15, gap=20, material="silver", filter=0, snap=64, snap_dtype="f32")
_3D = dict(kind="yee", npml=12, gap=4, material="gold", filter=0, snap=0, snap_dtype="f32")


def listed():
    return [
        # The smallest run: a ragged grid of the parity tests in FP64, where launches and latency are all there is.
        dict(_EZ, name="ez 41x37 f64", nx=41, ny=37, dw=17, dh=15, npml=6, real="f64", nsteps=400, dx_nm=20.0,
             half_thz=300.0, src_offset=2),
        # The FP64 configuration that is compared with the oracle in full: 160^2, 2000 steps, the whole history kept.
        dict(_EZ, name="ez 160x160 f64", nx=160, ny=160, dw=60, dh=60, real="f64", nsteps=2000, dx_nm=5.0,
             half_thz=300.0, src_offset=5),
        # One solve of the surrogate loop: 316^2, a 256^2 design box, 4000 steps, the whole history kept.
        dict(_EZ, name="ez 316x316 f32", nx=316, ny=316, dw=256, dh=256, real="f32", nsteps=4000, dx_nm=5.0,
             half_thz=100.0, src_offset=5),
        # A medium ragged grid: filtered design, 16-bit checkpoints every 32 steps.
        dict(_EZ, name="ez 530x303 f32 bf16", nx=530, ny=303, dw=251, dh=61, real="f32", nsteps=1000, dx_nm=10.0,
             half_thz=200.0, src_offset=20, filter=5, snap=32, snap_dtype="bf16"),
        # The largest 2D workload: 2048^2, a filtered 1024^2 design box, lossless checkpoints every 64 steps.
        dict(_EZ, name="ez 2048x2048 f32", nx=2048, ny=2048, dw=1024, dh=1024, real="f32", nsteps=1792, dx_nm=2.0,
             half_thz=600.0, src_offset=490, filter=5, snap=64),
        # The paper's two 2D antenna geometries (E in plane, 0.5 nm cells, 100 and 200 nm design boxes).
        dict(_IP, name="inplane 291x291 f32", nx=291, ny=291, dw=200, dh=200, real="f32", nsteps=2560, dx_nm=0.5,
             half_thz=600.0, src_offset=5),
        dict(_IP, name="inplane 491x491 f32", nx=491, ny=491, dw=400, dh=400, real="f32", nsteps=3072, dx_nm=0.5,
             half_thz=600.0, src_offset=5),
        # A small ragged 3D grid in FP64: current sheet over a substrate, the whole history kept.
        dict(_3D, name="yee 80x34x40 f64", nx=80, ny=34, nz=40, dw=26, dh=12, dd=10, npml=4, gap=2, real="f64",
             nsteps=300, dx_nm=20.0, half_thz=300.0, src="sheet", src_offset=2, substrate=True),
        # The 3D plane-wave workload: 256^3, a 128 x 128 x 64 slab on a substrate, BF16 checkpoints every 32 steps.
        dict(_3D, name="yee 256x256x256 f32 bf16", nx=256, ny=256, nz=256, dw=128, dh=128, dd=64, real="f32",
             nsteps=480, dx_nm=5.0, half_thz=600.0, src="tfsf", src_offset=5, substrate=True, snap=32,
             snap_dtype="bf16"),
        # The largest 3D workload: 512 x 512 x 384, a dipole in the gap, FP16 checkpoints.
        dict(_3D, name="yee 512x512x384 f32 f16", nx=512, ny=512, nz=384, dw=256, dh=256, dd=96, real="f32",
             nsteps=96, dx_nm=5.0, half_thz=2000.0, src="dipole", src_offset=5, substrate=False, snap=48,
             snap_dtype="f16"),
        # One training step of the surrogate network on a batch of 256^2 maps, and one prediction.
        dict(kind="train", name="unet train 8x256x256 bf16", base=24, batch=8, H=256, W=256, precision="bf16"),
        dict(kind="predict", name="unet predict 256x256 bf16", base=24, batch=1, H=256, W=256, precision="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ez", "ez", "inplane", "inplane", "yee", "yee", "train", "predict"])
    if kind in ("train", "predict"):
        h, w = (8 * _log_int(rng, 4, 32) for _ in range(2))
        return dict(kind=kind, base=rng.choice([8, 16, 24]), batch=rng.randint(1, 8) if kind == "train" else 1, H=h, W=w,
                    precision=rng.choice(["bf16", "bf16", "f32"]))
    c = dict({"ez": _EZ, "inplane": _IP, "yee": _3D}[kind])
    c["real"] = rng.choice(["f32", "f32", "f64"])
    c["material"] = rng.choice(["gold", "silver"])
    c["snap"] = rng.choice([0, rng.randint(8, 64)])
    c["snap_dtype"] = rng.choice(["f32", "bf16", "f16"])
    c["dx_nm"], c["half_thz"] = 20.0, 300.0
    if kind == "yee":
        top = 200 if c["real"] == "f32" else 90
        c["npml"] = rng.choice([4, 8, 12])
        n = [_log_int(rng, 2 * c["npml"] + 18, top) for _ in range(3)]
        c["nx"], c["ny"], c["nz"] = n
        c["dw"], c["dh"], c["dd"] = (max(6, int((v - 2 * c["npml"] - 8) * rng.uniform(0.4, 0.9))) for v in n)
        c["gap"], c["src"] = 2, rng.choice(["sheet", "tfsf", "dipole"])
        c["substrate"], c["src_offset"] = rng.random() < 0.5, 1
        if c["src"] == "tfsf":  # the total-field box lies strictly around the design box
            c["dd"] = max(4, min(c["dd"], c["nz"] - 2 * c["npml"] - 12))
        c["nsteps"] = rng.randint(150, 260) + c["nz"]
    else:
        top = 1400 if c["real"] == "f32" else 500
        c["npml"] = rng.choice([6, 10, 15])
        n = [_log_int(rng, 2 * c["npml"] + 18, top) for _ in range(2)]
        c["nx"], c["ny"] = n
        c["dw"], c["dh"] = (max(8, int((v - 2 * c["npml"] - 8) * rng.uniform(0.3, 0.95))) for v in n)
        c["gap"] = rng.choice([3, 4]) if kind == "ez" else rng.choice([2, 4, 6])
        c["filter"] = rng.choice([0, 3, 5]) if kind == "ez" else 0
        c["src_offset"] = max(1, (c["ny"] - c["dh"]) // 2 - c["npml"] - 3)
        c["nsteps"] = rng.randint(260, 500) + c["dh"]
    return c


def _workload(c):
    """The problem description of a case, through the library's own builders."""
    mat = I.SILVER if c["material"] == "silver" else I.GOLD
    common = dict(dx=c["dx_nm"] * 1e-9, nsteps=c["nsteps"], npml=c["npml"], real=c["real"], material=mat,
                  snapshot_every=c["snap"], snapshot_dtype=c["snap_dtype"], src_offset=c["src_offset"])
    g = c["gap"]
    if c["kind"] == "yee":
        w = I.workload_3d(c["nx"], c["ny"], c["nz"], design=(c["dw"], c["dh"], c["dd"]), gap=(g, g, g),
                          source=c["src"], substrate=c["substrate"], tf_margin=1, **common)
    elif c["kind"] == "inplane":
        w = I.workload_2d_inplane(c["nx"], c["ny"], design=(c["dw"], c["dh"]), gap=(g, g), **common)
    else:
        w = I.workload_2d(c["nx"], c["ny"], design=(c["dw"], c["dh"]), gap=(g, g), filter_radius=c["filter"],
                          **common)
    w.update(I.pulse(413e-9 if c["kind"] == "inplane" else 800e-9, c["half_thz"] * 1e12))
    return w


def _design(w, seed):
    """A design on its way: a bowtie that has not closed yet over a nearly empty box, as optimization loops hold it."""
    u = np.random.Generator(np.random.PCG64(seed)).random(I.design_shape(w), dtype=np.float32)
    return (0.03 * u + I.rho_bowtie(w).astype(np.float32) * (0.35 + 0.6 * u)).reshape(-1)


def _maps(c, seed):
    """Network inputs [2][B][H][W] (density, damping level) and targets [1][B][H][W] (maps scaled to a maximum of 1)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    B, H, W = c["batch"], c["H"], c["W"]
    x = np.empty((2, B, H, W), dtype=np.float32)
    x[0] = rng.random((B, H, W), dtype=np.float32)
    x[1] = rng.random((B, 1, 1), dtype=np.float32)
    yy, xx = np.mgrid[0:H, 0:W].astype(np.float32)
    t = np.empty((1, B, H, W), dtype=np.float32)
    for b in range(B):
        ky, kx, ph = rng.uniform(0.02, 0.2), rng.uniform(0.02, 0.2), rng.uniform(0, 6.28)
        m = np.sin(ky * yy + kx * xx + ph) * np.exp(-((yy - H / 2) / H) ** 2 - ((xx - W / 2) / W) ** 2) + 0.3 * x[0, b]
        t[0, b] = m / np.abs(m).max()
    return x, t


def prepare(case, seed):
    if case["kind"] in ("train", "predict"):
        x, t = (torch.from_numpy(a).cuda() for a in _maps(case, seed))
        net = UNet(base=case["base"], batch=case["batch"], H=case["H"], W=case["W"], seed=seed,
                   precision=case["precision"])
        return dict(kind=case["kind"], net=net, x=x, t=t)
    w = _workload(case)
    s = Solver(w)
    return dict(kind=case["kind"], s=s, rho=torch.from_numpy(_design(w, seed)).to("cuda", s.real))


def run(state):
    if state["kind"] == "predict":
        return state["net"].forward(state["x"])
    if state["kind"] == "train":
        net = state["net"]
        loss = net.train_step(state["x"], state["t"], LR)
        return dict(loss=loss, gw=net.gw, gb=net.gb, w=net.w, b=net.b)
    W, g = state["s"].evaluate(state["rho"], *DAMPING)
    return dict(W=W, gradient=g)


def work(case):
    """Inputs once, outputs once; arithmetic of the forward and adjoint steps (no recompute), or of the network's
    products."""
    if case["kind"] in ("train", "predict"):
        px = case["batch"] * case["H"] * case["W"]
        macs = sum(ci * co * k * k * px // 4 ** UNet._level(n) for n, ci, co, k in I.unet_layers(case["base"]))
        params = I.unet_param_count(case["base"])
        if case["kind"] == "predict":
            return dict(bytes=4 * (3 * px + params), flops=2 * macs)
        return dict(bytes=4 * (3 * px + 8 * params), flops=6 * macs)
    w = _workload(case)
    rb = 8 if case["real"] == "f64" else 4
    md, n, N = I.n_design(w), I.n_cells(w), case["nsteps"]
    node, ne = {"ez": (11, 1), "inplane": (13, 1), "yee": (36, 3)}[case["kind"]]
    return dict(bytes=md * rb + 8 * md + 8, flops=N * (2 * node * n + ne * md * (2 * 14 + 10)))


# ------------------------------------------------------------------ 64-bit references

def exact(case, seed):
    if case["kind"] in ("train", "predict"):
        return _exact_net(case, seed)
    w = _workload(case)
    W, g = _exact_fields(w, _design(w, seed).astype(np.float64), *DAMPING, device="cuda")
    return dict(W=W, gradient=g)


def _exact_net(c, seed):
    F = torch.nn.functional
    x, t = (torch.from_numpy(a).cuda().double().transpose(0, 1) for a in _maps(c, seed))
    layers = I.unet_layers(c["base"])
    p = {k: torch.tensor(np.asarray(v, dtype=np.float32), device="cuda").double().requires_grad_(c["kind"] == "train")
         for k, v in I.unet_params(c["base"], seed).items()}
    size = {n: k for n, _, _, k in layers}

    def conv(n, v, act=True):
        if size[n] == 1:
            y = torch.einsum("oi,bihw->bohw", p[n + ".w"][:, :, 0, 0], v) + p[n + ".b"][None, :, None, None]
        else:
            # nine shifted products instead of a 64-bit library convolution
            pad = F.pad(v, (1, 1, 1, 1))
            y = p[n + ".b"][None, :, None, None]
            for q in range(9):
                sh = pad[:, :, q // 3:q // 3 + v.shape[2], q % 3:q % 3 + v.shape[3]]
                y = y + torch.einsum("oi,bihw->bohw", p[n + ".w"][:, :, q // 3, q % 3], sh)
        return F.relu(y) if act else y

    def up(v):
        return v.repeat_interleave(2, 2).repeat_interleave(2, 3)

    e1 = conv("enc1b", conv("enc1a", x))
    e2 = conv("enc2b", conv("enc2a", F.avg_pool2d(e1, 2)))
    e3 = conv("enc3b", conv("enc3a", F.avg_pool2d(e2, 2)))
    bo = conv("botb", conv("bota", F.avg_pool2d(e3, 2)))
    d3 = conv("dec3b", conv("dec3a", torch.cat([up(bo), e3], 1)))
    d2 = conv("dec2b", conv("dec2a", torch.cat([up(d3), e2], 1)))
    d1 = conv("dec1b", conv("dec1a", torch.cat([up(d2), e1], 1)))
    y = conv("head", d1, act=False)
    if c["kind"] == "predict":
        return y.transpose(0, 1).contiguous()
    loss = ((y - t) ** 2).mean()
    loss.backward()
    out = dict(loss=loss.detach().reshape(1), gw={}, gb={}, w={}, b={})
    for n, ci, co, k in layers:
        for s in ("w", "b"):
            v, g = p[n + "." + s].detach(), p[n + "." + s].grad
            shape = (co, ci * k * k) if s == "w" else (co,)
            out["g" + s][n] = g.reshape(shape)
            # Adam's first step: both moments' bias corrections cancel.  The biases start at zero, so theirs is the
            # gradient's sign alone, which 16-bit products do not settle where the gradient is next to nothing.
            out[s][n] = (v - LR * g / (g.abs() + 1e-8)).reshape(shape) if s == "w" else None
    return out


_C0, _MU0 = 299792458.0, 1.25663706212e-6
_EPS0 = 1.0 / (_MU0 * _C0 * _C0)


def _cpml(w, n, half):
    """b, c and 1/kappa of the absorbing layer's recursive convolution at the n (half-)positions of an axis."""
    L, dt = w["npml"], w["courant"] * w["dx"] / _C0
    b, c, ki = np.zeros(n), np.zeros(n), np.ones(n)
    for i in range(n):
        p = i + (0.5 if half else 0.0)
        d = max(L - p, p - (n - 1 - L), 0.0)
        if L <= 0 or d <= 0 or (half and i == n - 1):
            continue
        x = d / L
        sig = w["pml_sigma_factor"] * (w["pml_m"] + 1) / (_MU0 * _C0 * w["dx"]) * x ** w["pml_m"]
        kap, alp = 1 + (w["pml_kappa_max"] - 1) * x ** w["pml_m"], w["pml_alpha_max"] * (1 - x)
        b[i] = math.exp(-(sig / kap + alp) * dt / _EPS0)
        c[i] = sig / (sig * kap + kap * kap * alp) * (b[i] - 1)
        ki[i] = 1 / kap
    return b, c, ki


def _signal(w, dt):
    u = (np.arange(w["nsteps"]) + 0.5) * dt - w["t0"]
    return w["src_amp"] * w["courant"] * np.exp(-(u / w["tau"]) ** 2) * sum(
        np.sin(2 * math.pi * f * u) for f in w["f0"][:w["nbands"]])


def _gauss(w, v, transpose):
    """The truncated Gaussian design filter of a (rows, columns) map, normalised at the edges, or its transpose."""
    R = w["filter_radius"]
    for dim in (0, 1):
        n = v.shape[dim]
        k = torch.arange(n, device=v.device, dtype=v.dtype)
        d = k[:, None] - k[None, :]
        m = torch.exp(-d * d / (2 * w["filter_sigma"] ** 2)) * (d.abs() <= R)
        m = m / m.sum(1, keepdim=True)
        m = m.T if transpose else m
        v = m @ v if dim == 0 else v @ m.T
    return v


def _exact_fields(w, rho, sigma_max, gamma_scale, device="cpu"):
    """W~ and its gradient: the leapfrog of the fields and Drude currents, forward and adjoint, on whole 64-bit arrays."""
    nd, S, N = w["ndim"], w["courant"], w["nsteps"]
    n = [w["nx"], w["ny"], w["nz"]][:nd]
    dt = S * w["dx"] / _C0
    kw = dict(dtype=torch.float64, device=device)
    plane = nd == 2 and w.get("pol", 0) == 1
    x, y = 0, 1
    # curl terms (sign, component, axis) of every H and E component; the axis each E component lies along
    if nd == 3:
        hc = ec = [[(1, (c + 2) % 3, (c + 1) % 3), (-1, (c + 1) % 3, (c + 2) % 3)] for c in range(3)]
        along = [0, 1, 2]
    elif plane:
        hc, ec, along = [[(1, 1, x), (-1, 0, y)]], [[(1, 0, y)], [(-1, 0, x)]], [0, 1]
    else:
        hc, ec, along = [[(1, 0, y)], [(-1, 0, x)]], [[(1, 1, x), (-1, 0, y)]], [None]
    shape = tuple(reversed(n))

    def on(ax, v):  # a vector along an axis, as an array that broadcasts
        return torch.as_tensor(v, **kw).reshape([-1 if d == nd - 1 - ax else 1 for d in range(nd)])

    def box(lo, hi):
        return tuple(slice(int(lo[a]), int(hi[a])) for a in reversed(range(nd)))

    def ends(ax, first, last):
        v = np.ones(n[ax])
        v[-1] = 0.0 if last else 1.0
        v[0] = 0.0 if first else 1.0
        return v

    pmlE = [[on(a, t) for t in _cpml(w, n[a], False)] for a in range(nd)]
    pmlH = [[on(a, t) for t in _cpml(w, n[a], True)] for a in range(nd)]
    maskH = [math.prod([on(a, ends(a, False, True)) for _, _, a in t], start=torch.ones((), **kw)) for t in hc]
    # boxes of every E component: design, gap and source (edges of a cell box with E in plane)
    nE = len(ec)

    def comp_box(lo, hi, c):
        hi = [hi[a] + (1 if plane and a != along[c] else 0) for a in range(nd)]
        return list(lo[:nd]), hi

    des = [comp_box(w["design_lo"], w["design_hi"], c) for c in range(nE)]
    gap = [comp_box(w["gap_lo"], w["gap_hi"], c) for c in range(nE)]
    parts, at = [], 0
    for c in range(nE):
        sh = tuple(des[c][1][a] - des[c][0][a] for a in reversed(range(nd)))
        k = math.prod(sh)
        r = torch.as_tensor(rho[at:at + k] if plane else rho, **kw).reshape(sh)
        parts.append(_gauss(w, r, False) if w["filter_radius"] else r)
        at += k if plane else 0
    inv, dru = [], []
    kJ = (1 - 0.5 * w["gamma_p"] * gamma_scale * dt) / (1 + 0.5 * w["gamma_p"] * gamma_scale * dt)
    i1g = 1 / (1 + 0.5 * w["gamma_p"] * gamma_scale * dt)
    psi_m = (w["omega_p"] * dt) ** 2
    for c in range(nE):
        e = torch.full(shape, 1 / w["eps_s"], **kw)
        if nd == 3 and w["sub_hi"] > 0:
            e[:w["sub_hi"]] = 1 / w["sub_eps"]
        e[box(*gap[c])] = 1 / w["eps_g"]
        for a in range(nd):
            e *= on(a, ends(a, a != along[c], True))
        rt = parts[c]
        free = torch.ones_like(rt)
        free[box([gap[c][0][a] - des[c][0][a] for a in range(nd)], [gap[c][1][a] - des[c][0][a] for a in range(nd)])] = 0
        e[box(*des[c])] *= 1 - free
        inv.append(e)
        eps = w["eps_s"] + rt * (w["eps_inf"] - w["eps_s"])
        psi = w["psi_s_ratio"] * psi_m + rt * (1 - w["psi_s_ratio"]) * psi_m
        smax = sigma_max * dt / _EPS0 * (4 if w["sigma_form"] else 1)
        bJ = 0.5 * psi * i1g
        hs = 0.5 * (smax * rt * (1 - rt) + bJ)
        dru.append(dict(free=free, ca=(eps - hs) / (eps + hs) * free, cb=free / (eps + hs), bJ=bJ * free, smax=smax,
                        a1=smax * (1 - 2 * rt) * 0.5, a2=(1 - w["psi_s_ratio"]) * psi_m * 0.5 / psi))
    src = _signal(w, dt)
    sbox = box(w["src_lo"], w["src_hi"])
    scomp = w["src_comp"] if nd == 3 else 0
    tf = _incident(w, src) if w.get("tfsf") else None

    def zeros():
        return dict(E=[torch.zeros(shape, **kw) for _ in ec], H=[torch.zeros(shape, **kw) for _ in hc],
                    J=[torch.zeros_like(p) for p in parts],
                    pE=[[torch.zeros(shape, **kw) for _ in t] for t in ec],
                    pH=[[torch.zeros(shape, **kw) for _ in t] for t in hc])

    def diff(f, ax, forward):
        d, m = torch.zeros_like(f), nd - 1 - ax
        a, b = f.narrow(m, 1, n[ax] - 1), f.narrow(m, 0, n[ax] - 1)
        torch.sub(a, b, out=d.narrow(m, 0 if forward else 1, n[ax] - 1))
        return d

    def curl(F, terms, psi, pml, forward):
        out = None
        for (sg, k, ax), p in zip(terms, psi):
            d = diff(F[k], ax, forward)
            b, c, ki = pml[ax]
            p.mul_(b).addcmul_(d, c)
            d.mul_(ki).add_(p)
            out = d.mul_(sg) if out is None else out.add_(d, alpha=sg)
        return out.mul_(S)

    def step(s, forward_n=None, gap_src=None):
        for c, t in enumerate(hc):
            s["H"][c] -= maskH[c] * curl(s["E"], t, s["pH"][c], pmlH, True)
        if tf is not None and forward_n is not None:
            _faces_h(w, s["H"], tf[0][forward_n], S)
        old = []
        for c, t in enumerate(ec):
            E, q = s["E"][c], dru[c]
            cu = curl(s["H"], t, s["pE"][c], pmlE, False)
            if forward_n is not None:
                if tf is None and c == scomp:
                    cu[sbox] -= src[forward_n]
            else:
                cu[box(*gap[c])] += w["eps_g"] * gap_src[c]
            b = box(*des[c])
            eo, jo = E[b].clone(), s["J"][c]
            E.addcmul_(inv[c], cu)
            en = E[b] * (1 - q["free"]) + q["ca"] * eo + q["cb"] * (cu[b] - 0.5 * (1 + kJ) * jo)
            E[b] = en
            jn = kJ * jo + q["bJ"] * (en + eo)
            old.append((eo, en, jo, jn))
            s["J"][c] = jn
        if tf is not None and forward_n is not None:
            _faces_e(w, s["E"], tf[1][forward_n], S)
        return old

    s, rec, gaps = zeros(), [], [[torch.zeros_like(s_[box(*g)]) for s_, g in zip([torch.zeros(shape, **kw)] * nE, gap)]]
    W = torch.zeros((), **kw)
    for k in range(N):
        step(s, forward_n=k)
        rec.append([s["E"][c][box(*des[c])].clone() for c in range(nE)])
        gaps.append([s["E"][c][box(*gap[c])].clone() for c in range(nE)])
        W += sum((g * g).sum() for g in gaps[-1])
    scale = dt * w["dx"] ** nd
    W *= 0.5 * w["eps_g"] * scale
    s, G = zeros(), [torch.zeros_like(p) for p in parts]
    for m in range(N, 0, -1):
        for c, (eo, en, jo, jn) in enumerate(step(s, gap_src=gaps[m])):
            q = dru[c]
            term = -(w["eps_inf"] - w["eps_s"]) * (en - eo) - q["a1"] * (en + eo) - q["a2"] * (jn + jo)
            G[c] += rec[m - 1][c] * term * q["free"]
    g = torch.cat([v.reshape(-1) for v in G]) if plane else sum(G)
    if w["filter_radius"]:
        g = _gauss(w, g, True) * dru[0]["free"]
    return W.reshape(1), scale * g.reshape(-1)


def _incident(w, src):
    """E_x^n and H_y^{n+1/2} of the plane wave's column, one row per step."""
    nz, S = w["nz"], w["courant"]
    (bE, cE, kE), (bH, cH, kH) = _cpml(w, nz, False), _cpml(w, nz, True)
    E, H, pE, pH = (np.zeros(nz) for _ in range(4))
    inv = np.where(np.arange(nz) < w["sub_hi"], 1 / w["sub_eps"], 1 / w["eps_s"])
    inv[0] = inv[-1] = 0.0
    rows = [[], []]
    for v in src:
        rows[0].append(E.copy())
        d = np.append(E[1:] - E[:-1], 0.0)
        pH = bH * pH + cH * d
        H[:-1] -= S * (d * kH + pH)[:-1]
        rows[1].append(H.copy())
        d = np.append(0.0, H[1:] - H[:-1])
        pE = bE * pE + cE * d
        J = np.zeros(nz)
        J[w["src_lo"][2]] = v
        E = E + inv * (-S * (d * kE + pE) - J)
    return rows


def _faces_h(w, H, e, S):
    (lx, ly, lz), (ux, uy, uz) = w["tf_lo"], w["tf_hi"]
    H[1][lz - 1, ly:uy + 1, lx:ux] += S * e[lz]
    H[1][uz, ly:uy + 1, lx:ux] -= S * e[uz]
    col = torch.as_tensor(e[lz:uz + 1], dtype=H[2].dtype, device=H[2].device)[:, None]
    H[2][lz:uz + 1, ly - 1, lx:ux] -= S * col
    H[2][lz:uz + 1, uy, lx:ux] += S * col


def _faces_e(w, E, h, S):
    (lx, ly, lz), (ux, uy, uz) = w["tf_lo"], w["tf_hi"]
    eps = np.where(np.arange(w["nz"]) < w["sub_hi"], w["sub_eps"], w["eps_s"])
    E[0][lz, ly:uy + 1, lx:ux] += S * h[lz - 1] / eps[lz]
    E[0][uz, ly:uy + 1, lx:ux] -= S * h[uz] / eps[uz]
    col = torch.as_tensor((h / eps)[lz:uz], dtype=E[2].dtype, device=E[2].device)[:, None]
    E[2][lz:uz, ly:uy + 1, lx] -= S * col
    E[2][lz:uz, ly:uy + 1, ux] += S * col
