"""The work this framework is used for, as timed passes through its public entry points.

Three kinds of program use it.  A dose calculation creates a handle for a phantom once and then
runs plans on it: reset, transport, fetch (the water, slab, insert, sphere and CT cases: from the
10^4-proton pencil beam, where latency counts, to a 2000-spot plan).  The learned dose runs a
10^5-history plan and one inference of the denoiser; training it takes Adam steps on such pairs.
The convolutions under it are public calls of their own, forward, data gradient (the forward
call on flipped weights) and weight gradient, and a dose is judged with the gamma index.
"""
import math
import os

import numpy as np
import torch
import torch.nn.functional as F

import paper_2511_03115_gb300 as S
import sde_workloads as W

#: Outputs of a transport are whole numbers (the 64-bit tally and the balance), so they are equal
#: for equal seeds; the dose is those numbers over the voxel masses.
BALANCE = ("incident", "deposited", "escaped", "removed", "histories", "steps", "jumps_elastic", "jumps_inelastic")


# ------------------------------------------------------------------------------ the cases
def _transport(name, phantom, histories, *, nx=0, ny=0, nz=0, h=1.0, n_spots=1, e_lo=150.0, e_hi=150.0, sigma=3.0,
               chord=False, cut=0.0, secondaries=0.0, resident=False, fetch="device"):
    return dict(name=name, kind="transport", phantom=phantom, histories=histories, nx=nx, ny=ny, nz=nz, h=h,
                n_spots=n_spots, e_lo=e_lo, e_hi=e_hi, sigma=sigma, chord=chord, cut=cut, secondaries=secondaries,
                resident=resident, fetch=fetch)


def _conv(name, n, d, h, w, cin, cout, *, relu=True, fp32=False, bias=True):
    return dict(name=name, kind="conv", n=n, d=d, h=h, w=w, cin=cin, cout=cout, relu=relu, fp32=fp32, bias=bias)


def listed():
    return [
        # the first call of anyone: a 100 MeV pencil beam in water, results on the host
        _transport("pencil_water_10k", "water", 10_000, e_lo=100.0, e_hi=100.0, sigma=0.0, fetch="host"),
        # the input of the learned dose: 24 Gaussian spots, 10^5 protons, the dose left on the device
        _transport("low_history_plan_100k", "spheres", 100_000, nx=128, ny=128, nz=192, n_spots=24, e_lo=70.0,
                   e_hi=200.0, fetch="f32"),
        # one Gaussian beam at half-millimetre voxels through bone and lung
        _transport("slab_half_mm_1m", "slab", 1_000_000),
        # a spread-out Bragg peak in a CT with five materials, deposits split along the chord
        _transport("ct_sobp_chord_1m", "ct", 1_000_000, nx=120, ny=120, nz=240, n_spots=256, chord=True),
        # the two extensions of the model together: energy-dependent cut-off and secondary protons
        _transport("insert_cut_branching_300k", "insert", 300_000, cut=2.5, secondaries=0.6),
        # a treatment plan in one launch: 2000 spots in 12 million voxels, spots resident on the device
        _transport("plan_2000_spots_30m", "spheres", 30_000_000, nx=200, ny=200, nz=300, n_spots=2000, e_lo=70.0,
                   e_hi=200.0, sigma=0.0, resident=True),
        # a full-resolution layer of the denoiser
        _conv("conv_full_32_32", 1, 192, 128, 128, 32, 32),
        # a volume of no round size, two samples, FP32 results (as a data gradient is checked)
        _conv("conv_ragged_48_80", 2, 37, 51, 75, 48, 80, relu=False, fp32=True),
        # the weight gradient of the full-resolution layer
        dict(name="wgrad_full_32_32", kind="wgrad", n=1, d=192, h=128, w=128, cin=32, cout=32),
        # one inference of the trained network on the volume it was trained for
        dict(name="infer_192_128_128", kind="infer", n=1, d=192, h=128, w=128),
        # one Adam step of its training on the same volume
        dict(name="train_step_192_128_128", kind="train", n=1, d=192, h=128, w=128),
        # a low-history dose judged against the high-history one, 2 %/0.5 mm
        dict(name="gamma_192_128_128", kind="gamma", d=192, h=128, w=128, noise=0.02, dta=0.5, steps=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["transport", "transport", "transport", "transport", "conv", "conv", "wgrad", "infer", "train",
                       "gamma"])
    if kind == "transport":
        phantom = rng.choice(["water", "slab", "insert", "spheres", "spheres", "ct"])
        c = _transport(None, phantom, 0, sigma=rng.choice([0.0, 3.0, round(rng.uniform(1.0, 6.0), 1)]))
        del c["name"]
        if phantom == "spheres":
            c.update(nx=rng.randint(33, 200), ny=rng.randint(33, 200), nz=rng.randint(97, 300), n_spots=_log(rng, 1, 2000))
        elif phantom == "ct":
            c.update(nx=rng.randint(60, 120), ny=rng.randint(60, 120), nz=rng.randint(180, 240), n_spots=256)
        c["e_lo"] = round(rng.uniform(70.0, 160.0), 1)
        c["e_hi"] = round(c["e_lo"] + rng.uniform(0.0, 40.0), 1) if phantom == "spheres" else c["e_lo"]
        c["chord"] = rng.random() < 0.25
        c["cut"] = rng.choice([0.0, 0.0, 0.0, 2.5, round(rng.uniform(2.0, 4.0), 2)])
        c["secondaries"] = rng.choice([0.0, 0.0, 0.0, round(rng.uniform(0.2, 1.0), 2)])
        c["resident"] = rng.random() < 0.3
        c["fetch"] = rng.choice(["device", "device", "host", "f32"])
        c["histories"] = _log(rng, 10_000, 1_000_000 if c["cut"] or c["secondaries"] else 10_000_000)
        return c
    if kind in ("conv", "wgrad"):
        cin, cout = 16 * rng.randint(1, 12), 16 * rng.randint(1, 8)
        w = rng.choice([rng.randint(16, 128), rng.choice([32, 64, 128, 256])])
        h = rng.randint(8, 128)
        # as many planes as keep the layer below the full-resolution 96 -> 32 one
        top = max(4, min(192, int(192 * 128 * 128 * 64 * 32 / (w * h * cin * cout))))
        d = max(2, _log(rng, 4, top))
        n = 2 if d <= 24 and rng.random() < 0.4 else 1
        if kind == "wgrad":  # up to the network's own row width
            return dict(kind="wgrad", n=n, d=d, h=h, w=min(w, 128), cin=cin, cout=cout)
        c = _conv(None, n, d, h, w, cin, cout, relu=rng.random() < 0.6, fp32=rng.random() < 0.4, bias=rng.random() < 0.8)
        del c["name"]
        return c
    d, h, w = 4 * rng.randint(6, 48), 4 * rng.randint(6, 32), 4 * rng.randint(6, 32)
    if kind == "gamma":
        return dict(kind="gamma", d=d + rng.randint(0, 3), h=h + rng.randint(0, 3) - 3, w=w + rng.randint(0, 3) - 3,
                    noise=round(rng.uniform(0.008, 0.03), 3), dta=rng.choice([0.5, 1.0, 2.0]), steps=rng.choice([5, 10]))
    return dict(kind=kind, n=2 if d * h * w < 400_000 and rng.random() < 0.4 else 1, d=d, h=h, w=w)


# ----------------------------------------------------------------------- phantoms and plans
def _workload(c, seed):
    """The phantom (of `seed` where it is drawn) and its spots, host arrays."""
    n, E = c["histories"], c["e_lo"]
    if c["phantom"] == "water":
        wl = W.water100(n)
    elif c["phantom"] == "slab":
        wl = W.slab150(n)
    elif c["phantom"] == "insert":
        wl = W.insert150(n)
    elif c["phantom"] == "ct":
        return W.ct_sobp(n, seed=seed % 100_003, shape=(c["nx"], c["ny"], c["nz"]), h=c["h"])
    else:
        shape = (c["nx"], c["ny"], c["nz"])
        origin, dens, mid = W.sphere_phantom(shape, c["h"], seed % 100_003, r_range=(5.0, 15.0 if c["nx"] <= 128 else 25.0))
        half = 30.0 if c["n_spots"] <= 144 else 0.5 * min(c["nx"], c["ny"]) * c["h"]
        half = min(half, 0.5 * min(c["nx"], c["ny"]) * c["h"])
        spots = W.plan_spots(c["n_spots"], n, seed % 100_003, (E, c["e_hi"]), 5.0, half)
        spots["sigma_xy_mm"] = c["sigma"]
        return W.Workload("spheres", shape, (c["h"],) * 3, origin, dens, mid, [W.WATER, W.TISSUE, W.BONE], spots)
    wl.spots = W.pencil(E, n, sigma_xy=c["sigma"])
    return wl


def _prepare_transport(c, seed):
    wl = _workload(c, seed)
    d = S.SdeDose(wl, tally_mode=int(c["chord"]), theta_cut_sigmas=c["cut"], secondary_fraction=c["secondaries"])
    nx, ny, nz = wl.shape
    s = dict(d=d, spots=wl.spots, seed=seed * 2 + 1)
    if c["resident"]:
        s["d_spots"] = torch.from_numpy(wl.spots.view(np.uint8).copy()).cuda()
    if c["fetch"] == "f32":
        s["dose"] = torch.empty(nz, ny, nx, dtype=torch.float32, device="cuda")
    elif c["fetch"] == "device":
        s["dose"] = torch.empty(nz, ny, nx, dtype=torch.float64, device="cuda")
        s["edep"] = torch.empty(nz, ny, nx, dtype=torch.int64, device="cuda")
    return s


def _run_transport(c, s):
    d = s["d"]
    d.reset()
    if "d_spots" in s:
        d.run_device(s["d_spots"].data_ptr(), len(s["spots"]), s["seed"])
    else:
        d.run(s["spots"], s["seed"])
    if c["fetch"] == "f32":  # what the denoiser takes; asynchronous
        return {"dose": d.dose_into(s["dose"])}
    if c["fetch"] == "device":
        bal = d.fetch_device(s["dose"].data_ptr(), s["edep"].data_ptr(), balance=True)
        return {"dose": s["dose"], "edep": s["edep"], **bal}
    dose, edep, bal = d.fetch()
    return {"dose": dose, "edep": edep.view(np.int64), **bal}


# ------------------------------------------------------------------------------ convolutions
def _conv_inputs(c, seed):
    """Activations and weights of a trained network's size, channels-last."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(c["n"], c["d"], c["h"], c["w"], c["cin"], device="cuda", generator=g)
    x = (0.5 * F.leaky_relu(x, 0.1)).to(torch.bfloat16)
    w = (torch.randn(c["cout"], 27, c["cin"], device="cuda", generator=g) * (27 * c["cin"]) ** -0.5).to(torch.bfloat16)
    b = 0.1 * torch.randn(c["cout"], device="cuda", generator=g)
    return x, w, b


def _prepare_conv(c, seed):
    x, w, b = _conv_inputs(c, seed)
    y = (torch.empty(c["n"], c["d"], c["h"], c["w"], c["cout"], device="cuda") if c["fp32"]
         else S.pcg_zeros(c["n"], c["cout"], c["d"], c["h"], c["w"]))
    return dict(x=S.to_pcg(x), w=w, b=b if c["bias"] else None, y=y)


def _wgrad_inputs(c, seed):
    x, w, b = _conv_inputs(c, seed)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    dy = (0.1 * torch.randn(c["n"], c["d"], c["h"], c["w"], c["cout"], device="cuda", generator=g)).to(torch.bfloat16)
    return x, dy


def _prepare_wgrad(c, seed):
    x, dy = _wgrad_inputs(c, seed)
    return dict(x=S.to_pcg(x), dy=S.to_pcg(dy), dw=torch.zeros(c["cout"], 27, c["cin"], device="cuda"))


# ------------------------------------------------------------------- doses and the denoiser
def _doses(c, seed, noise=0.1):
    """A dose as the transport leaves it: pencil beams with a Bragg curve of their own, counted
    with Poisson noise (relative `noise` at the maximum), the same with a hundredth of its
    variance, and a density map of water with spheres."""
    n, D, H, Wd = c.get("n", 1), c["d"], c["h"], c["w"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(64, generator=torch.Generator().manual_seed(seed)).tolist()
    z = torch.arange(D, device="cuda").view(D, 1, 1) + 0.5
    y = torch.arange(H, device="cuda").view(1, H, 1) + 0.5
    x = torch.arange(Wd, device="cuda").view(1, 1, Wd) + 0.5
    base = torch.zeros(D, H, Wd, device="cuda")
    for k in range(12):
        a, b, r, w = u[4 * k:4 * k + 4]
        R = (0.4 + 0.55 * r) * D
        s2 = (3.0 + 2.0 * z / D) ** 2
        curve = torch.where(z < R, (R - z + 1.0).clamp(min=1.0) ** -0.435, torch.zeros_like(z))
        spot = torch.exp(-((x - (0.3 + 0.4 * a) * Wd) ** 2 + (y - (0.3 + 0.4 * b) * H) ** 2) / (2 * s2)) / s2
        base += (0.3 + w) * curve * spot
    rho = torch.ones(D, H, Wd, device="cuda")
    for k in range(4):
        a, b, e, r = u[48 + 4 * k:52 + 4 * k]
        inside = (x - a * Wd) ** 2 + (y - b * H) ** 2 + (z - e * D) ** 2 < (0.05 + 0.1 * r) ** 2 * D * D
        rho[inside] = 0.2 + 1.7 * b
    base = (base / base.max()).repeat(n, 1, 1, 1)
    k = noise ** -2
    low = torch.poisson(base * k, generator=g) / k
    high = torch.poisson(base * (100 * k), generator=g) / k
    return 1e-4 * low, rho, 1e-4 * high  # high: a hundred times the histories


def _weights():
    return np.load(os.path.join(os.path.dirname(S.__file__), "weights", "denoiser_128x128x192.npy")).astype(np.float32)


def _prepare_net(c, seed):
    low, rho, high = _doses(c, seed)
    net = S.Denoiser(c["d"], c["h"], c["w"], batch_max=c["n"], seed=1)
    net.set_params(_weights())
    return dict(net=net, low=low, rho=rho, high=high, out=torch.empty_like(low))


LR = 1e-5  # within the schedule of a fine-tuning run


def _run_train(s):
    loss = s["net"].train_step(s["low"], s["rho"], s["high"], lr=LR, target_scale=0.01)
    return {"loss": loss, "params": s["net"].get_params()}


def _prepare_gamma(c, seed):
    low, rho, high = _doses(c, seed, noise=c["noise"])
    return dict(ref=(0.01 * high[0]).contiguous(), ev=low[0].contiguous())


# -------------------------------------------------------------------------------- the passes
def prepare(case, seed):
    torch.cuda.init()
    make = {"transport": _prepare_transport, "conv": _prepare_conv, "wgrad": _prepare_wgrad, "infer": _prepare_net,
            "train": _prepare_net, "gamma": _prepare_gamma}[case["kind"]]
    return dict(make(case, seed), case=case)


def run(state):
    c, s = state["case"], state
    if c["kind"] == "transport":
        return _run_transport(c, s)
    if c["kind"] == "conv":
        return S.conv3d(s["x"], s["w"], s["b"], relu=c["relu"], y=s["y"], fp32=c["fp32"])
    if c["kind"] == "wgrad":  # the call adds to dw, as a step with several micro-batches does
        s["dw"].zero_()
        return S.conv3d_wgrad(s["x"], s["dy"], s["dw"])
    if c["kind"] == "infer":
        return s["net"].infer(s["low"], s["rho"], s["out"])
    if c["kind"] == "train":
        return _run_train(s)
    return S.gamma3d(s["ref"], s["ev"], (1.0, 1.0, 1.0), dd=0.02, dta_mm=c["dta"], steps=c["steps"])


# ------------------------------------------------------------------------------- needed work
# (Cin, Cout, level) of the network's layers; two of the first layer's input channels are live, one
# output channel of the last.
LAYERS = [(16, 32, 0), (32, 32, 0), (32, 64, 1), (64, 64, 1), (64, 128, 2), (128, 128, 2), (192, 64, 1), (64, 64, 1),
          (96, 32, 0), (32, 32, 0), (32, 16, 0)]
OPS_PER_STEP = 200  # arithmetic of one Euler step: random block, tables, energy, direction, position, tally


def work(case):
    c = case
    if c["kind"] == "transport":
        nx, ny, nz, h = {"water": (40, 40, 120, 1.0), "slab": (120, 120, 400, 0.5), "insert": (80, 80, 200, 1.0)}.get(
            c["phantom"], (c["nx"], c["ny"], c["nz"], c["h"]))
        E = 130.0 if c["phantom"] == "ct" else 0.5 * (c["e_lo"] + c["e_hi"])
        steps = min(10 * 0.0022 * E ** 1.77, nz * h) / 0.5  # half-millimetre steps over the range in water
        per_voxel = 8 + 4 + 4 + {"f32": 8 + 4, "device": 8 + 8 + 8, "host": 8 + 8 + 8}[c["fetch"]]
        return {"bytes": nx * ny * nz * per_voxel, "flops": c["histories"] * steps * OPS_PER_STEP}
    v = c["d"] * c["h"] * c["w"] * c.get("n", 1)
    if c["kind"] in ("conv", "wgrad"):
        out = 27 * c["cin"] * c["cout"] * 4 if c["kind"] == "wgrad" else v * c["cout"] * (4 if c["fp32"] else 2)
        read = v * 2 * (c["cin"] + (c["cout"] if c["kind"] == "wgrad" else 0))
        return {"bytes": read + out, "flops": 2.0 * v * 27 * c["cin"] * c["cout"]}
    if c["kind"] == "gamma":  # every voxel of both grids once
        return {"bytes": 8 * v, "flops": 8 * v}
    flops = 2.0 * v * sum(27 * ci * co / 8 ** lv for ci, co, lv in LAYERS[1:-1]) + 2.0 * v * 27 * (2 * 32 + 32)
    if c["kind"] == "infer":  # dose and density in, dose out; every activation stays on chip
        return {"bytes": 12 * v, "flops": flops}
    n_par = sum(27 * ci * co + co for ci, co, _ in LAYERS)
    # activations are kept for the backward pass: written once, read once
    acts = 2 * v * sum(co / 8 ** lv for _, co, lv in LAYERS[:-1])
    return {"bytes": 16 * v + 2 * acts + n_par * 28, "flops": 3 * flops}


# ----------------------------------------------------------------- the same in 64 bits, plainly
def _conv64(x, w):
    """3x3x3 convolution of channels-last x by w [Cout, 27, Cin]: 27 shifted products."""
    n, D, H, Wd, _ = x.shape
    xp = F.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    y = torch.zeros(n, D, H, Wd, w.shape[0], dtype=x.dtype, device=x.device)
    for t in range(27):
        kz, ky, kx = t // 9, t // 3 % 3, t % 3
        y += xp[:, kz:kz + D, ky:ky + H, kx:kx + Wd] @ w[:, t].T
    return y


def _wgrad64(x, dy):
    n, D, H, Wd, ci = x.shape
    xp = F.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    d2 = dy.reshape(-1, dy.shape[-1]).T
    return torch.stack([d2 @ xp[:, t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + Wd].reshape(-1, ci)
                        for t in range(27)], 1)


class _Conv(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, w):
        ctx.save_for_backward(x, w)
        return _conv64(x, w)

    @staticmethod
    def backward(ctx, dy):
        x, w = ctx.saved_tensors
        dx = _conv64(dy, w.flip(1).permute(2, 1, 0)) if ctx.needs_input_grad[0] else None
        return dx, _wgrad64(x, dy)


def _grouped(y):
    """Channels-last to [n, C/8, D+2, H+2, W+2, 8] with a zero border."""
    n, D, H, Wd, C = y.shape
    return F.pad(y.reshape(n, D, H, Wd, C // 8, 8).permute(0, 4, 1, 2, 3, 5), (0, 0, 1, 1, 1, 1, 1, 1))


def _split(p):
    out, o = [], 0
    for ci, co, _ in LAYERS:
        k = co * 27 * ci
        out.append((p[o:o + k].view(co, 27, ci), p[o + k:o + k + co]))
        o += k + co
    return out


def _net64(params, low, rho):
    """The denoiser's prediction over the dose scale, and the scale of each sample."""
    L = _split(params)
    s = 1.0 / low.abs().amax(dim=(1, 2, 3), keepdim=True)
    first = torch.stack([low * s, (0.5 * rho).expand_as(low)], -1)

    def conv(t, i):
        w, b = L[i]
        w = w[:, :, :2] if i == 0 else w[:1] if i == 10 else w  # the live channels
        y = _Conv.apply(t, w) + b[:w.shape[0]]
        return F.leaky_relu(y, 0.1) if i < 10 else y

    def pool(t):
        n, D, H, Wd, C = t.shape
        return t.view(n, D // 2, 2, H // 2, 2, Wd // 2, 2, C).mean(dim=(2, 4, 6))

    def up(t):
        n, D, H, Wd, C = t.shape
        return t.view(n, D, 1, H, 1, Wd, 1, C).expand(n, D, 2, H, 2, Wd, 2, C).reshape(n, 2 * D, 2 * H, 2 * Wd, C)

    e1 = conv(conv(first, 0), 1)
    e2 = conv(conv(pool(e1), 2), 3)
    b2 = conv(conv(pool(e2), 4), 5)
    d2 = conv(conv(torch.cat([up(b2), e2], -1), 6), 7)
    d1 = conv(conv(torch.cat([up(d2), e1], -1), 8), 9)
    return low * s + conv(d1, 10)[..., 0], s


def _gamma64(ref, ev, dta, steps, dd=0.02, threshold=0.01):
    """Pass rate of the local gamma index: some position of a grid of step dta/steps within dta of
    the voxel (trilinear interpolation, clamped to the volume) agrees."""
    D, H, Wd = ref.shape
    at = torch.nonzero((ref >= threshold * ref.max()) & (ref > 0))
    n = len(at)
    r = ref[at[:, 0], at[:, 1], at[:, 2]]
    left = (ev[at[:, 0], at[:, 1], at[:, 2]] - r).abs() > dd * r
    at, r = at[left].double(), r[left]
    hi = torch.tensor([D - 1, H - 1, Wd - 1], device=ref.device, dtype=torch.float64)
    o = torch.arange(-steps, steps + 1, dtype=torch.float64) / steps
    offs = torch.cartesian_prod(o, o, o)
    d2s = (offs ** 2).sum(1)
    keep = d2s <= 1.0 + 1e-9
    order = torch.argsort(d2s[keep])
    flat = ev.reshape(-1)
    for off, d2 in zip((offs[keep][order] * dta).to(ref.device), d2s[keep][order].tolist()):
        p = torch.minimum((at + off).clamp(min=0.0), hi)
        i0 = torch.minimum(p.floor(), (hi - 1).clamp(min=0.0))
        f = p - i0
        i0, i1 = i0.long(), torch.minimum(i0 + 1, hi).long()
        e = 0.0
        for b in range(8):
            q = [i1[:, a] if b >> a & 1 else i0[:, a] for a in range(3)]
            wt = [f[:, a] if b >> a & 1 else 1 - f[:, a] for a in range(3)]
            e = e + flat[(q[0] * H + q[1]) * Wd + q[2]] * (wt[0] * wt[1] * wt[2])
        bad = d2 + ((e - r) / (dd * r)) ** 2 > 1.0
        at, r = at[bad], r[bad]
        if not len(r):
            break
    return 1.0 - len(r) / max(n, 1)


def exact(case, seed):
    c = case
    if c["kind"] == "transport":
        return None  # histories are random walks: there is no closed value
    with torch.no_grad():
        if c["kind"] == "conv":
            x, w, b = _conv_inputs(c, seed)
            y = _conv64(x.double(), w.double())
            y = y + b.double() if c["bias"] else y
            y = y.clamp(min=0) if c["relu"] else y
            return y if c["fp32"] else _grouped(y)
        if c["kind"] == "wgrad":
            x, dy = _wgrad_inputs(c, seed)
            return _wgrad64(x.double(), dy.double())
        if c["kind"] == "gamma":
            s = _prepare_gamma(c, seed)
            return _gamma64(s["ref"].double(), s["ev"].double(), c["dta"], c["steps"])
        low, rho, high = (t.double() for t in _doses(c, seed))
        p = torch.from_numpy(_weights()).cuda().double()
        if c["kind"] == "infer":
            pred, s = _net64(p, low, rho)
            return pred / s
    p.requires_grad_(True)
    pred, s = _net64(p, low, rho)
    t = high * 0.01 * s
    err = (pred - t) ** 2 / (t.abs() + 0.05)
    err.sum().backward()
    with torch.no_grad():  # Adam's first step: m / (1 - b1) = g, v / (1 - b2) = g^2
        return {"loss": float(err.mean()), "params": p - LR * p.grad / (p.grad.abs() + 1e-8)}
