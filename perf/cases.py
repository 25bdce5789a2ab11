"""Performance cases of the library: the calls a user's program makes, over the sizes they are made at.

A case is a plain dict; `prepare` builds what the program holds before the call (scene handle, network,
carried state, log frames on the GPU), `run` makes one pass through the public entry points of
paper_2508_18071_gb300 (api.render_frames, api.threshold_events, api.evsnet_forward and the training calls)
and returns everything the pass computes.  `exact` restates the networks, the threshold model and the
training gradients in 64-bit torch.

Kinds:
  render     frames of a camera path through a scene (Cornell box, procedural scene, city block)
  threshold  contrast-threshold events of log frames, the reference and the training target
  evsnet     the spiking network on log frames of a video in progress, state carried in
  train      forward, EMD + count loss and backward of one batch of clips
"""
import functools
import math
import os

import numpy as np
import torch

from paper_2508_18071_gb300 import _lib as L
from paper_2508_18071_gb300 import api, inputs, train_evsnet, training

DTYPES = {"f32": L.ET_F32, "bf16": L.ET_BF16, "fp8": L.ET_FP8}
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(train_evsnet.__file__)), "weights")
TRAINED = {"stem": "evsnet_city.npz", "temporal": "evsnet_city_temporal.npz", "conv3": "evsnet_city_spatial.npz"}
C_THR = 0.2           # contrast threshold of the reference events
EVENT_RATE = 0.04     # reference events per pixel and step on the city path
LAMBDA = 0.01         # count-loss weight of the trainer
CKPT = 16             # membrane checkpoint interval of the trainer


def listed():
    return [
        # The tiny configuration (32 triangles, 64 x 64): latency and launches, as in a preview or a unit test.
        {"name": "render_cornell", "kind": "render", "scene": "cornell", "boxes": 0, "W": 64, "H": 64, "frames": 8,
         "spp": 4, "depth": 4, "rgb": True},
        # The rotating-camera configuration (20k triangles, 256 x 256, 4 SPP): one chunk of a training clip.
        {"name": "render_procedural", "kind": "render", "scene": "random", "boxes": 200, "W": 256, "H": 256,
         "frames": 16, "spp": 4, "depth": 5, "rgb": True},
        # The benchmark's frames (500k triangles, 720p, 2 SPP, depth 5): log luminance only, for the event stage.
        {"name": "render_city", "kind": "render", "scene": "city", "boxes": 40000, "W": 1280, "H": 720, "frames": 4,
         "spp": 2, "depth": 5, "rgb": False},
        # Reference events of high-SPP 720p frames (the noise left at 256 SPP is well below the threshold).
        {"name": "threshold_720p", "kind": "threshold", "W": 1280, "H": 720, "frames": 25, "noise": 0.05},
        # The benchmark's event stage: trained stem network in BF16 on low-SPP 720p frames.
        {"name": "evsnet_stem_bf16", "kind": "evsnet", "form": "stem", "net": "trained", "dtype": "bf16", "W": 1280,
         "H": 720, "frames": 25, "noise": 0.7},
        # The same network in FP8 with calibrated scales on a small frame with ragged tiles.
        {"name": "evsnet_stem_fp8", "kind": "evsnet", "form": "stem", "net": "trained", "dtype": "fp8", "W": 253,
         "H": 187, "frames": 16, "noise": 0.7},
        # The 3x3 stack of the workload configurations in BF16 at 720p.
        {"name": "evsnet_conv3_bf16", "kind": "evsnet", "form": "conv3", "net": "trained", "dtype": "bf16", "W": 1280,
         "H": 720, "frames": 25, "noise": 0.7},
        # Its FP32 path (the parity path), odd frame size.
        {"name": "evsnet_conv3_f32", "kind": "evsnet", "form": "conv3", "net": "trained", "dtype": "f32", "W": 641,
         "H": 363, "frames": 16, "noise": 0.7},
        # The paper's pixel-wise temporal form in FP32.
        {"name": "evsnet_temporal_f32", "kind": "evsnet", "form": "temporal", "net": "trained", "dtype": "f32",
         "W": 640, "H": 360, "frames": 16, "noise": 0.7},
        # Training: the 3x3 stack in FP32 on a small batch of odd-sized clips.
        {"name": "train_conv3_f32", "kind": "train", "form": "conv3", "net": "trained", "dtype": "f32", "B": 2,
         "K": 50, "W": 93, "H": 67, "noise": 0.7},
        # Training: the temporal form in FP32, half a workload batch.
        {"name": "train_temporal_f32", "kind": "train", "form": "temporal", "net": "trained", "dtype": "f32", "B": 4,
         "K": 64, "W": 128, "H": 128, "noise": 0.7},
        # Training: the city form (stem + temporal blocks) with BF16 convolutions at the workload's batch.
        {"name": "train_stem_bf16", "kind": "train", "form": "stem", "net": "trained", "dtype": "bf16", "B": 8,
         "K": 64, "W": 128, "H": 128, "noise": 0.7},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "threshold", "evsnet", "evsnet", "evsnet", "evsnet", "train",
                       "train", "train"])
    if kind == "render":
        scene = rng.choice(["cornell", "random", "city"])
        boxes = {"cornell": 0, "random": rng.choice([60, 200]), "city": rng.choice([4000, 12000])}[scene]
        c = {"kind": kind, "scene": scene, "boxes": boxes, "W": _logint(rng, 48, 1280), "H": _logint(rng, 36, 720),
             "frames": 0, "spp": rng.choice([1, 2, 3, 4, 8]), "depth": rng.choice([3, 4, 5]),
             "rgb": rng.random() < 0.5}
        paths = c["W"] * c["H"] * c["spp"]
        c["frames"] = max(1, min(_logint(rng, 1, 32), 1280 * 720 * 8 // paths))
        c["spp"] = min(c["spp"], max(1, 1280 * 720 * 8 // (c["W"] * c["H"])))
        return c
    if kind == "threshold":
        return {"kind": kind, "W": _logint(rng, 33, 1280), "H": _logint(rng, 25, 720), "frames": rng.randint(2, 25),
                "noise": rng.choice([0.02, 0.05, 0.2])}
    form = rng.choice(["stem", "temporal", "conv3"])
    net = rng.choice(["trained", "random"])
    if kind == "evsnet":
        return {"kind": kind, "form": form, "net": net, "dtype": rng.choice(["f32", "bf16", "fp8"]),
                "W": _logint(rng, 45, 1280), "H": _logint(rng, 37, 720), "frames": rng.randint(2, 25), "noise": 0.7}
    c = {"kind": kind, "form": form, "net": net, "dtype": rng.choice(["f32", "bf16"]), "B": rng.randint(1, 8),
         "K": rng.randint(8, 64), "W": _logint(rng, 20, 128), "H": _logint(rng, 18, 128), "noise": 0.7}
    if c["dtype"] == "f32":
        c["B"] = min(c["B"], 4)   # an FP32 step costs more than twice a BF16 one
    return c


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _scene(name, boxes):
    """Host geometry of a scene (an asset on disk in a user's program), made once per process."""
    if name == "cornell":
        return inputs.cornell_box()
    if name == "random":
        return inputs.random_scene(n_boxes=boxes // 2, n_spheres=boxes - boxes // 2)
    return inputs.city_block(n_boxes=boxes)


def _path(name, frames, first):
    if name == "cornell":
        return inputs.cornell_path(frames, first=first % 64)
    if name == "random":
        return inputs.random_scene_path(frames, first=first)
    return inputs.city_path(frames, first=first)


def _network(case, seed):
    form = case["form"]
    if case["net"] == "trained":
        return train_evsnet.load(os.path.join(WEIGHTS, TRAINED[form]))
    if form == "conv3":
        return inputs.random_evsnet(0, 4, 16, 1, 3, seed=seed, vth=0.5, beta=0.9)
    return inputs.random_evsnet(1, 7, 16, 7, 1, seed=seed, vth=0.5, beta=0.9, ks0=3 if form == "stem" else 0)


def _clip(gen, B, F, H, W, noise):
    """Log frames [B, F, H, W]: a smooth image that drifts, per-pixel steps, and Monte Carlo noise that is
    independent from frame to frame (about 0.7 log units at 2 SPP, 0.05 at 256)."""
    dev = "cuda"
    base = torch.randn((B, 1, max(2, H // 16), max(2, W // 16)), generator=gen, device=dev)
    drift = torch.randn((B, 1, max(2, H // 16), max(2, W // 16)), generator=gen, device=dev)
    up = functools.partial(torch.nn.functional.interpolate, size=(H, W), mode="bilinear", align_corners=False)
    t = torch.arange(F, device=dev, dtype=torch.float32).view(1, F, 1, 1)
    l = up(base) * 0.5 - 1.0 + up(drift) * (0.03 * t)
    return (l + noise * torch.randn((B, F, H, W), generator=gen, device=dev)).contiguous()


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _evsnet_frames(case, seed):
    """(frame before the call [H, W], frames of the call [F, H, W], calibration clip [9, H, W])."""
    l = _clip(_generator(seed), 1, case["frames"] + 10, case["H"], case["W"], case["noise"])[0]
    return l[9], l[10:].contiguous(), l[:9].contiguous()


def _train_batch(case, seed):
    """Log frames [B, K + 1, H, W] and signed target counts [B, K, H, W] at the reference's event rate."""
    gen = _generator(seed)
    B, K, H, W = case["B"], case["K"], case["H"], case["W"]
    logl = _clip(gen, B, K + 1, H, W, case["noise"])
    u = torch.rand((B, K, H, W), generator=gen, device="cuda")
    return logl, (u < EVENT_RATE / 2).float() - (u > 1 - EVENT_RATE / 2).float()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "render":
        first = seed % 900
        shape = (case["frames"], case["H"], case["W"])
        return {"case": case, "scene": api.Scene(_scene(case["scene"], case["boxes"])),
                "cams": _path(case["scene"], case["frames"], first), "first": first, "seed": seed,
                "rgb": torch.empty(shape + (3,), device="cuda") if case["rgb"] else None,
                "logl": torch.empty(shape, device="cuda")}
    if kind == "threshold":
        F, H, W = case["frames"], case["H"], case["W"]
        logl = _clip(_generator(seed), 1, F + 1, H, W, case["noise"])[0]
        return {"case": case, "logl": logl[1:].contiguous(), "ref": logl[0].double().reshape(-1).contiguous(),
                "buf": api.EventBuffer(F * H * W)}
    d = _network(case, seed)
    net = api.EvsNetDev.from_dict(d, DTYPES[case["dtype"]])
    if kind == "train":
        logl, E = _train_batch(case, seed)
        return {"case": case, "net": net, "logl": logl, "E": E}
    before, logl, calibration = _evsnet_frames(case, seed)
    if case["dtype"] == "fp8" and net.ks == 1:
        b16 = api.EvsNetDev.from_dict(d, L.ET_BF16)
        net.scales = api.evsnet_fp8_scales(calibration, b16, api.EvsStateDev(b16, case["H"], case["W"]))
    state = api.EvsStateDev(net, case["H"], case["W"])
    state.last_l.copy_(before.reshape(-1))
    state.initialized = 1
    return {"case": case, "net": net, "state": state, "logl": logl,
            "buf": api.EventBuffer(case["frames"] * case["H"] * case["W"])}


# -------------------------------------------------------------------- passes
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "render":
        rgb, logl, _ = api.render_frames(state["scene"], state["cams"], case["W"], case["H"], case["spp"],
                                         case["depth"], state["seed"], first_frame=state["first"], rgb=state["rgb"],
                                         logl=state["logl"], want_rgb=case["rgb"])
        return {"rgb": rgb, "logl": logl}
    if kind == "threshold":
        buf = api.threshold_events(state["logl"], C_THR, state["ref"], True, t0=1, buf=state["buf"])
        return {"ref": state["ref"], "events": buf.count}
    if kind == "evsnet":
        st = state["state"]
        buf, I, spikes = api.evsnet_forward(state["logl"], state["net"], st, t0=1, buf=state["buf"], want_I=True,
                                            want_spikes=True)
        return {"I": I, "spikes": spikes, "V": st.V, "hist": st.hist if state["net"].kt > 1 else None,
                "last_l": st.last_l, "events": buf.count}
    net = state["net"]
    out = training.train_forward(state["logl"], net, net.w, net.b, ckpt_every=CKPT, want_S=False)
    loss, dS_on, dS_off = training.emd_count_loss(out["spikes"], state["E"], LAMBDA)
    gw, gb = training.train_backward(state["logl"], net, net.w, net.b, out["V_ckpt"], dS_on, dS_off, ckpt_every=CKPT)
    return {"loss": loss, "grad_w": gw, "grad_b": gb, "spikes": out["spikes"], "V_ckpt": out["V_ckpt"],
            "dS_on": dS_on, "dS_off": dS_off}


# ---------------------------------------------------------------------- work
def _macs(form):
    """Multiply-adds per pixel and step of the 16-channel networks."""
    if form == "conv3":
        return 9 * 16 + 3 * 9 * 256 + 16
    return (9 if form == "stem" else 7) * 16 + 6 * 7 * 256 + 16


def work(case):
    kind, npix = case["kind"], case["H"] * case["W"]
    if kind == "render":
        n_tris = len(_scene(case["scene"], case["boxes"])["tris"])
        pixels = npix * case["frames"]
        # rays per sample: 5 of the 2 depth - 1 at most on the city path; per ray about 60 flop for each
        # level of the hierarchy (24 per node visit, 40 per triangle test)
        rays = pixels * case["spp"] * 0.55 * (2 * case["depth"] - 1)
        return {"bytes": 36 * n_tris + (16 if case["rgb"] else 4) * pixels,
                "flops": rays * 60 * math.log2(max(2, n_tris))}
    if kind == "threshold":
        steps = npix * case["frames"]
        return {"bytes": 4 * steps + 16 * npix + 12 * EVENT_RATE * steps, "flops": 5 * steps}
    if kind == "evsnet":
        steps = npix * case["frames"]
        # frames in, current and spikes out, events, membrane and previous frame in and out
        nbytes = (4 + 4 + 1 + 12 * EVENT_RATE) * steps + 16 * npix
        if case["form"] != "conv3":    # past inputs of the temporal layers in and out
            nbytes += 2 * 4 * 6 * (6 * 16 + (1 if case["form"] == "temporal" else 0)) * npix
        return {"bytes": nbytes, "flops": 2 * _macs(case["form"]) * steps}
    steps = case["B"] * case["K"] * npix
    # log frames and targets in, spikes and both loss gradients out; forward, data and weight gradient
    return {"bytes": (4 + 4 + 1 + 8) * steps, "flops": 3 * 2 * _macs(case["form"]) * steps}


# ------------------------------------------------------------- 64-bit restatement
def _conv(x, w, b):
    """x [B, Ci, K, H, W], w [Co, Ci, kt, ks, ks]: causal along K, zero padding in space."""
    kt, ks = w.shape[2], w.shape[3]
    K, H, W = x.shape[2:]
    r = ks // 2
    xp = torch.nn.functional.pad(x, (r, r, r, r, kt - 1, 0))
    out = b.view(1, -1, 1, 1, 1)
    for t in range(kt):
        for dy in range(ks):
            for dx in range(ks):
                out = out + torch.einsum("oi,bikhw->bokhw", w[:, :, t, dy, dx],
                                         xp[:, :, t:t + K, dy:dy + H, dx:dx + W])
    return out


def _forward64(d, w, b, X):
    """Currents [B, K, H, W] and the input of every layer for X [B, K, H, W]."""
    C = d["C"]
    ins, off = [], 0
    x, h = X[:, None], None
    for i in range(d["n_layers"]):
        cin, kt, ks = inputs.layer_shape(d, i)
        n = C * cin * kt * ks * ks
        ins.append(x)
        z = _conv(x, w[off:off + n].view(C, cin, kt, ks, ks), b[i * C:(i + 1) * C])
        off += n
        closing = d["kind"] == L.ET_NET_RESIDUAL and i >= 2 and i % 2 == 0
        x = torch.relu(h + z) if closing else torch.relu(z)
        if closing or i == 0 or d["kind"] != L.ET_NET_RESIDUAL:
            h = x
    I = torch.einsum("c,bckhw->bkhw", w[off:off + C], x) + b[-1]
    return I, ins


class _Spike(torch.autograd.Function):
    """1(x >= 0) with the arctangent surrogate, alpha = 2."""

    @staticmethod
    def forward(ctx, x):
        ctx.save_for_backward(x)
        return (x >= 0).to(x.dtype)

    @staticmethod
    def backward(ctx, g):
        (x,) = ctx.saved_tensors
        return g / (1 + (math.pi * x) ** 2)


def _loss64(I, E, d):
    """EMD + count loss of the spike trains that the currents I drive."""
    V = torch.zeros_like(I[:, 0])
    on, off = [], []
    for k in range(I.shape[1]):
        vp = d["beta"] * V + I[:, k]
        on.append(_Spike.apply(vp - d["vth"]))
        off.append(_Spike.apply(-vp - d["vth"]))
        V = vp - d["reset"] * (on[-1] - off[-1])
    on, off = torch.stack(on, 1), torch.stack(off, 1)
    npx, K = I[:, 0].numel(), I.shape[1]
    emd = 0.0
    for s, e in ((on, E.clamp(min=0)), (off, (-E).clamp(min=0))):
        diff = s - e
        emd = emd + 0.5 / K * (diff.cumsum(1).abs().sum() + diff.flip(1).cumsum(1).abs().sum())
    count = (on.sum(1) + off.sum(1) - E.abs().sum(1)).abs().sum()
    return torch.stack([emd + LAMBDA * count, emd, count]) / npx


def exact(case, seed):
    kind = case["kind"]
    if kind == "render":
        return None     # path tracing at these sizes takes minutes in plain torch
    if kind == "threshold":
        l = _clip(_generator(seed), 1, case["frames"] + 1, case["H"], case["W"], case["noise"])[0].double()
        thr = float(np.float32(C_THR))
        ref = l[0].clone()
        for k in range(1, l.shape[0]):
            diff = l[k] - ref
            ref = ref + torch.sign(diff) * torch.floor(diff.abs() / thr) * thr
        return {"ref": ref.reshape(-1), "events": None}
    d = _network(case, seed)
    d = dict(d, **{k: float(np.float32(d[k])) for k in ("beta", "vth", "reset")})
    w = torch.as_tensor(np.asarray(d["w"], np.float64)).cuda()
    b = torch.as_tensor(np.asarray(d["b"], np.float64)).cuda()
    if kind == "evsnet":
        before, logl, _ = _evsnet_frames(case, seed)
        l = torch.cat([before[None], logl]).double()
        I, ins = _forward64(d, w, b, (l[1:] - l[:-1])[None])
        hist = None
        if d["kt"] > 1:
            n, hk, C = d["n_layers"], d["kt"] - 1, d["C"]
            hist = torch.zeros((n, hk, C, case["H"], case["W"]), dtype=torch.float64, device="cuda")
            keep = min(hk, case["frames"])
            for i in range(1 if d["ks0"] > 0 else 0, n):
                hist[i, hk - keep:, :ins[i].shape[1]] = ins[i][0, :, -keep:].transpose(0, 1)
            hist = hist.reshape(-1)
        # spikes and potentials follow from threshold decisions, which a rounding of the current can turn; the
        # currents of the FP8 networks differ from 64 bits by the rounding of their E4M3 operands (up to a third)
        return {"I": None if case["dtype"] == "fp8" else I[0], "hist": hist, "last_l": l[-1].reshape(-1)}
    logl, E = _train_batch(case, seed)
    l = logl.double()
    w.requires_grad_(True)
    b.requires_grad_(True)
    I, _ = _forward64(d, w, b, l[:, 1:] - l[:, :-1])
    loss = _loss64(I, E.double(), d)
    loss[0].backward()
    if case["dtype"] == "bf16":   # the gradients follow spikes that BF16 currents turn (a tenth of their norm)
        return {"loss": loss.detach(), "grad_w": None, "grad_b": None}
    return {"loss": loss.detach(), "grad_w": w.grad, "grad_b": b.grad}
