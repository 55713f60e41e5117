"""Performance cases: what programs built on this package have it compute, through its public
entry points, with a plain 64-bit torch evaluation of each to compare against.

Six kinds of work:
  das      one plan beamforming one acquisition held on the GPU (frames and Power Doppler);
  batch    many acquisitions of different sizes in one persistent launch;
  convert  acquisition-order IQ into the beamformer's layout and storage type;
  rf       real RF channel data demodulated into IQ;
  layer    one convolution layer of the compounding network, forward and backward;
  unet     the whole network: a prediction, or the loss and gradients of a training step.

Geometries and sizes are those of the package's own workloads (2D linear arrays at 0.3 mm pitch,
32 x 32 matrix arrays, grids of about 0.1 mm) and of its ragged batches (64-256 or 256-1024
elements, 128-384 pixels or 64-112 voxels a side, 1-48 frames, 1-15 plane waves) and sweeps
(up to 512 frames).
"""
import math
import os

import numpy as np
import torch

import paper_2604_06257_gb300 as mach
from paper_2604_06257_gb300 import learned, nn

C0 = 1540.0          # speed of sound, m/s
APOD = {"boxcar": 0, "hann": 1, "gauss": 2}


def listed():
    return [
        # B-mode of single acquisitions (three steered plane waves, 128 x 128 px): the smallest
        # call, as in a live view, where launch latency counts
        dict(name="bmode_1_frame", kind="das", array="linear", elems=128, tx=3, frames=1, nx=128, nz=128,
             samples=1152, dtype="c64", apod="hann", f_number=1.5, spread=5.0, step=0.28e-3),
        # the 2D Power Doppler benchmark: 256 x 256 px, 32 frames, split complex64 rows
        dict(name="doppler_32_frames", kind="das", array="linear", elems=128, tx=1, frames=32, nx=256, nz=256,
             samples=2048, dtype="c64split", apod="boxcar", f_number=1.0, spread=0.0, step=0.1e-3),
        # compounded Doppler from float16 storage, odd grid sides, an ensemble off the vector grid of 16
        dict(name="doppler_f16_20_frames", kind="das", array="linear", elems=192, tx=3, frames=20, nx=201, nz=233,
             samples=864, dtype="f16x2", apod="hann", f_number=1.5, spread=10.0, step=0.1e-3),
        # the rotating-disk grid of 251 x 251 px as plain complex64 with an odd ensemble
        dict(name="doppler_c64_25_frames", kind="das", array="linear", elems=128, tx=1, frames=25, nx=251, nz=251,
             samples=2048, dtype="c64", apod="boxcar", f_number=1.0, spread=0.0, step=0.1e-3),
        # functional-imaging ensembles of a few hundred frames
        dict(name="doppler_200_frames", kind="das", array="linear", elems=128, tx=1, frames=200, nx=192, nz=224,
             samples=1024, dtype="c64split", apod="boxcar", f_number=1.0, spread=0.0, step=0.1e-3),
        # the 3D localisation-microscopy volume (94 x 94 x 178 voxels, 1024 elements, 5 plane waves): the largest
        dict(name="volume_32_frames", kind="das", array="matrix", elems=1024, tx=5, frames=32, nx=94, ny=94, nz=178,
             samples=968, dtype="c64split", apod="gauss", f_number=1.0, spread=5.0, step=96e-6),
        # offline reconstruction of mixed 2D / 3D acquisitions stored as float16
        dict(name="ragged_batch_f16", kind="batch", count=10, shapes=11, scale=0.75, dtype="f16x2"),
        # scanner order to the beamformer's layout, for the odd ensemble above
        dict(name="convert_25_frames", kind="convert", tx=1, elems=128, samples=2048, frames=25, order="ftcs", dtype="c64"),
        # RF of the 2D benchmark (four times the IQ rate, 32 taps) into IQ
        dict(name="rf_32_frames", kind="rf", rows=128, samples=8189, frames=32, taps=32, decim=4),
        # one 32-channel layer of the network at half resolution, batch of 8, forward and backward
        dict(name="layer_32_to_32", kind="layer", ci=32, co=32, nx=64, ny=64, nz=64, batch=8),
        # the network's prediction for a batch of 8 volumes of 128^3
        dict(name="unet_predict", kind="unet", nx=128, ny=128, nz=128, batch=8, train=False),
        # loss and gradients of one training batch at the recipe's size
        dict(name="unet_gradients", kind="unet", nx=128, ny=128, nz=128, batch=8, train=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.55:
        if rng.random() < 0.7:
            case = dict(kind="das", array="linear", elems=_log(rng, 64, 256), tx=_log(rng, 1, 15), frames=_log(rng, 1, 256),
                        nx=_log(rng, 96, 384), nz=_log(rng, 96, 384), apod=rng.choice(["boxcar", "hann"]),
                        f_number=rng.choice([1.0, 1.5]), spread=10.0, step=0.1e-3)
            deepest = 10e-3 + case["nz"] * case["step"]
            case["samples"] = int(math.ceil(2.3 * deepest * 20.8e6 / C0)) + 32
            cap = 6e10
        else:
            case = dict(kind="das", array="matrix", elems=_log(rng, 16, 32) ** 2, tx=_log(rng, 1, 11),
                        frames=_log(rng, 1, 64), nx=_log(rng, 32, 96), ny=_log(rng, 32, 96), nz=_log(rng, 48, 128),
                        apod="gauss", f_number=1.0, spread=10.0, step=0.1e-3)
            deepest = 3e-3 + case["nz"] * case["step"]
            case["samples"] = int(math.ceil(2.3 * deepest * 31.2e6 / C0)) + 32
            cap = 6e10
        while _points(case) > cap and case["tx"] > 1:
            case["tx"] -= 1
        while _points(case) > cap:
            case["frames"] = max(1, case["frames"] * 3 // 4)
        types = ["c64", "f16x2", "bf16x2"]
        if case["frames"] % 4 == 0 and case["frames"] > 4:
            types += ["c64split"] * 3
        case["dtype"] = rng.choice(types)
        return case
    if u < 0.65:
        return dict(kind="batch", count=rng.randint(4, 10), shapes=rng.randint(1, 10 ** 6),
                    scale=round(rng.uniform(0.3, 0.7), 3), dtype=rng.choice(["f16x2", "f16x2", "bf16x2", "c64"]))
    if u < 0.75:
        frames = _log(rng, 1, 200)
        types = ["c64", "f16x2", "bf16x2"] + (["c64split"] if frames % 4 == 0 and frames > 4 else [])
        case = dict(kind="convert", tx=_log(rng, 1, 7), elems=_log(rng, 64, 256), samples=_log(rng, 512, 2048),
                    frames=frames, order=rng.choice(["ftcs", "ftcs", "ftcs", "tcsf"]), dtype=rng.choice(types))
        while case["tx"] * case["elems"] * case["samples"] * case["frames"] > 3e7 and case["frames"] > 1:
            case["frames"] = max(4, case["frames"] // 8 * 4) if case["dtype"] == "c64split" else case["frames"] // 2
            if case["frames"] <= 4 and case["dtype"] == "c64split":
                case.update(frames=8, tx=1)
                break
        return case
    if u < 0.85:
        decim = rng.choice([2, 3, 4, 5, 8])
        return dict(kind="rf", rows=_log(rng, 64, 256), samples=_log(rng, 1500, 8192), frames=_log(rng, 1, 64),
                    taps=rng.choice([16, 24, 31, 32, 48, 63]), decim=decim)
    if u < 0.93:
        ci, co = rng.choice([(16, 16), (48, 16), (32, 32), (96, 32), (64, 64), (192, 64), (128, 128)])
        top = {16: 96, 48: 96, 32: 64, 96: 64, 64: 32, 192: 32, 128: 24}[ci]
        return dict(kind="layer", ci=ci, co=co, nx=rng.randint(top // 3, top), ny=rng.randint(top // 3, top),
                    nz=rng.randint(top // 3, top), batch=rng.randint(1, 8))
    return dict(kind="unet", nx=8 * rng.randint(4, 12), ny=8 * rng.randint(4, 12), nz=8 * rng.randint(4, 12),
                batch=rng.randint(1, 6), train=rng.random() < 0.5)


# ---- geometry --------------------------------------------------------------------------------

def _geometry(case):
    """Keyword arguments of mach.Plan (everything but the storage type)."""
    step = case["step"]
    T, tilt = case["tx"], math.radians(case["spread"])
    ang = np.zeros((T, 2))
    ang[:, 0] = np.linspace(-tilt, tilt, T) if T > 1 else 0.0
    if case["array"] == "linear":
        n = case["elems"]
        e = np.zeros((n, 3))
        e[:, 0] = (np.arange(n) - (n - 1) / 2.0) * 0.3e-3
        nx, nz, z0 = case["nx"], case["nz"], case.get("z0", 10e-3 if case["apod"] == "boxcar" else 5e-3)
        return dict(ndim=2, elem_pos=e.astype(np.float32), tx_angles=ang, fs=20.8e6, fc=5.2e6, c=C0, t0=0.0,
                    f_number=case["f_number"], apod=case["apod"], n_samples=case["samples"], n_frames=case["frames"],
                    grid_dims=(nx, 1, nz), grid_origin=(-(nx - 1) * step / 2, 0.0, z0), grid_step=(step, 0.0, step))
    n = int(round(math.sqrt(case["elems"])))
    j, i = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    e = np.stack([(i.ravel() - (n - 1) / 2.0) * 0.3e-3, (j.ravel() - (n - 1) / 2.0) * 0.3e-3, np.zeros(n * n)], 1)
    ang[1::2] = ang[1::2, ::-1]                      # azimuth and elevation tilts in turn
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return dict(ndim=3, elem_pos=e.astype(np.float32), tx_angles=ang, fs=31.2e6, fc=7.8e6, c=C0, t0=0.0,
                f_number=case["f_number"], apod=case["apod"], n_samples=case["samples"], n_frames=case["frames"],
                grid_dims=(nx, ny, nz), grid_origin=(-(nx - 1) * step / 2, -(ny - 1) * step / 2, 3e-3),
                grid_step=(step, step, step))


def _points(case):
    return case["nx"] * case.get("ny", 1) * case["nz"] * case["elems"] * case["tx"] * case["frames"]


def _instances(case):
    """The batch's acquisitions: sizes log-uniform as in the ragged batches, grids scaled."""
    r, got = np.random.default_rng(case["shapes"]), []

    def logu(lo, hi):
        return math.exp(r.uniform(math.log(lo), math.log(hi)))

    for i in range(case["count"]):
        d = dict(kind="das", frames=int(round(logu(1, 48))), tx=int(round(logu(1, 15))), spread=10.0, step=0.1e-3)
        if i % 2 == 0:
            side = int(round(logu(128, 384) * case["scale"]))
            d.update(array="linear", elems=int(round(logu(64, 256))), nx=side, nz=side, apod="hann", f_number=1.5)
            deepest, fs = 5e-3 + side * 1e-4, 20.8e6
        else:
            side = int(round(logu(64, 112) * case["scale"]))
            d.update(array="matrix", elems=int(round(math.sqrt(logu(256, 1024)))) ** 2, nx=side, ny=side, nz=side,
                     apod="gauss", f_number=1.0)
            deepest, fs = 3e-3 + side * 1e-4, 31.2e6
        d["samples"] = int(math.ceil(2.3 * deepest * fs / C0)) + 32
        got.append(d)
    return got


# ---- inputs ----------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _iq(shape, gen):
    """Complex64 [T, C, S, F]: band-limited speckle that is mostly still over the frames, as tissue
    is, plus an independent part per frame (flow and noise)."""
    T, C, S, F = shape
    base = torch.randn((T * C, 2, S), device="cuda", generator=gen)
    kern = torch.exp(-0.5 * (torch.arange(-6, 7, device="cuda") / 2.5) ** 2)
    kern = (kern / kern.square().sum().sqrt())[None, None]
    base = torch.nn.functional.conv1d(base.view(-1, 1, S), kern, padding=6).view(T, C, 2, S)
    x = torch.randn((T, C, S, F, 2), device="cuda", generator=gen)
    x.mul_(0.3).add_(base.permute(0, 1, 3, 2)[:, :, :, None, :])
    return torch.view_as_complex(x)


def _store(iq, dtype):
    if dtype == "c64":
        return iq
    r = torch.view_as_real(iq)
    if dtype == "c64split":
        return r.transpose(-1, -2).contiguous()
    return r.to(torch.float16 if dtype == "f16x2" else torch.bfloat16).contiguous()


def _rows64(stored, dtype, t, c):
    """Complex128 [S, F] samples of one (transmit, element), as stored."""
    x = stored[t, c]
    if dtype == "c64":
        return x.to(torch.complex128)
    x = x.double()
    return torch.complex(x[:, 0], x[:, 1]) if dtype == "c64split" else torch.complex(x[..., 0], x[..., 1])


def _das_input(case, gen):
    return _store(_iq((case["tx"], case["elems"], case["samples"], case["frames"]), gen), case["dtype"])


def _taps(n, decim):
    """Windowed-sinc low-pass of unit DC gain."""
    k = np.arange(n) - (n - 1) / 2.0
    h = np.sinc(k / (2.0 * decim)) * np.hamming(n) if n > 1 else np.ones(1)
    return (h / h.sum()).astype(np.float32)


def _rf_input(case, gen):
    S, F = case["samples"], case["frames"]
    x = torch.randn((1, case["rows"], S, F), device="cuda", generator=gen)
    t = torch.arange(S, device="cuda", dtype=torch.float64) / 83.2e6
    return x.mul_(torch.cos(2 * math.pi * 5.2e6 * t).float()[None, None, :, None])


def _volumes(case, gen):
    """(few-angle, many-angle) complex64 [V, batch] volumes: smooth complex noise, and a sharper
    volume correlated with it."""
    n, shape = case["batch"], (case["nz"], case["ny"], case["nx"])
    x = torch.randn((2 * n, 1) + shape, device="cuda", generator=gen)
    y = torch.nn.functional.avg_pool3d(x, 3, stride=1, padding=1)
    a, b = (2.0 * y + 0.3 * x).view(n, 2, -1), (2.0 * y + 0.6 * x).view(n, 2, -1)
    return tuple(torch.view_as_complex(v.permute(2, 0, 1).contiguous()) for v in (a, b))


def _weights():
    path = os.path.join(learned.WEIGHTS_DIR, "unet_few3_many21_128.npz")
    return learned.load(path)          # params, gain, levels, base channels, coords


def _layer_input(case, gen):
    ci, co = case["ci"], case["co"]
    shape = (case["batch"], case["nz"], case["ny"], case["nx"])
    x = torch.randn(shape + (ci,), device="cuda", generator=gen)
    x = torch.where(x > 0, x, x / 64).to(torch.bfloat16)
    w = (torch.randn((27, ci, co), device="cuda", generator=gen) * math.sqrt(2.0 / (27 * ci))).to(torch.bfloat16).float()
    b = torch.randn((co,), device="cuda", generator=gen) * 0.1
    g = torch.randn(shape + (co,), device="cuda", generator=gen).to(torch.bfloat16)
    return x, w, b, g


def prepare(case, seed):
    gen, kind = _gen(seed), case["kind"]
    if kind == "das":
        return dict(case=case, plan=mach.Plan(iq_dtype=case["dtype"], **_geometry(case)), iq=_das_input(case, gen))
    if kind == "batch":
        inst = [dict(d, dtype=case["dtype"]) for d in _instances(case)]
        iqs = [_das_input(d, gen) for d in inst]
        vox = [d["nx"] * d.get("ny", 1) * d["nz"] for d in inst]
        ys = [torch.empty((v, d["frames"]), dtype=torch.complex64, device="cuda") for v, d in zip(vox, inst)]
        pds = [torch.empty((v,), dtype=torch.float32, device="cuda") for v in vox]
        batch = mach.Batch([dict(_geometry(d), iq_dtype=d["dtype"]) for d in inst])
        batch.bind(iqs, ys, pds)
        return dict(case=case, batch=batch, iqs=iqs, ys=ys, pds=pds)
    if kind == "convert":
        x = _iq((case["tx"], case["elems"], case["samples"], case["frames"]), gen)
        return dict(case=case, src=x.permute(3, 0, 1, 2).contiguous() if case["order"] == "ftcs" else x)
    if kind == "rf":
        return dict(case=case, rf=_rf_input(case, gen), taps=_taps(case["taps"], case["decim"]))
    if kind == "layer":
        x, w, b, g = _layer_input(case, gen)
        wpk, wpkt = nn.mach_nn_pack_weights(w, case["ci"], case["co"])
        return dict(case=case, x=x, b=b, g=g, wpk=wpk, wpkt=wpkt, w=w)
    params, gain, levels, base, coords = _weights()
    net = nn.UNet(case["nx"], case["ny"], case["nz"], case["batch"], levels=levels, base_ch=base,
                  inference_only=not case["train"], coords=coords)
    net.set_params(params)
    net.set_gain(gain)
    few, many = _volumes(case, gen)
    return dict(case=case, net=net, few=few, many=many if case["train"] else None,
                loss=torch.zeros(1, device="cuda") if case["train"] else None)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "das":
        if case["frames"] == 1:
            return {"y": state["plan"].run(state["iq"])}
        pd, y = state["plan"].power_doppler(state["iq"], want_y=True)
        return {"y": y, "pd": pd}
    if kind == "batch":
        state["batch"].run()
        return {"y": state["ys"], "pd": state["pds"]}
    if kind == "convert":
        return {"iq": mach.prepare_iq(state["src"], case["order"], case["dtype"])}
    if kind == "rf":
        return {"iq": mach.mach_rf_to_iq(state["rf"], state["taps"], 83.2e6, 5.2e6, 0.0, case["decim"])}
    if kind == "layer":
        x, g, ci, co = state["x"], state["g"], case["ci"], case["co"]
        y = torch.empty(x.shape[:4] + (co,), dtype=torch.bfloat16, device="cuda")
        dx = torch.empty_like(x)
        dw, db = torch.zeros((27, ci, co), device="cuda"), torch.zeros((co,), device="cuda")
        nn.mach_nn_conv3d_tc(x, state["wpk"], co, state["b"], y, None, act=True)
        nn.mach_nn_conv3d_wgrad(x, g, dw)
        nn.mach_nn_bias_grad(g, db)
        nn.mach_nn_conv3d_tc(g, state["wpkt"], ci, None, dx, None, flip=True)
        return {"y": y, "dx": dx, "dw": dw, "db": db}
    if not case["train"]:
        return {"y": state["net"].forward(state["few"])}
    state["net"].backward(state["few"], state["many"], state["loss"])
    return {"loss": state["loss"], "grads": state["net"].grads()}


# ---- what a pass cannot do without -------------------------------------------------------------

_BYTES = {"c64": 8, "c64split": 8, "f16x2": 4, "bf16x2": 4}


def _inside(case):
    """Share of (voxel, element) pairs inside the aperture, from a sample of the voxels."""
    g = _geometry(case)
    nx, ny, nz = g["grid_dims"]
    v = np.unique(np.linspace(0, nx * ny * nz - 1, 1024).astype(np.int64))
    p = np.stack([v % nx, (v // nx) % ny, v // (nx * ny)], 1) * np.array(g["grid_step"]) + np.array(g["grid_origin"])
    d = p[:, None, :] - g["elem_pos"][None].astype(np.float64)
    return float(np.mean(np.hypot(d[..., 0], d[..., 1]) * 2 * g["f_number"] <= d[..., 2]))


def _das_work(case, dtype):
    v = case["nx"] * case.get("ny", 1) * case["nz"]
    f = case["frames"]
    rd = case["tx"] * case["elems"] * case["samples"] * f * _BYTES[dtype]
    return rd + v * f * 8 + (v * 4 if f > 1 else 0), 16.0 * _points(case) * _inside(case)


def work(case):
    kind = case["kind"]
    if kind == "das":
        by, fl = _das_work(case, case["dtype"])
    elif kind == "batch":
        got = [_das_work(d, case["dtype"]) for d in _instances(case)]
        by, fl = sum(g[0] for g in got), sum(g[1] for g in got)
    elif kind == "convert":
        by, fl = case["tx"] * case["elems"] * case["samples"] * case["frames"] * (8 + _BYTES[case["dtype"]]), 0
    elif kind == "rf":
        n_iq = (case["samples"] - 1) // case["decim"] + 1
        by = case["rows"] * case["frames"] * (4 * case["samples"] + 8 * n_iq)
        fl = 4.0 * case["rows"] * case["frames"] * n_iq * case["taps"]
    elif kind == "layer":
        v = case["batch"] * case["nx"] * case["ny"] * case["nz"]
        by, fl = 2 * v * 2 * (case["ci"] + case["co"]), 3 * 54.0 * v * case["ci"] * case["co"]
    else:
        v = case["batch"] * case["nx"] * case["ny"] * case["nz"]
        # real channel counts at the network's two ends (2), 16 / 32 / 64 / 128 in between
        macs = 27.0 * (2 * 16 + 16 * 16 + 48 * 16 + 16 * 16 + 16 * 2
                       + (16 * 32 + 32 * 32 + 96 * 32 + 32 * 32) / 8
                       + (32 * 64 + 64 * 64 + 192 * 64 + 64 * 64) / 64 + (64 * 128 + 128 * 128) / 512)
        # volumes in and out; every layer's activations written and read once each way
        acts = 2.0 * v * (5 * 16 + 4 * 32 / 8 + 4 * 64 / 64 + 2 * 128 / 512)
        by, fl = 16 * v + 2 * acts * (3 if case["train"] else 1), 2 * macs * v * (3 if case["train"] else 1)
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("das", "batch"):
        return {"rel": 1e-5, "max": 1e-4}       # float32 sums of up to 16,000 terms in another order
    if kind == "convert":
        return "exact"
    if kind == "rf":
        return {"rel": 1e-6, "max": 1e-5}        # float32 sums of up to 64 taps in another order
    if kind == "layer":
        return {"rel": 4e-3, "max": 3e-2}       # bfloat16 results, float32 sums
    return {"rel": 1e-2, "max": 0.4}            # some thirty bfloat16 roundings in a row


# ---- the same in 64 bits ------------------------------------------------------------------------

def _f32(x):
    return x.float().double()


def _das_exact(case, stored):
    """Delay-and-sum: delays, sample index and aperture decided in float32 as the interface states
    (every step rounded to float32), interpolation, phase, window and sums in 64 bits."""
    g = _geometry(case)
    k = g["fs"] / g["c"]
    nx, ny, nz = g["grid_dims"]
    F, S = case["frames"], case["samples"]
    o, st = g["grid_origin"], g["grid_step"]
    ax = [o[i] + torch.arange(n, device="cuda", dtype=torch.float64) * st[i] for i, n in enumerate((nx, ny, nz))]
    pz, py, px = (a.reshape(-1) for a in torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij"))
    vx, vy, vz = _f32(px * k), _f32(py * k), _f32(pz * k)
    el = np.float32(g["elem_pos"].astype(np.float64) * k).astype(np.float64)
    V = px.numel()
    y = torch.zeros((V, F), dtype=torch.complex128, device="cuda")
    fn = g["f_number"]
    four = float(np.float32(4 * fn * fn))
    stx = []
    for az, ev in g["tx_angles"]:
        u = (math.sin(az) * math.cos(ev), math.sin(ev), math.cos(az) * math.cos(ev))
        stx.append(_f32((u[0] * px + u[1] * py + u[2] * pz) * k))
    for c in range(case["elems"]):
        dx, dy, dz = _f32(vx - el[c, 0]), _f32(vy - el[c, 1]), _f32(vz - el[c, 2])
        rx = _f32(torch.sqrt(_f32(dx * dx + _f32(dy * dy + _f32(dz * dz)))))
        rho2, dz2 = _f32(dx * dx + _f32(dy * dy)), _f32(dz * dz)
        inside = ((dz > 0) & (_f32(rho2 * four) <= dz2)).nonzero().flatten()
        t2 = (rho2 * fn * fn / (dz * dz))[inside]
        if g["apod"] == "hann":
            a = torch.cos(math.pi * torch.sqrt(t2)) ** 2
        else:
            a = torch.exp(-8 * t2) if g["apod"] == "gauss" else torch.ones_like(t2)
        rx = rx[inside]
        for t in range(case["tx"]):
            s = _f32(stx[t][inside] + rx)
            ok = (s >= 0) & (s < S - 1)
            v, s, w = inside[ok], s[ok], a[ok]
            i0 = torch.floor(s)
            f = s - i0
            ph = 2 * math.pi * g["fc"] * (s / g["fs"])
            cw = torch.complex(w * torch.cos(ph), w * torch.sin(ph))
            rows = _rows64(stored, case["dtype"], t, c)
            i0 = i0.long()
            y.index_add_(0, v, (cw * (1 - f))[:, None] * rows[i0] + (cw * f)[:, None] * rows[i0 + 1])
    return y, (y.real ** 2 + y.imag ** 2).sum(1)


def _conv64(x, w, b=None):
    """x [N, D, H, W, ci], w [27, ci, co] (taps z, y, x), zero padding, in 64 bits."""
    ci, co = w.shape[1:]
    k = w.view(3, 3, 3, ci, co).permute(4, 3, 0, 1, 2)
    y = torch.nn.functional.conv3d(x.permute(0, 4, 1, 2, 3), k, b, padding=1)
    return y.permute(0, 2, 3, 4, 1)


def _lrelu(x):
    return torch.where(x > 0, x, x / 64)


def _unet64(case, p, gain, x, levels, base):
    """Network output in units of each volume's RMS, [N, D, H, W, 2], and the scaled input."""
    n, shape = case["batch"], (case["nz"], case["ny"], case["nx"])
    at = [0]

    def conv(a, ci, co, act=True):
        w = p[at[0]:at[0] + 27 * ci * co].view(27, ci, co)
        b = p[at[0] + 27 * ci * co:at[0] + 27 * ci * co + co]
        at[0] += 27 * ci * co + co
        a = _conv64(a, w, b)
        return _lrelu(a) if act else a

    h = torch.nn.functional.pad(x, (0, base - 2))
    skips, c_in = [], base
    for lv in range(levels):
        if lv:
            h = torch.nn.functional.avg_pool3d(h.permute(0, 4, 1, 2, 3), 2).permute(0, 2, 3, 4, 1)
        c = base << lv
        h = conv(conv(h, c_in, c), c, c)
        skips.append(h)
        c_in = c
    for lv in range(levels - 2, -1, -1):
        c = base << lv
        h = h.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
        h = conv(conv(torch.cat([h, skips[lv]], -1), 3 * c, c), c, c)
    return conv(h, base, base, act=False)[..., :2] + gain * x


def _as_volumes(v, case):
    n = case["batch"]
    return torch.view_as_real(v.to(torch.complex128)).permute(1, 0, 2).reshape(n, case["nz"], case["ny"], case["nx"], 2)


def exact(case, seed):
    gen, kind = _gen(seed), case["kind"]
    if kind == "das":
        y, pd = _das_exact(case, _das_input(case, gen))
        return {"y": y} if case["frames"] == 1 else {"y": y, "pd": pd}
    if kind == "batch":
        inst = [dict(d, dtype=case["dtype"]) for d in _instances(case)]
        got = [_das_exact(d, _das_input(d, gen)) for d in inst]
        return {"y": [g[0] for g in got], "pd": [g[1] for g in got]}
    if kind == "convert":
        x = _iq((case["tx"], case["elems"], case["samples"], case["frames"]), gen)
        r = torch.view_as_real(x)
        if case["dtype"] == "c64":
            return {"iq": x.to(torch.complex128)}
        return {"iq": (r.transpose(-1, -2) if case["dtype"] == "c64split" else r).double().contiguous()}
    if kind == "rf":
        rf, h, D = _rf_input(case, gen), _taps(case["taps"], case["decim"]), case["decim"]
        S, L = case["samples"], case["taps"]
        n = torch.arange((S - 1) // D + 1, device="cuda")
        out = torch.zeros((1, case["rows"], n.numel(), case["frames"]), dtype=torch.complex128, device="cuda")
        for k in range(L):
            m = n * D + k - (L - 1) // 2
            ok = ((m >= 0) & (m < S)).double()
            ph = -2 * math.pi * torch.remainder(m.double() * 5.2e6 / 83.2e6, 1.0)
            e = float(h[k]) * ok * torch.exp(1j * ph)
            out += rf[:, :, m.clamp(0, S - 1), :].double() * e[None, None, :, None]
        return {"iq": out}
    if kind == "layer":
        x, w, b, g = _layer_input(case, gen)
        x64, w64 = x.double().requires_grad_(), w.double().requires_grad_()
        y = _conv64(x64, w64, None)
        dx, dw = torch.autograd.grad(y, (x64, w64), g.double())
        return {"y": _lrelu(y.detach() + b.double()).contiguous(), "dx": dx.contiguous(), "dw": dw,
                "db": g.double().sum((0, 1, 2, 3))}
    params, gain, levels, base, coords = _weights()
    few, many = _volumes(case, gen)
    p = torch.as_tensor(params, device="cuda").double().requires_grad_(case["train"])
    x = _as_volumes(few, case)
    rms = x.square().sum(-1).mean((1, 2, 3)).sqrt()[:, None, None, None, None]
    if not case["train"]:
        with torch.no_grad():
            o = rms * _unet64(case, p, gain, x / rms, levels, base)
        return {"y": torch.view_as_complex(o.reshape(case["batch"], -1, 2).permute(1, 0, 2).contiguous())}
    o = _unet64(case, p, gain, x / rms, levels, base)
    loss = (o - _as_volumes(many, case) / rms).square().mean()
    loss.backward()
    return {"loss": loss.detach().reshape(1), "grads": p.grad}
