"""Performance cases of the real-time controller: what users have it do, at the sizes they do it.

A case is a dict of plain values; ``prepare`` builds what a user's program holds before
the call (controller handle, matrix, frames on the device or in pinned memory, network),
``run`` makes one pass through the public entry points, ``exact`` recomputes the pass in
64 bits with plain torch, without the library.

Kinds of case
  frame     Rtc.process_frame_async: one frame in device memory -> DM commands (and slopes)
  host      Rtc.process_frame on pinned buffers: one frame, host to host
  slopes    Rtc.centroid_async over a chunk of frames: a slope sequence is recorded
  mvm       mvm_integrate_noalloc: reconstruction on the caller's own device buffers
  predict   Mlp.predict_seq: the slope predictor over a recorded sequence
  train     Mlp.train_seq steps on a recorded sequence, then Mlp.get_params
  loop      Rtc.run_loop: the persistent loop over a run of frames, every command kept
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1805_07254_gb300 import Mlp, Rtc
from paper_1805_07254_gb300.rtc import mvm_integrate_noalloc

STORES = ("f32", "bf16", "f16", "fp8", "int8")
NPARAMS = 17154
SIZES = (200, 64, 64, 2)


def _frame(name, nsub, npx, obs, store, **kw):
    c = {"name": name, "kind": "frame", "nsub": nsub, "npx": npx, "obs": obs, "n_wfs": 1, "store": store,
         "pred": False, "slopes": False, "thr_mode": 0}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest system (8x8 subapertures of 8x8 px, 69 actuators): a laboratory
        # bench or a truth sensor, its telemetry wanting the slopes of every frame.
        # Latency and launches are all there is.
        _frame("frame_8x8_f32", 8, 8, 0.0, "f32", slopes=True),
        # An 8 m class system with odd boxes and the subtract-and-clip threshold, 16-bit
        # matrix: neither the box size nor the row widths are the tuned ones.
        _frame("frame_41x41_f16", 41, 7, 0.14, "f16", thr_mode=1),
        # The extremely-large-telescope system the framework is quoted on, FP32 matrix.
        _frame("frame_elt_f32", 74, 10, 0.28, "f32"),
        # The same system with the 8-bit matrix that meets the accuracy target.
        _frame("frame_elt_int8", 74, 10, 0.28, "int8"),
        # The same system with the learned slope predictor in the loop, BF16 matrix.
        _frame("frame_elt_bf16_pred", 74, 10, 0.28, "bf16", pred=True),
        # Six such sensors on one mirror (the stress sizing), FP8 matrix: the largest frame.
        _frame("frame_6wfs_fp8", 74, 10, 0.28, "fp8", n_wfs=6),
        # A camera thread with its own pinned buffers, one synchronous call per frame.
        {"name": "host_elt_f32", "kind": "host", "nsub": 74, "npx": 10, "obs": 0.28, "n_wfs": 1,
         "store": "f32", "thr_mode": 0},
        # Recording a slope sequence for training: frames come in chunks of 64.
        {"name": "slopes_elt_64", "kind": "slopes", "nsub": 74, "npx": 10, "obs": 0.28, "frames": 64,
         "thr_mode": 0},
        # The reconstruction of a host framework that owns every buffer, FP32, at the
        # size of an 80x80 system (5169 x 9416).
        {"name": "mvm_80x80_f32", "kind": "mvm", "nact": 5169, "nslopes": 9416, "store": "f32", "ksplit": 1},
        # Scoring a trained predictor on held-out frames.
        {"name": "predict_elt_1000", "kind": "predict", "nsub": 74, "obs": 0.28, "frames": 1000},
        # Refining a predictor on a recorded sequence: 16 steps at the batch size the
        # trainer uses, then the parameters.
        {"name": "train_elt_16x4096", "kind": "train", "nsub": 74, "obs": 0.28, "frames": 400,
         "batch": 4096, "steps": 16},
        # The persistent loop flat out over 100 frames, the mirror taking every command.
        {"name": "loop_elt_bf16_100", "kind": "loop", "nsub": 74, "npx": 10, "obs": 0.28, "n_wfs": 1,
         "store": "bf16", "pred": False, "thr_mode": 0, "frames": 100, "preload": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes spread over the kind's whole range."""
    kind = rng.choice(("frame", "frame", "frame", "host", "slopes", "mvm", "predict", "train", "loop"))
    nsub = _log_int(rng, 4, 80)
    npx = rng.randint(4, 12)
    obs = rng.choice((0.0, 0.14, 0.25, 0.28))
    thr_mode = rng.randint(0, 1)
    if kind == "frame":
        n_wfs = rng.choice((1, 1, 1, 2, 3))
        store = rng.choice(STORES) if n_wfs == 1 else rng.choice(("fp8", "int8"))
        return {"kind": kind, "nsub": nsub, "npx": npx, "obs": obs, "n_wfs": n_wfs, "store": store,
                "pred": n_wfs == 1 and rng.random() < 0.3, "slopes": rng.random() < 0.5, "thr_mode": thr_mode}
    if kind == "host":
        return {"kind": kind, "nsub": nsub, "npx": npx, "obs": obs, "n_wfs": 1, "store": rng.choice(STORES),
                "thr_mode": thr_mode}
    if kind == "slopes":
        return {"kind": kind, "nsub": nsub, "npx": npx, "obs": obs, "frames": _log_int(rng, 1, 64),
                "thr_mode": thr_mode}
    if kind == "mvm":
        return {"kind": kind, "nact": _log_int(rng, 50, 5169), "nslopes": _log_int(rng, 60, 9416),
                "store": rng.choice(STORES), "ksplit": rng.choice((1, 1, 2, 5, 16))}
    if kind == "predict":
        return {"kind": kind, "nsub": min(nsub, 74), "obs": obs, "frames": _log_int(rng, 5, 1000)}
    if kind == "train":
        return {"kind": kind, "nsub": min(nsub, 74), "obs": obs, "frames": _log_int(rng, 6, 400),
                "batch": _log_int(rng, 50, 4096), "steps": _log_int(rng, 1, 16)}
    return {"kind": kind, "nsub": nsub, "npx": npx, "obs": obs, "n_wfs": 1, "store": rng.choice(STORES),
            "pred": rng.random() < 0.3, "thr_mode": thr_mode, "frames": _log_int(rng, 10, 100),
            "preload": rng.randint(1, 8)}


# ---- inputs --------------------------------------------------------------------------


def _subaps(nsub, obs):
    """Valid subapertures (row, col): centres inside the annulus, row-major order."""
    c = np.arange(nsub) + 0.5 - nsub / 2.0
    d2 = c[:, None] ** 2 + c[None, :] ** 2
    return np.argwhere((d2 <= (nsub / 2.0) ** 2) & (d2 >= (float(np.float32(obs)) * nsub / 2.0) ** 2)).astype(np.int32)


def _n_act(nsub):
    """Actuators of the (nsub + 1)-square mirror inside its circle."""
    c = np.arange(nsub + 1) - nsub / 2.0
    return int(np.count_nonzero(np.hypot(c[:, None], c[None, :]) <= nsub / 2.0 + 0.5))


def _gen(seed, part):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + part)


def _maps(c, seed):
    side = c["nsub"] * c["npx"]
    g = _gen(seed, 1)
    shape = (c.get("n_wfs", 1), side, side)
    dark = 90.0 + 20.0 * torch.rand(shape, generator=g, device="cuda")
    flat = 1.0 + 0.02 * torch.randn(shape, generator=g, device="cuda")
    return dark, flat


def _frames(c, seed, n, dark, flat):
    """Detector frames uint16 [n][n_wfs][H][W]: one pixel-integrated Gaussian spot of 1000
    photo-electrons per valid subaperture (0.3 px slopes, sigma 1.2 px), photon and read
    noise, the detector's own dark and flat."""
    nsub, npx, nw = c["nsub"], c["npx"], c.get("n_wfs", 1)
    sa = torch.from_numpy(_subaps(nsub, c["obs"]).astype(np.int64)).cuda()
    g = _gen(seed, 2)
    side = nsub * npx
    x = torch.arange(npx, device="cuda", dtype=torch.float32)
    k = 1.0 / (1.2 * math.sqrt(2.0))
    out = torch.empty((n, nw, side, side), dtype=torch.uint16, device="cuda")
    for f in range(n):
        mu = (npx - 1) / 2.0 + 0.3 * torch.randn((nw, sa.shape[0], 2), generator=g, device="cuda")
        box = 0.5 * (torch.erf((x + 0.5 - mu[..., None]) * k) - torch.erf((x - 0.5 - mu[..., None]) * k))
        photons = torch.poisson(1000.0 * box[:, :, 1, :, None] * box[:, :, 0, None, :], generator=g)
        img = torch.zeros((nw, nsub, nsub, npx, npx), device="cuda")
        img[:, sa[:, 0], sa[:, 1]] = photons
        img = img.permute(0, 1, 3, 2, 4).reshape(nw, side, side)
        img = img + torch.randn(img.shape, generator=g, device="cuda")
        out[f] = torch.clamp(torch.round(flat * img + dark), 0, 65535).to(torch.int32).to(torch.uint16)
    return out


def _matrix(seed, nact, ncol):
    return torch.randn((nact, ncol), generator=_gen(seed, 3), device="cuda") / math.sqrt(ncol)


def _fp8(m):
    """E4M3 codes (as bytes) and row scales of a matrix."""
    scale = m.abs().amax(dim=1) / 448.0
    return (m / scale[:, None]).to(torch.float8_e4m3fn).view(torch.uint8), scale


def _int8(m):
    scale = m.abs().amax(dim=1) / 127.0
    return torch.round(m / scale[:, None]).clamp(-127, 127).to(torch.int8), scale


def _params(seed):
    """A network's parameters: each layer uniform in +-1/sqrt(fan in)."""
    rng = np.random.default_rng(seed)
    parts = []
    for i in range(3):
        b = 1.0 / math.sqrt(SIZES[i])
        parts += [rng.uniform(-b, b, SIZES[i + 1] * SIZES[i]), rng.uniform(-b, b, SIZES[i + 1])]
    return np.concatenate(parts).astype(np.float32)


def _sequence(c, seed):
    """A slope sequence float32 [frames][2 n_valid]: plane waves crossing the pupil plus
    measurement noise, 0.3 px RMS."""
    sa = torch.from_numpy(_subaps(c["nsub"], c["obs"])).cuda().float()
    g = _gen(seed, 4)
    n, nv = c["frames"], sa.shape[0]
    t = torch.arange(n, device="cuda", dtype=torch.float32)[:, None]
    s = torch.zeros((n, 2 * nv), device="cuda")
    for _ in range(8):
        kx, ky, w, p, a = torch.randn(5, generator=g, device="cuda")
        wave = torch.cos(0.3 * (kx * sa[:, 1] + ky * sa[:, 0])[None, :] + 0.3 * w * t + 6.3 * p)
        s[:, :nv] += a * kx * wave
        s[:, nv:] += a * ky * wave
    s *= 0.3 / torch.clamp(s.square().mean().sqrt(), min=1e-6)
    s += 0.05 * torch.randn(s.shape, generator=g, device="cuda")
    return s.contiguous()


SIGMA = 0.3
LR = 1e-5


def _controller(c, seed, dark, flat):
    nact = _n_act(c["nsub"])
    nv = _subaps(c["nsub"], c["obs"]).shape[0]
    r = Rtc(c["nsub"], c["npx"], nact, n_wfs=c["n_wfs"], obs=c["obs"], thr_mode=c["thr_mode"],
            thr=3.0 if c["thr_mode"] else 0.0)
    r.load_calib(dark.cpu().numpy(), flat.cpu().numpy())
    m = _matrix(seed, nact, 2 * nv * c["n_wfs"])
    if c["store"] == "fp8":         # quantised by the user: codes and row scales
        codes, scale = _fp8(m)
        r.load_cmat(codes.cpu().numpy(), store="fp8", src="fp8", row_scales=scale.cpu().numpy())
    else:
        r.load_cmat(m.cpu().numpy(), store=c["store"])
    if c.get("pred"):
        r.load_predictor(_params(seed), SIGMA)
        r.set_predictor(True)
    return r


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"kind": kind, "case": c}
    if kind in ("frame", "host", "loop"):
        dark, flat = _maps(c, seed)
        r = st["rtc"] = _controller(c, seed, dark, flat)
        nact = _n_act(c["nsub"])
        frames = _frames(c, seed, c.get("preload", 1), dark, flat)
        if kind == "frame":
            st["frame"] = frames[0].contiguous()
            st["dm"] = torch.zeros(nact, device="cuda")
            st["s"] = torch.zeros(r.info()["nslopes"], device="cuda") if c["slopes"] else None
        elif kind == "host":
            st["frame"] = frames[0].cpu().pin_memory()
            st["dm"] = torch.zeros(nact).pin_memory()
        else:
            st["frames"] = frames.cpu().numpy()
    elif kind == "slopes":
        c = dict(c, n_wfs=1)
        dark, flat = _maps(c, seed)
        r = st["rtc"] = Rtc(c["nsub"], c["npx"], _n_act(c["nsub"]), obs=c["obs"], thr_mode=c["thr_mode"],
                            thr=3.0 if c["thr_mode"] else 0.0)
        r.load_calib(dark.cpu().numpy(), flat.cpu().numpy())
        # each frame a buffer of its own (the entry point wants them 16-byte aligned)
        st["frames"] = [f.clone() for f in _frames(c, seed, c["frames"], dark, flat)]
        st["S"] = torch.zeros((c["frames"], r.info()["nslopes"]), device="cuda")
    elif kind == "mvm":
        nact, ncol = c["nact"], c["nslopes"]
        kpad = (ncol + 15) // 16 * 16
        m = torch.zeros((nact, kpad), device="cuda")
        m[:, :ncol] = _matrix(seed, nact, ncol)
        scale = None
        if c["store"] == "fp8":
            m, scale = _fp8(m)
        elif c["store"] == "int8":
            m, scale = _int8(m)
        elif c["store"] != "f32":
            m = m.to(torch.bfloat16 if c["store"] == "bf16" else torch.float16)
        s = torch.zeros(kpad, device="cuda")
        s[:ncol] = 0.3 * torch.randn(ncol, generator=_gen(seed, 5), device="cuda")
        st.update(M=m.contiguous(), scale=scale, s=s, kpad=kpad, a=torch.zeros(nact, device="cuda"),
                  dm=torch.zeros(nact, device="cuda"))
    else:                            # predict, train
        m = st["mlp"] = Mlp(params=_params(seed))
        sa = _subaps(c["nsub"], c["obs"])
        m.set_geometry(sa, c["nsub"])
        st["S"] = _sequence(c, seed)
        if kind == "predict":
            st["out"] = torch.zeros_like(st["S"])
        else:
            st["samples"] = _samples(c, seed)
            st["loss"] = torch.zeros(1, device="cuda")
    return st


def _samples(c, seed):
    """(subaperture, frame) of every sample: int32 [steps][batch][2]."""
    g = _gen(seed, 6)
    nv = _subaps(c["nsub"], c["obs"]).shape[0]
    shape = (c["steps"], c["batch"])
    i = torch.randint(0, nv, shape, generator=g, device="cuda", dtype=torch.int32)
    k = torch.randint(3, c["frames"] - 1, shape, generator=g, device="cuda", dtype=torch.int32)
    return torch.stack([i, k], dim=-1).contiguous()


def run(state):
    c, kind = state["case"], state["kind"]
    if kind == "frame":
        state["rtc"].process_frame_async(state["frame"], state["dm"], state["s"],
                                         stream=torch.cuda.current_stream())
        return [state["dm"], state["s"]]
    if kind == "host":
        return state["rtc"].process_frame(state["frame"], dm_out=state["dm"])
    if kind == "slopes":
        r, st = state["rtc"], torch.cuda.current_stream()
        for f, s in zip(state["frames"], state["S"]):
            r.centroid_async(f, s, stream=st)
        return state["S"]
    if kind == "mvm":
        mvm_integrate_noalloc(state["M"], c["store"], state["scale"], c["nact"], state["kpad"], state["s"],
                              state["a"], state["dm"], ksplit=c["ksplit"], stream=torch.cuda.current_stream())
        return [state["dm"], state["a"]]
    if kind == "predict":
        state["mlp"].predict_seq(state["S"], SIGMA, state["out"], stream=torch.cuda.current_stream())
        return state["out"]
    if kind == "train":
        m, st = state["mlp"], torch.cuda.current_stream()
        for samples in state["samples"]:
            m.train_seq(state["S"], samples, SIGMA, LR, state["loss"], stream=st)
        return [m.get_params(), state["loss"]]
    got = []
    state["rtc"].run_loop(c["frames"], frames=state["frames"], sink=lambda k, dm: got.append(dm), record=False)
    return np.stack(got)


# ---- cost ----------------------------------------------------------------------------


def _esize(store):
    return {"f32": 4, "bf16": 2, "f16": 2}.get(store, 1)


def _frame_work(c, mvm=True):
    """Bytes and operations of one frame: pixels, calibration, matrix, state, commands."""
    nw = c.get("n_wfs", 1)
    nt, npp = nw * _subaps(c["nsub"], c["obs"]).shape[0], c["npx"] ** 2
    b, f = nt * npp * (2 + 8) + 8 * nt, 10 * nt * npp
    if mvm:
        nact, es = _n_act(c["nsub"]), _esize(c["store"])
        b += nact * 2 * nt * es + (4 * nact if es == 1 else 0) + 12 * nact
        f += 4 * nact * nt
    if c.get("pred"):
        b += 3 * 8 * nt + 4 * NPARAMS
        f += 2 * nt * (200 * 64 + 64 * 64 + 128)
    return b, f


def work(case):
    c, kind = case, case["kind"]
    if kind in ("frame", "host"):
        b, f = _frame_work(c)
    elif kind == "slopes":
        b, f = _frame_work(c, mvm=False)
        cal = 8 * c["npx"] ** 2 * _subaps(c["nsub"], c["obs"]).shape[0]
        b, f = (b - cal) * c["frames"] + cal, f * c["frames"]
    elif kind == "mvm":
        b = c["nact"] * c["nslopes"] * _esize(c["store"]) + 4 * c["nslopes"] + 12 * c["nact"]
        f = 2 * c["nact"] * c["nslopes"]
    elif kind == "predict":
        nv, n = _subaps(c["nsub"], c["obs"]).shape[0], c["frames"]
        b = 8 * nv * (2 * n - 4) + 4 * NPARAMS
        f = 2 * nv * (n - 4) * (200 * 64 + 64 * 64 + 128)
    elif kind == "train":
        nv = _subaps(c["nsub"], c["obs"]).shape[0]
        b = c["steps"] * (8 * c["batch"] + 6 * 4 * NPARAMS) + min(c["frames"] * nv * 8, c["steps"] * c["batch"] * 800)
        f = c["steps"] * 6 * c["batch"] * (200 * 64 + 64 * 64 + 128)
    else:
        # the matrix and the maps are kept on the chip or read again: each frame's own data counts once
        b, f = _frame_work(c)
        b, f = b + (c["frames"] - 1) * (4 * _n_act(c["nsub"]) + 2 * c["npx"] ** 2), f * c["frames"]
    return {"bytes": float(b), "flops": float(f)}


# ---- the same in 64 bits -------------------------------------------------------------


def _slopes64(c, frames, dark, flat):
    """Slopes float64 [frames][n_wfs * 2 * n_valid] of detector frames."""
    nsub, npx, nw = c["nsub"], c["npx"], c.get("n_wfs", 1)
    sa = torch.from_numpy(_subaps(nsub, c["obs"]).astype(np.int64)).cuda()
    x = torch.arange(npx, device="cuda", dtype=torch.float64) - (npx - 1) / 2.0
    out = []
    for f in frames:
        p = (f.to(torch.int32).double().reshape(dark.shape) - dark.double()) / flat.double()
        p = torch.clamp(p - 3.0, min=0.0) if c["thr_mode"] else torch.clamp(p, min=0.0)
        p = p.reshape(nw, nsub, npx, nsub, npx).permute(0, 1, 3, 2, 4)[:, sa[:, 0], sa[:, 1]]
        flux = p.sum((-1, -2))
        sx, sy = (p * x).sum((-1, -2)), (p * x[:, None]).sum((-1, -2))
        ok = flux > 0
        safe = torch.where(ok, flux, torch.ones_like(flux))
        z = torch.zeros_like(flux)
        out.append(torch.stack([torch.where(ok, sx / safe, z), torch.where(ok, sy / safe, z)], dim=1).reshape(-1))
    return torch.stack(out)


def _stored64(m, store):
    """The values a stored matrix stands for, chunk by chunk of rows."""
    if store == "f32":
        return m.double()
    if store in ("bf16", "f16"):
        return m.to(torch.bfloat16 if store == "bf16" else torch.float16).double()
    q, scale = _fp8(m) if store == "fp8" else _int8(m)
    q = q.view(torch.float8_e4m3fn).float() if store == "fp8" else q
    return q.double() * scale.double()[:, None]


def _product64(m, store, s):
    """M s for slope vectors s [n][ncol], in 64 bits."""
    return torch.cat([s @ _stored64(rows, store).T for rows in m.split(256)], dim=1)


def _net64(params):
    p, out, o = torch.from_numpy(params).cuda().double(), [], 0
    for i in range(3):
        n = SIZES[i + 1] * SIZES[i]
        out += [p[o:o + n].reshape(SIZES[i + 1], SIZES[i]), p[o + n:o + n + SIZES[i + 1]]]
        o += n + SIZES[i + 1]
    return out


def _forward64(net, x):
    gelu = torch.nn.functional.gelu
    h = gelu(x @ net[0].T + net[1])
    h = gelu(h @ net[2].T + net[3])
    return h @ net[4].T + net[5]


def _neighbours(sa, nsub):
    """Index of each subaperture's 25 neighbours, n_valid where there is none."""
    grid = np.full((nsub + 4, nsub + 4), sa.shape[0], np.int64)
    grid[sa[:, 0] + 2, sa[:, 1] + 2] = np.arange(sa.shape[0])
    return torch.from_numpy(np.stack([grid[sa[:, 0] + dr, sa[:, 1] + dc] for dr in range(5) for dc in range(5)],
                                     axis=1)).cuda()


def _features64(rows, nbr):
    """[..., 200] features of the 4 slope rows (newest first) [..., 2 n_valid] at neighbours nbr [..., 25]."""
    nv = rows[0].shape[-1] // 2
    out = []
    for lag in range(4):
        for axis in range(2):
            v = torch.nn.functional.pad(rows[lag][..., axis * nv:(axis + 1) * nv], (0, 1))
            out.append(torch.gather(v.expand(nbr.shape[0], -1), 1, nbr) if v.dim() == 2 else v[nbr])
    return torch.cat(out, dim=-1) / float(np.float32(SIGMA))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("frame", "host", "loop", "slopes"):
        if kind == "slopes":
            c = dict(c, n_wfs=1)
        dark, flat = _maps(c, seed)
        nf = c["frames"] if kind == "slopes" else c.get("preload", 1)
        s = _slopes64(c, _frames(c, seed, nf, dark, flat), dark, flat)
        if kind == "slopes":
            return s
        m = _matrix(seed, _n_act(c["nsub"]), s.shape[1])
        if not c.get("pred"):
            d = _product64(m, c["store"], s)
            if kind != "loop":
                return [0.4 * d[0], s[0] if c.get("slopes") else None] if kind == "frame" else 0.4 * d[0]
        net, sa = _net64(_params(seed)), _subaps(c["nsub"], c["obs"])
        nbr, zero = _neighbours(sa, c["nsub"]), torch.zeros_like(s[0])
        a, out, hist = torch.zeros(m.shape[0], device="cuda", dtype=torch.float64), [], [zero] * 4
        g, leak = float(np.float32(0.4)), float(np.float32(0.99))
        for k in range(c["frames"] if kind == "loop" else 1):
            f = k % nf
            if c.get("pred"):
                hist = [s[f]] + hist[:3]
                y = _forward64(net, _features64(hist, nbr))
                e = s[f] + float(np.float32(SIGMA)) * y.T.reshape(-1)
                a = leak * a + g * _product64(m, c["store"], e[None])[0]
            else:
                a = leak * a + g * d[f]
            out.append(a)
        if kind == "loop":
            return torch.stack(out)
        return [out[0], s[0] if c["slopes"] else None]
    if kind == "mvm":
        m = torch.zeros((c["nact"], (c["nslopes"] + 15) // 16 * 16), device="cuda")
        m[:, :c["nslopes"]] = _matrix(seed, c["nact"], c["nslopes"])
        s = 0.3 * torch.randn(c["nslopes"], generator=_gen(seed, 5), device="cuda")
        a = 0.4 * _product64(m, c["store"], torch.nn.functional.pad(s, (0, m.shape[1] - s.shape[0])).double()[None])[0]
        return [a, a]
    S, net = _sequence(c, seed).double(), _net64(_params(seed))
    sa = _subaps(c["nsub"], c["obs"])
    nbr, nv = _neighbours(sa, c["nsub"]), sa.shape[0]
    if kind == "predict":
        out = torch.zeros_like(S)
        for k in range(3, c["frames"] - 1):
            y = _forward64(net, _features64([S[k - lag] for lag in range(4)], nbr))
            out[k + 1] = S[k] + float(np.float32(SIGMA)) * y.T.reshape(-1)
        return out
    # training: the same steps of Adam on the definition's loss
    mom = [(torch.zeros_like(p), torch.zeros_like(p)) for p in net]
    loss = None
    for step, sm in enumerate(_samples(c, seed), 1):
        i, k = sm[:, 0].long(), sm[:, 1].long()
        x = _features64([S[k - lag] for lag in range(4)], nbr[i])
        t = torch.stack([S[k + 1, i] - S[k, i], S[k + 1, nv + i] - S[k, nv + i]], dim=1) / float(np.float32(SIGMA))
        for p in net:
            p.requires_grad_(True)
        loss = ((_forward64(net, x) - t) ** 2).sum() / (2 * x.shape[0])
        grads = torch.autograd.grad(loss, net)
        with torch.no_grad():
            new = []
            for j, (p, gr) in enumerate(zip(net, grads)):
                m1, m2 = 0.9 * mom[j][0] + 0.1 * gr, 0.999 * mom[j][1] + 0.001 * gr * gr
                mom[j] = (m1, m2)
                new.append(p - LR * (m1 / (1 - 0.9 ** step)) / ((m2 / (1 - 0.999 ** step)).sqrt() + 1e-8))
            net = [p.detach() for p in new]
    return [torch.cat([p.reshape(-1) for p in net]), loss.detach().reshape(1)]
