"""What the performance of this repository is measured on.

Every case is a piece of work a correlation plenoptic imaging program has this
library do, through the public binding (``paper_2407_20692_gb300``), from the
smallest acquisition of the configurations (16x16 vs 16x16) to the largest
single calls (128x128 vs 64x64 counts, 128x128 vs 128x128 binary).  ``listed()``
names them, ``draw(rng)`` gives others of the same ranges, odd and ragged sizes
among them.  Inputs are chaotic-light frames (a few complex Gaussian modes shared
by both detectors, so that Gamma is not just noise) or, for the steps that start
from Gamma, a smooth correlation plus the noise of few frames.
"""

import math
import os

import numpy as np
import torch

import paper_2407_20692_gb300 as cpi

ROOT = os.path.dirname(os.path.abspath(cpi.__file__))
DEV = "cuda"


# ----------------------------------------------------------------------------- the cases

def listed():
    return [
        # A small acquisition in a live loop: correlate, then refocus a few
        # planes.  Latency and the number of launches count.
        dict(name="step_u8_16_16", kind="step", bits=8, ha=16, wa=16, hb=16, wb=16, n=2000, mean=2.0, planes=4),
        # One SPAD acquisition: binary frames, Gamma and its 32 planes.
        dict(name="step_bits_64_32", kind="step", bits=1, ha=64, wa=64, hb=32, wb=32, n=20000, mean=0.3, planes=32),
        # The same detector streamed block by block from pinned host memory while
        # it is acquired, Gamma finalised at the end.
        dict(name="stream_bits_64_32", kind="stream", bits=1, ha=64, wa=64, hb=32, wb=32, n=8192 * 16, block=8192,
             mean=0.3),
        # The paper's way with long binary acquisitions: blocks of 64 files of 512
        # frames (.bin layout) added to running sums, then one finalisation.
        dict(name="blocks_bits_128_128", kind="blocks", bits=1, ha=128, wa=128, hb=128, wb=128, n=65536, block=32768,
             mean=0.1),
        # The largest single correlation: sums of 255 binary sub-frames.
        dict(name="corr_u8_128_64", kind="corr", bits=8, ha=128, wa=128, hb=64, wb=64, n=50000, mean=0.3,
             binomial=True),
        # A region of interest of odd size: rows and regions that start at no
        # aligned byte, frames that fill no whole block.
        dict(name="corr_u8_83_37", kind="corr", bits=8, ha=83, wa=83, hb=37, wb=37, n=17321, mean=2.0),
        # Refocusing of a large Gamma into a full stack.
        dict(name="refocus_128_64_p128", kind="refocus", ha=128, wa=128, hb=64, wb=64, planes=128),
        # 4-D multilinear refocusing at the paper's prototype region of interest.
        dict(name="refocus4d_128_128_p100", kind="refocus4d", ha=128, wa=128, hb=128, wb=128, planes=100),
        # Many uneven acquisitions in one replayed call, 256 planes each.
        dict(name="batch_8_uneven", kind="batch", items=8, lo_a=32, hi_a=96, lo_b=16, hi_b=48, lo_n=5000, hi_n=40000,
             planes=256, shapes=7),
        # The learned denoiser: one Gamma through the trained model.
        dict(name="denoise_64_32", kind="denoise", ha=64, wa=64, hb=32, wb=32),
        # The same network on a Gamma of an odd region of interest.
        dict(name="denoise_83_37", kind="denoise", ha=83, wa=83, hb=37, wb=37),
        # One training step of the denoiser: loss, gradients, Adam.
        dict(name="train_64_32", kind="train", ha=64, wa=64, hb=32, wb=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi, most):
    """Height and width; square detectors as often as others."""
    h = _log(rng, lo, hi)
    w = h if rng.random() < 0.5 else _log(rng, lo, hi)
    while h * w > most:
        h, w = max(lo, h * 7 // 8), max(lo, w * 7 // 8)
    return h, w


def draw(rng):
    kind = rng.choice(["step", "step", "corr", "refocus", "refocus", "refocus4d", "denoise", "train", "stream",
                       "blocks", "batch"])
    if kind in ("step", "corr"):
        bits = rng.choice([1, 8])
        ha, wa = _sides(rng, 16, 128, 128 * 128)
        hb, wb = _sides(rng, 8, 64, 64 * 64)
        n = _log(rng, 1000, 50000)
        c = dict(kind=kind, bits=bits, ha=ha, wa=wa, hb=hb, wb=wb, n=n, mean=0.3 if bits == 1 else 2.0)
        if kind == "step":
            c["planes"] = rng.randint(1, 64)
        return c
    if kind == "refocus":
        ha, wa = _sides(rng, 16, 128, 128 * 128)
        hb, wb = _sides(rng, 8, 64, 64 * 64)
        return dict(kind=kind, ha=ha, wa=wa, hb=hb, wb=wb, planes=_log(rng, 4, 128))
    if kind == "refocus4d":
        ha, wa = _sides(rng, 16, 112, 112 * 112)
        hb, wb = _sides(rng, 8, 112, 112 * 112)
        return dict(kind=kind, ha=ha, wa=wa, hb=hb, wb=wb, planes=_log(rng, 4, 100))
    if kind in ("denoise", "train"):
        if rng.random() < 0.5:   # the tensor-core widths as often as others
            wa = rng.choice([32, 64, 64, 128] if kind == "denoise" else [64])
            ha = _log(rng, 24, 96)
        else:
            ha, wa = _sides(rng, 24, 96, 96 * 96)
        hb, wb = _sides(rng, 8, 32, 32 * 32)
        most = (1 << 22) if kind == "denoise" or wa == 64 else (1 << 20)
        while ha * wa * hb * wb > most:
            hb, wb = max(4, hb * 7 // 8), max(4, wb * 7 // 8)
            ha = max(8, ha * 15 // 16)
        return dict(kind=kind, ha=ha, wa=wa, hb=hb, wb=wb)
    if kind == "stream":
        bits = rng.choice([1, 1, 8])
        ha, wa = _sides(rng, 16, 64, 64 * 64)
        hb, wb = _sides(rng, 8, 32, 32 * 32)
        block = _log(rng, 1024, 8192)
        return dict(kind=kind, bits=bits, ha=ha, wa=wa, hb=hb, wb=wb, n=block * rng.randint(2, 8) + rng.randint(0, 999),
                    block=block, mean=0.3 if bits == 1 else 2.0)
    if kind == "blocks":
        side = 32 * rng.randint(1, 3)
        block = 512 * rng.randint(8, 64)
        return dict(kind=kind, bits=1, ha=side, wa=side, hb=side, wb=side, n=block * rng.randint(1, 2), block=block,
                    mean=0.1)
    return dict(kind="batch", items=rng.randint(2, 6), lo_a=32, hi_a=96, lo_b=16, hi_b=48, lo_n=5000, hi_n=20000,
                planes=rng.choice([16, 64, 128, 256]), shapes=rng.randint(0, 10 ** 6))


# ----------------------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _counts(gen, n, ma, mb, case):
    """Photon counts (or clicks) of both detectors, uint8 [n][ma + mb]: thermal
    light of a few modes seen by both."""
    modes = 24
    maps = torch.complex(torch.randn((modes, ma + mb), generator=gen, device=DEV),
                         torch.randn((modes, ma + mb), generator=gen, device=DEV)) / math.sqrt(4.0 * modes)
    out = torch.empty((n, ma + mb), dtype=torch.uint8, device=DEV)
    step = max(256, (1 << 26) // (ma + mb))
    for i in range(0, n, step):
        k = min(step, n - i)
        e = torch.complex(torch.randn((k, modes), generator=gen, device=DEV),
                          torch.randn((k, modes), generator=gen, device=DEV)) * math.sqrt(2.0)
        f = torch.view_as_real(e @ maps)
        lam = f.square().sum(-1) * (0.5 * case["mean"])
        if case["bits"] == 1:
            v = torch.rand(lam.shape, generator=gen, device=DEV) < 1.0 - torch.exp(-lam)
        elif case.get("binomial"):   # sums of 255 sub-frames, each clicking with 1 - exp(-lam)
            p = 1.0 - torch.exp(-lam)
            v = (255.0 * p + torch.sqrt(255.0 * p * (1.0 - p)) * torch.randn(lam.shape, generator=gen, device=DEV))
            v = v.round().clamp_(0, 255)
        else:
            v = torch.poisson(lam, generator=gen).clamp_(0, 255)
        out[i:i + k] = v.to(torch.uint8)
    return out


def _frames(case, seed, salt=0):
    """Frames with A on the left and B on the right ([n][rows][wa + wb], one byte
    or one bit per pixel, least significant bit first), and the two regions."""
    ha, wa, hb, wb, n = (case[k] for k in ("ha", "wa", "hb", "wb", "n"))
    v = _counts(_gen(seed, salt), n, ha * wa, hb * wb, case)
    rows, cols = max(ha, hb), wa + wb
    img = torch.zeros((n, rows, cols), dtype=torch.uint8, device=DEV)
    img[:, :ha, :wa] = v[:, :ha * wa].view(n, ha, wa)
    img[:, :hb, wa:] = v[:, ha * wa:].view(n, hb, wb)
    if case["bits"] == 8:
        stride = rows * cols
    else:
        flat = img.view(n, rows * cols)
        pad = -(rows * cols) % 32
        if pad:
            flat = torch.nn.functional.pad(flat, (0, pad))
        stride = flat.shape[1] // 8
        weights = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], dtype=torch.uint8, device=DEV)
        packed = torch.empty((n, stride), dtype=torch.uint8, device=DEV)
        for i in range(0, n, 8192):
            packed[i:i + 8192] = (flat[i:i + 8192].view(-1, stride, 8) * weights).sum(-1, dtype=torch.uint8)
        img = packed
    a = dict(height=ha, width=wa, x0=0, row_stride=cols, frame_stride_bytes=stride)
    b = dict(height=hb, width=wb, x0=wa, row_stride=cols, frame_stride_bytes=stride)
    return img, a, b


def _values(case, seed, salt=0):
    """The counts _frames() lays out: (A [n][ma], B [n][mb]), uint8."""
    ma, mb = case["ha"] * case["wa"], case["hb"] * case["wb"]
    v = _counts(_gen(seed, salt), case["n"], ma, mb, case)
    return v[:, :ma], v[:, ma:]


def _gamma_input(case, seed):
    """Gamma in the slice-major layout [hb * wb][ha * wa]: an object's smooth
    correlation, which moves with the angular pixel, plus the noise of few frames."""
    ha, wa, hb, wb = (case[k] for k in ("ha", "wa", "hb", "wb"))
    gen = _gen(seed, 17)
    obj = torch.randn((1, 1, ha + 24, wa + 24), generator=gen, device=DEV)
    k = torch.exp(-0.5 * (torch.arange(-8, 9, device=DEV).float() / 3.0) ** 2)
    k = (k[:, None] * k[None, :] / k.sum() ** 2)[None, None]
    obj = torch.nn.functional.conv2d(obj, k)[0, 0] * 8.0
    g = torch.empty((hb * wb, ha, wa), dtype=torch.float32, device=DEV)
    for br in range(hb):
        oy = round(8.0 * br / max(1, hb - 1))
        for bc in range(wb):
            ox = round(8.0 * bc / max(1, wb - 1))
            g[br * wb + bc] = obj[oy:oy + ha, ox:ox + wa]
    g += torch.randn(g.shape, generator=gen, device=DEV)
    return g.view(hb * wb, ha * wa) * 0.02


def _planes(n):
    """Uniformly spaced planes; (1, 0) is the plane the spatial detector is focused on."""
    alpha = np.linspace(0.5, 1.5, n) if n > 1 else np.array([1.0])
    return alpha, 1.0 - alpha


def _planes4(n):
    alpha, beta = _planes(n)
    gamma = 0.5 * (alpha - 1.0)
    return alpha, beta, gamma, 1.0 - gamma


def _batch_shapes(case):
    r = np.random.Generator(np.random.Philox(case["shapes"]))
    return [dict(bits=8, ha=s, wa=s, hb=t, wb=t, n=int(r.integers(case["lo_n"], case["hi_n"] + 1)),
                 mean=float(r.uniform(1.0, 4.0)))
            for s, t in zip(r.integers(case["lo_a"], case["hi_a"] + 1, case["items"]).tolist(),
                            r.integers(case["lo_b"], case["hi_b"] + 1, case["items"]).tolist())]


def _trained_model():
    return np.load(os.path.join(ROOT, "models", "denoiser_64x64_32x32_n1000.npy")).astype(np.float32).reshape(-1)


_LAYERS = [(9, 32), (32, 32), (32, 32), (32, 1)]


def _untrained_model(gen):
    """He-normal weights, the last layer small, small biases: an early training step."""
    parts = []
    for l, (ci, co) in enumerate(_LAYERS):
        w = torch.randn(co * ci * 9, generator=gen, device=DEV) * math.sqrt(2.0 / (ci * 9))
        parts += [w * (0.1 if l == 3 else 1.0), 0.05 * torch.randn(co, generator=gen, device=DEV)]
    return torch.cat(parts).float()


def _train_inputs(case, seed):
    gen = _gen(seed, 31)
    g = _gamma_input(case, seed)
    target = _gamma_input(case, seed + 500009) * 0.25 + 0.5 * g
    model = _untrained_model(gen)
    m = 1e-4 * torch.randn(model.shape, generator=gen, device=DEV)
    v = 1e-7 * torch.rand(model.shape, generator=gen, device=DEV) + 1e-8
    return g, target, model, m, v


def _empty(shape, dtype):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _sums(ma, mb):
    return dict(s_ab=_empty((ma, mb), torch.int64), s_a=_empty(ma, torch.int64), s_b=_empty(mb, torch.int64))


def _regions(data, a, b, bits):
    return cpi.frames(data, bits, **a), cpi.frames(data, bits, **b)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind)
    if kind in ("step", "corr", "blocks", "stream"):
        ma, mb = case["ha"] * case["wa"], case["hb"] * case["wb"]
        img, a, b = _frames(case, seed)
        st.update(_sums(ma, mb), ma=ma, mb=mb)
        st["a"], st["b"] = _regions(img, a, b, case["bits"])
        st["gamma_f32"] = _empty((mb, ma), torch.float32)
    if kind in ("step", "corr"):
        st["frames"] = img
        st["gamma"] = _empty((ma, mb), torch.float64)
        st["ws"] = _empty(cpi.cpi_correlate_workspace_size(st["a"], st["b"], case["n"]), torch.uint8)
    elif kind == "blocks":
        st["gamma"] = _empty((ma, mb), torch.float64)
        st["frames"] = img
        st["blocks"] = []
        for i in range(0, case["n"], case["block"]):
            blk = img[i:i + case["block"]]
            st["blocks"].append((*_regions(blk, a, b, case["bits"]), blk.shape[0]))
        st["ws"] = _empty(cpi.cpi_correlate_workspace_size(st["a"], st["b"], case["block"]), torch.uint8)
    elif kind == "stream":
        st["host"] = img.cpu().pin_memory()
        st["ws"] = _empty(cpi.cpi_acq_workspace_size(st["a"], st["b"], case["block"]), torch.uint8)
    if kind in ("step", "refocus"):
        ha, wa, hb, wb, p = (case[k] for k in ("ha", "wa", "hb", "wb", "planes"))
        st["planes"] = cpi.plane_array(*_planes(p))
        st["rws"] = _empty(cpi.cpi_refocus_workspace_size(ha, wa, hb, wb, p), torch.uint8)
        st["out"] = _empty((p, ha, wa), torch.float32)
    if kind == "refocus":
        st["gamma_f32"] = _gamma_input(case, seed)
    elif kind == "refocus4d":
        ha, wa, hb, wb, p = (case[k] for k in ("ha", "wa", "hb", "wb", "planes"))
        st["gamma_f32"] = _gamma_input(case, seed)
        st["planes"] = cpi.plane4_array(*_planes4(p))
        st["rws"] = _empty(cpi.cpi_refocus4d_workspace_size(ha, wa, hb, wb, p), torch.uint8)
        st["out"] = _empty((p, ha, wa), torch.float32)
    elif kind == "batch":
        planes = cpi.plane_array(*_planes(case["planes"]))
        entries, keep = [], []
        for i, s in enumerate(_batch_shapes(case)):
            ma, mb = s["ha"] * s["wa"], s["hb"] * s["wb"]
            img, a, b = _frames(s, seed, 100 + i)
            ra, rb = _regions(img, a, b, 8)
            entries.append(dict(_sums(ma, mb), a=ra, b=rb, n_frames=s["n"], gamma=_empty((ma, mb), torch.float64),
                                gamma_f32=_empty((mb, ma), torch.float32), planes=planes,
                                refocus_out=_empty((case["planes"], s["ha"], s["wa"]), torch.float32)))
            keep.append(img)
        st.update(entries=entries, frames=keep, items=cpi.batch_items(entries))
        st["ws"] = _empty(cpi.cpi_batch_workspace_size(st["items"]), torch.uint8)
    elif kind == "denoise":
        st["gamma_in"] = _gamma_input(case, seed)
        st["model"] = torch.from_numpy(_trained_model()).to(DEV)
        st["out"] = torch.empty_like(st["gamma_in"])
        st["ws"] = _empty(cpi.cpi_denoise_workspace_size(*_shape(case)), torch.uint8)
    elif kind == "train":
        st["gamma_in"], st["target"], st["model"], st["m"], st["v"] = _train_inputs(case, seed)
        st["grad"] = torch.empty_like(st["model"])
        st["loss"] = _empty(1, torch.float32)
        st["ws"] = _empty(cpi.cpi_denoise_workspace_size(*_shape(case), training=True), torch.uint8)
    return st


def _shape(case):
    return tuple(case[k] for k in ("ha", "wa", "hb", "wb"))


# ----------------------------------------------------------------------------- one pass

def run(st):
    case, kind = st["case"], st["kind"]
    if kind in ("step", "corr"):
        cpi.cpi_correlate(st["a"], st["b"], case["n"], st["s_ab"], st["s_a"], st["s_b"], st["gamma"],
                          st["gamma_f32"], st["ws"])
        out = {k: st[k] for k in ("s_ab", "s_a", "s_b", "gamma", "gamma_f32")}
        if kind == "step":
            cpi.cpi_refocus(st["gamma_f32"], *_shape(case), st["planes"], st["out"], st["rws"])
            out["planes"] = st["out"]
        return out
    if kind == "blocks":
        for k in ("s_ab", "s_a", "s_b"):
            st[k].zero_()
        for a, b, n in st["blocks"]:
            cpi.cpi_correlate_accumulate(a, b, n, st["s_ab"], st["s_a"], st["s_b"], st["ws"])
        cpi.cpi_correlate_finalize(st["s_ab"], st["s_a"], st["s_b"], st["ma"], st["mb"], case["n"], st["gamma"],
                                   st["gamma_f32"])
        return {k: st[k] for k in ("s_ab", "s_a", "s_b", "gamma", "gamma_f32")}
    if kind == "stream":
        h = cpi.cpi_acq_begin(st["a"], st["b"], case["block"], st["s_ab"], st["s_a"], st["s_b"], st["ws"])
        for i in range(0, case["n"], case["block"]):
            blk = st["host"][i:i + case["block"]]
            cpi.cpi_acq_push(h, blk, blk.shape[0])
        cpi.cpi_acq_finalize(h, None, st["gamma_f32"])
        cpi.cpi_acq_end(h)
        return {k: st[k] for k in ("s_ab", "s_a", "s_b", "gamma_f32")}
    if kind == "refocus":
        cpi.cpi_refocus(st["gamma_f32"], *_shape(case), st["planes"], st["out"], st["rws"])
        return {"planes": st["out"]}
    if kind == "refocus4d":
        cpi.cpi_refocus4d(st["gamma_f32"], *_shape(case), st["planes"], st["out"], st["rws"])
        return {"planes": st["out"]}
    if kind == "batch":
        cpi.cpi_batch_correlate(st["items"], st["ws"])
        return [{k: e[k] for k in ("s_ab", "s_a", "s_b", "gamma", "gamma_f32", "refocus_out")} for e in st["entries"]]
    if kind == "denoise":
        cpi.cpi_denoise(st["model"], st["gamma_in"], st["out"], *_shape(case), st["ws"])
        return {"gamma": st["out"]}
    # train: one step from the state at hand (the same step each time)
    model, m, v = st["model"].clone(), st["m"].clone(), st["v"].clone()
    cpi.cpi_denoise_grad(model, st["gamma_in"], st["target"], *_shape(case), st["grad"], st["loss"], st["ws"])
    cpi.cpi_denoise_adam(model, m, v, st["grad"], 100, 2e-3)
    return {"grad": st["grad"], "loss": st["loss"], "model": model, "m": m, "v": v}


# ----------------------------------------------------------------------------- work

def _corr_work(c, gamma64, gamma32):
    ma, mb, n = c["ha"] * c["wa"], c["hb"] * c["wb"], c["n"]
    frames = n * (ma + mb) * (1.0 if c["bits"] == 8 else 0.125)
    return frames + ma * mb * (8.0 + 8.0 * gamma64 + 4.0 * gamma32) + 8.0 * (ma + mb), 2.0 * ma * mb * n


def _refocus_work(c, taps):
    ma, mb, p = c["ha"] * c["wa"], c["hb"] * c["wb"], c["planes"]
    # one interpolation along x per (plane, pixel, angular pixel); the rest is 1 / wb of it
    return 4.0 * ma * mb + 4.0 * p * ma, 2.0 * taps * p * ma * mb


def work(case):
    kind = case["kind"]
    if kind in ("corr", "blocks"):
        b, f = _corr_work(case, True, True)
    elif kind == "stream":
        b, f = _corr_work(case, False, True)
    elif kind == "step":
        b, f = _corr_work(case, True, True)
        rb, rf = _refocus_work(case, 2)
        b, f = b + 4.0 * case["planes"] * case["ha"] * case["wa"], f + rf
    elif kind == "refocus":
        b, f = _refocus_work(case, 2)
    elif kind == "refocus4d":
        b, f = _refocus_work(case, 4)
    elif kind == "batch":
        b = f = 0.0
        for s in _batch_shapes(case):
            cb, cf = _corr_work(s, True, True)
            rb, rf = _refocus_work(dict(s, planes=case["planes"]), 2)
            b, f = b + cb + 4.0 * case["planes"] * s["ha"] * s["wa"], f + cf + rf
    else:
        px = float(case["ha"] * case["wa"] * case["hb"] * case["wb"])
        macs = sum(ci * co * 9 for ci, co in _LAYERS)
        if kind == "denoise":
            b, f = 8.0 * px, 2.0 * macs * px
        else:   # forward, weight gradients, input gradients (not the first layer's)
            b, f = 8.0 * px + 4.0 * 4 * 21409, 2.0 * px * (3 * macs - _LAYERS[0][0] * _LAYERS[0][1] * 9)
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- 64-bit values

def _gamma64(case, seed, salt=0):
    """Eq. (1) from the counts.  Binary products are summed in float32 matrix
    products of at most 65536 frames, where every partial sum is an exact integer."""
    A, B = _values(case, seed, salt)
    ma, mb, n = A.shape[1], B.shape[1], A.shape[0]
    s_ab = torch.zeros((ma, mb), dtype=torch.float64, device=DEV)
    step = 65536 if case["bits"] == 1 else 8192
    dt = torch.float32 if case["bits"] == 1 else torch.float64
    for i in range(0, n, step):
        s_ab += (A[i:i + step].to(dt).T @ B[i:i + step].to(dt)).double()
    s_a, s_b = A.sum(0, dtype=torch.int64).double(), B.sum(0, dtype=torch.int64).double()
    s_ab.mul_(float(n)).addr_(s_a, s_b, alpha=-1.0).div_(float(n) * float(n))
    return s_ab


def _tap_matrix(points, size):
    """[len(points)...][size] weights of linear interpolation at `points`; outside the grid 0."""
    i = torch.floor(points)
    f = points - i
    w = torch.zeros((*points.shape, size), dtype=torch.float64, device=DEV)
    for k, v in ((i, 1.0 - f), (i + 1, f)):
        ok = (k >= 0) & (k < size)
        w.scatter_add_(-1, k.clamp(0, size - 1).long().unsqueeze(-1), torch.where(ok, v, torch.zeros_like(v)).unsqueeze(-1))
    return w


def _centred(n):
    return torch.arange(n, dtype=torch.float64, device=DEV) - 0.5 * (n - 1)


def _refocus64(g, ha, wa, hb, wb, coef):
    """Refocused stack from the float32 Gamma [hb * wb][ha * wa], in 64 bits.  coef:
    per plane (alpha, beta) or (alpha, beta, gamma, delta)."""
    G = g.double().view(hb, wb, ha, wa)
    out = torch.empty((len(coef), ha, wa), dtype=torch.float64, device=DEV)
    xa, ya, xb, yb = _centred(wa), _centred(ha), _centred(wb), _centred(hb)
    G2 = G.permute(0, 2, 1, 3).reshape(hb * ha, wb * wa) if len(coef) > 1 else None
    for p, co in enumerate(coef):
        al, be = float(co[0]), float(co[1])
        wx = _tap_matrix(al * xa[:, None] + be * (wa / wb) * xb[None] + 0.5 * (wa - 1), wa)     # [c][bc][wa]
        wy = _tap_matrix(al * ya[:, None] + be * (ha / hb) * yb[None] + 0.5 * (ha - 1), ha)     # [r][br][ha]
        if len(co) == 2:
            mx = wx.reshape(wa, wb * wa)
            my = wy.reshape(ha, hb * ha)
        else:
            ga, de = float(co[2]), float(co[3])
            vx = _tap_matrix(ga * (wb / wa) * xa[:, None] + de * xb[None] + 0.5 * (wb - 1), wb)  # [c][bc][wb]
            vy = _tap_matrix(ga * (hb / ha) * ya[:, None] + de * yb[None] + 0.5 * (hb - 1), hb)
            mx = torch.einsum("cjb,cja->cba", vx, wx).reshape(wa, wb * wa)
            my = torch.einsum("rjb,rja->rba", vy, wy).reshape(ha, hb * ha)
        u = (G2 if G2 is not None else G.permute(0, 2, 1, 3).reshape(hb * ha, wb * wa)) @ mx.T     # [hb * ha][c]
        out[p] = my @ u
    return out


def _bf16(x):
    return x.to(torch.bfloat16).to(x.dtype)


class _Stored(torch.autograd.Function):
    """A value kept in bfloat16; gradients pass unrounded."""

    @staticmethod
    def forward(ctx, x):
        return _bf16(x)

    @staticmethod
    def backward(ctx, g):
        return g


def _conv64(x, w, bias):
    """3 x 3 convolution, zero padding 1; x [b][ci][h][w] in 64 bits."""
    n, ci, h, wd = x.shape
    co = w.shape[0]
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1))
    y = bias.view(1, co, 1).expand(n, co, h * wd)
    for ky in range(3):
        for kx in range(3):
            y = y + torch.matmul(w[:, :, ky, kx], xp[:, :, ky:ky + h, kx:kx + wd].reshape(n, ci, h * wd))
    return y.view(n, co, h, wd)


def _unpack(model):
    parts, o = [], 0
    for ci, co in _LAYERS:
        w = model[o:o + co * ci * 9].view(co, ci, 3, 3)
        o += co * ci * 9
        parts.append((w, model[o:o + co]))
        o += co
    return parts


def _network64(model, x):
    """The network of include/cpi.h: bfloat16 storage of x, the weights and the
    hidden activations, everything else in 64 bits."""
    h = x
    for l, (w, b) in enumerate(_unpack(model)):
        h = _conv64(h, _Stored.apply(w), b)
        if l < 3:
            h = _Stored.apply(torch.relu(h))
    return x[:, 4] + h[:, 0]


def _stack64(g, case, scale, rows):
    """The 9-channel input of the angular rows `rows`."""
    ha, wa, hb, wb = _shape(case)
    gp = torch.zeros((hb + 2, wb + 2, ha, wa), dtype=torch.float32, device=DEV)
    gp[1:-1, 1:-1] = g.view(hb, wb, ha, wa)
    x = torch.stack([gp[r + dy, dx:dx + wb] for r in rows for dy in range(3) for dx in range(3)])
    x = x.view(len(rows), 9, wb, ha, wa).transpose(1, 2).reshape(len(rows) * wb, 9, ha, wa)
    return _bf16(x * scale).double()      # the scaled float32 value, stored in bfloat16


def _row_groups(case):
    ha, wa, hb, wb = _shape(case)
    k = max(1, int(400000 // (wb * ha * wa)))
    return [list(range(i, min(hb, i + k))) for i in range(0, hb, k)]


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind in ("step", "corr", "blocks", "stream"):
            g = _gamma64(case, seed)
            out = {"s_ab": None, "s_a": None, "s_b": None, "gamma_f32": g.T}
            if kind != "stream":
                out["gamma"] = g
            if kind == "step":
                out["planes"] = _refocus64(g.T.contiguous(), *_shape(case), list(zip(*_planes(case["planes"]))))
            return out
        if kind == "refocus":
            return {"planes": _refocus64(_gamma_input(case, seed), *_shape(case), list(zip(*_planes(case["planes"]))))}
        if kind == "refocus4d":
            return {"planes": _refocus64(_gamma_input(case, seed), *_shape(case),
                                         list(zip(*_planes4(case["planes"]))))}
        if kind == "batch":
            outs = []
            for i, s in enumerate(_batch_shapes(case)):
                g = _gamma64(s, seed, 100 + i)
                outs.append({"s_ab": None, "s_a": None, "s_b": None, "gamma": g, "gamma_f32": g.T,
                             "refocus_out": _refocus64(g.T.contiguous(), s["ha"], s["wa"], s["hb"], s["wb"],
                                                       list(zip(*_planes(case["planes"]))))})
            return outs
        if kind == "denoise":
            g = _gamma_input(case, seed)
            model = torch.from_numpy(_trained_model()).to(DEV).double()
            scale = (1.0 / g.double().square().mean().sqrt()).float()
            y = torch.cat([_network64(model, _stack64(g, case, scale, r)) for r in _row_groups(case)])
            return {"gamma": y.reshape(g.shape) / scale.double()}
    g, target, model, m, v = _train_inputs(case, seed)
    scale = (1.0 / g.double().square().mean().sqrt()).float()
    w = model.double().requires_grad_(True)
    count = float(g.numel())
    loss = 0.0
    t = target.double().view(case["hb"], case["wb"], case["ha"], case["wa"]) * scale.double()
    for rows in _row_groups(case):
        y = _network64(w, _stack64(g, case, scale, rows))
        part = (y - t[rows].reshape(y.shape)).square().sum() / count
        part.backward()
        loss += float(part)
    with torch.no_grad():
        gr = w.grad
        m1 = 0.9 * m.double() + 0.1 * gr
        v1 = 0.999 * v.double() + 0.001 * gr.square()
        w1 = model.double() - 2e-3 * (m1 / (1.0 - 0.9 ** 100)) / ((v1 / (1.0 - 0.999 ** 100)).sqrt() + 1e-8)
    return {"grad": gr, "loss": torch.tensor([loss], dtype=torch.float64), "model": w1, "m": m1, "v": v1}
