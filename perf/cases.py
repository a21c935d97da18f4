"""The work this library is measured on: what its users have it compute, through its public entry points.

A user has a point cloud on the GPU and wants a hologram of it: an amplitude hologram for display (the field and its
8-bit codes), an off-axis hologram with a reference wave, a phase-only hologram (the complex wave and its kinoform),
many frames of a video at once, a large layered scene, or one of the two wave-optics paths (Fresnel diffraction, the
wavefront-recording method).  The sizes are those of the repository's workloads, tests and benchmark; `draw` takes
others from the same ranges, odd ones among them.

Clouds follow paper_1309_2734_gb300/workloads.py (integer x, y on the pixel grid, z in metres, uniform amplitudes),
drawn on the GPU from the seed.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1309_2734_gb300 import Hologram, batch

PITCH = 8e-6
LAMBDA = 532e-9
FRAME_SIZES = ((1024, 1024), (1920, 1080), (3840, 2160))


def listed():
    return [
        # the smallest call: a preview of a small object, where launches and latency count
        dict(name="preview-256x256-n1024", kind="cloud", form="direct_sfu", width=256, height=256, points=1024,
             piston=False, reference=False, codes=True),
        # the ordinary display hologram in the FP32 direct form, with its 8-bit codes (the benchmark's workload)
        dict(name="display-1920x1080-n10000", kind="cloud", form="direct_sfu", width=1920, height=1080, points=10000,
             piston=False, reference=False, codes=True),
        # an off-axis hologram (piston of Eq. 2, tilted reference wave) in the accurate form, odd in every size
        dict(name="offaxis-1283x717-n3001", kind="cloud", form="direct_accurate", width=1283, height=717, points=3001,
             piston=True, reference=True, codes=False),
        # a dense cloud at display size on the tensor cores, FP16
        dict(name="dense-f16-1920x1080-n50000", kind="cloud", form="gemm_f16", width=1920, height=1080, points=50000,
             piston=False, reference=False, codes=False),
        # the same form family in the FP32-like accuracy class, a square panel and an odd number of points
        dict(name="dense-split-1024x1024-n20011", kind="cloud", form="gemm_split16", width=1024, height=1024,
             points=20011, piston=False, reference=False, codes=False),
        # the largest: a scene sliced into depth planes on a large panel
        dict(name="layered-4096x4096-n1000000", kind="layered", form="gemm_split16", width=4096, height=4096,
             points=1000000, planes=16),
        # the phase-only hologram the paper times, in the direct form ...
        dict(name="kinoform-sfu-1920x1080-n10000", kind="wave", form="direct_sfu", width=1920, height=1080,
             points=10000),
        # ... and with its largest point count on the tensor cores
        dict(name="kinoform-split-1920x1080-n100000", kind="wave", form="gemm_split16", width=1920, height=1080,
             points=100000),
        # the exact distance of Eq. 1 (near objects, wide angles)
        dict(name="spherical-1920x1080-n10000", kind="spherical", width=1920, height=1080, points=10000, z_lo=0.3,
             z_hi=1.0),
        # propagation of a complex plane (reconstruction, refocusing)
        dict(name="fresnel-2048x2048", kind="fresnel", width=2048, height=2048, z=0.5),
        # the wavefront-recording method for an object close to its virtual plane, with the kinoform
        dict(name="wrp-2048x2048-n100000", kind="wrp", width=2048, height=2048, points=100000),
        # frames of a holographic video, uneven in size and point count, in one call
        dict(name="video-12-frames", kind="batch", form="gemm_split16", frames=12, mix=7, n_lo=1000, n_hi=100000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi_w, hi_h):
    return _log_int(rng, lo, hi_w), _log_int(rng, lo, hi_h)


def draw(rng):
    kind = rng.choice(["cloud", "cloud", "gemm", "gemm", "layered", "wave", "spherical", "fresnel", "wrp", "batch"])
    if kind == "cloud":      # direct forms: up to the display case's number of terms
        w, h = _size(rng, 128, 2048, 2048)
        n = min(_log_int(rng, 300, 20000), int(2.07e10 / (w * h)))
        return dict(kind="cloud", form=rng.choice(["direct_sfu", "direct_sfu", "direct_accurate"]), width=w, height=h,
                    points=n, piston=rng.random() < 0.3, reference=rng.random() < 0.3, codes=rng.random() < 0.5)
    if kind == "gemm":       # tensor-core forms: up to about 5 10^11 terms
        w, h = _size(rng, 256, 4096, 4096)
        n = min(_log_int(rng, 1000, 200000), int(5e11 / (w * h)))
        return dict(kind="cloud", form=rng.choice(["gemm_f16", "gemm_split16", "gemm_bf16"]), width=w, height=h,
                    points=n, piston=rng.random() < 0.2, reference=rng.random() < 0.2, codes=False)
    if kind == "layered":
        w, h = _size(rng, 512, 4096, 4096)
        planes = rng.randint(2, 24)
        return dict(kind="layered", form=rng.choice(["gemm_split16", "gemm_f16"]), width=w, height=h,
                    points=max(_log_int(rng, 65536, 1000000), min(1000000, 5 * planes * w)), planes=planes)
    if kind == "wave":
        form = rng.choice(["direct_sfu", "gemm_f16", "gemm_split16"])
        w, h = _size(rng, 128, 2048, 2048)
        n = _log_int(rng, 300, 100000)
        return dict(kind="wave", form=form, width=w, height=h,
                    points=min(n, int((2.07e10 if form == "direct_sfu" else 2.07e11) / (w * h))))
    if kind == "spherical":
        w, h = _size(rng, 128, 2048, 2048)
        z_lo = rng.uniform(0.1, 0.5)
        return dict(kind="spherical", width=w, height=h, points=min(_log_int(rng, 300, 10000), int(2.07e10 / (w * h))),
                    z_lo=z_lo, z_hi=z_lo + rng.uniform(0.1, 0.7))
    if kind == "fresnel":
        w, h = _size(rng, 128, 4096, 4096)
        return dict(kind="fresnel", width=w, height=h, z=rng.choice([-1.0, 1.0]) * rng.uniform(0.1, 1.0))
    if kind == "wrp":
        w, h = _size(rng, 256, 2048, 2048)
        return dict(kind="wrp", width=w, height=h, points=_log_int(rng, 1000, 100000))
    n_lo = _log_int(rng, 1000, 5000)
    return dict(kind="batch", form=rng.choice(["gemm_split16", "gemm_f16"]), frames=rng.randint(3, 12),
                mix=rng.randint(100, 10 ** 6), n_lo=n_lo, n_hi=n_lo * rng.randint(2, 15))


# ---- inputs ---------------------------------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(gen, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=gen, device="cuda", dtype=torch.float32)


def _cloud(gen, width, height, n, z, a_lo, a_hi):
    """xyz [n][3], amp [n]; z: (lo, hi), or a tensor of depth planes."""
    x = torch.randint(0, width, (n,), generator=gen, device="cuda").float()
    y = torch.randint(0, height, (n,), generator=gen, device="cuda").float()
    if torch.is_tensor(z):
        z = z[torch.randint(0, len(z), (n,), generator=gen, device="cuda")]
    else:
        z = _uniform(gen, n, *z)
    return torch.stack([x, y, z], 1).contiguous(), _uniform(gen, n, a_lo, a_hi)


def _frames(case):
    """Size and point count of each frame of a video, from the case alone."""
    rng = random.Random(case["mix"])
    return [(*rng.choice(FRAME_SIZES), _log_int(rng, case["n_lo"], case["n_hi"])) for _ in range(case["frames"])]


Z_WRP = 0.5
REFERENCE = (0.011, -0.007, 0.6)   # sines of the tilt and a phase offset, rad


def _inputs(case, seed):
    gen, kind = _generator(seed), case["kind"]
    if kind == "layered":
        planes = 0.2 + 0.8 * torch.arange(case["planes"], device="cuda", dtype=torch.float64) / (case["planes"] - 1)
        return _cloud(gen, case["width"], case["height"], case["points"], planes.float(), 0.1, 1.0)
    if kind == "fresnel":
        return torch.randn((2, case["height"], case["width"]), generator=gen, device="cuda")
    if kind == "batch":
        return [_cloud(gen, w, h, n, (0.3, 1.0), 0.5, 1.0) + (w, h, PITCH, LAMBDA) for w, h, n in _frames(case)]
    z = {"wrp": (Z_WRP + 0.002, Z_WRP + 0.010), "spherical": (case.get("z_lo"), case.get("z_hi"))}.get(kind, (0.3, 1.0))
    return _cloud(gen, case["width"], case["height"], case["points"], z, 0.5, 1.0)


def prepare(case, seed):
    kind = case["kind"]
    w, h = (64, 64) if kind == "batch" else (case["width"], case["height"])
    holo = Hologram(w, h, PITCH, LAMBDA, form=case.get("form", "direct_sfu"))
    if kind == "spherical":
        holo.set_phase_model("spherical")
    if case.get("piston"):
        holo.set_phase_model("fresnel_piston")
    if case.get("reference"):
        holo.set_reference(*REFERENCE)
    state = dict(case=case, holo=holo, inputs=_inputs(case, seed))
    if kind == "batch":   # a video player's frame buffers
        state["outs"] = [torch.empty((c[3], c[2]), device="cuda") for c in state["inputs"]]
    return state


def run(state):
    case, holo, inputs = state["case"], state["holo"], state["inputs"]
    kind = case["kind"]
    if kind == "batch":
        return {"fields": batch(holo, inputs, state["outs"])}
    if kind == "fresnel":
        return {"plane": holo.fresnel(inputs, case["z"])}
    if kind == "wrp":
        wave = holo.wrp(*inputs, Z_WRP)
        return {"wave": wave, "codes": holo.kinoform8(wave)}
    if kind == "wave":
        wave = holo.wave(*inputs)
        return {"wave": wave, "codes": holo.kinoform8(wave)}
    field = holo.point_cloud(*inputs)
    return {"field": field, "codes": holo.quantize8(field)} if case.get("codes") else {"field": field}


# ---- what a pass cannot do without ------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "batch":
        frames = _frames(case)
        return {"bytes": sum(16 * n + 4 * w * h for w, h, n in frames), "flops": sum(4 * w * h * n for w, h, n in frames)}
    w, h, n = case["width"], case["height"], case.get("points", 0)
    px = w * h
    if kind == "fresnel":   # the plane in and out; two transforms of the padded grid, 5 L log2 L each
        lx, ly = (1 << max(1, (2 * s - 2)).bit_length() for s in (w, h))
        return {"bytes": 16 * px, "flops": 10.0 * lx * ly * math.log2(lx * ly)}
    if kind == "wrp":       # the wave and its codes; the terms inside the windows and the transforms
        window = math.pi * (0.006 * LAMBDA / (2 * PITCH) / PITCH) ** 2
        lx, ly = (1 << max(1, (2 * s - 2)).bit_length() for s in (w, h))
        return {"bytes": 16 * n + 8 * px + px, "flops": 8.0 * n * window + 10.0 * lx * ly * math.log2(lx * ly)}
    if kind == "wave":      # four multiply-adds a term would be eight flops
        return {"bytes": 16 * n + 8 * px + px, "flops": 8.0 * px * n}
    if kind == "spherical":  # the exact distance does not factor: the phase and the cosine of each term
        return {"bytes": 16 * n + 4 * px, "flops": 8.0 * px * n}
    if kind == "layered":   # points of one plane and column share their column factor
        groups = min(n, case["planes"] * w)
        return {"bytes": 16 * n + 4 * px, "flops": 4.0 * px * groups + 4.0 * h * n}
    codes = px if case["codes"] else 0
    return {"bytes": 16 * n + 4 * px + codes, "flops": 4.0 * px * n}


def tolerance(case):
    # about four times the distance from `exact` at the listed sizes: 6e-7 to 7e-7 direct (9e-7 spherical, 1.0e-6 with
    # the two transforms of the recording method), 2.9e-6 to 3.3e-6 split FP16, 2.6e-4 to 3e-4 FP16, 2.1e-3 BF16
    if case["kind"] in ("spherical", "wrp"):
        rel = 4e-6
    else:
        rel = {"direct_sfu": 3e-6, "direct_accurate": 3e-6, "gemm_split16": 1.2e-5, "gemm_f16": 1.2e-3,
               "gemm_bf16": 9e-3}[case.get("form", "direct_sfu")]
    # codes: a value next to a step of the quantiser falls to either side (2e-5 to 5e-5 of them against `exact`; one
    # pixel of the smallest field drawn is 6e-5)
    if case["kind"] in ("wave", "wrp"):
        return {"rel": rel, "differ": min(0.01, max(2e-4, 40 * rel))}
    return {"rel": rel, "differ": 3e-4} if case.get("codes") else {"rel": rel}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------

def _angles(turns):
    return (2 * math.pi) * (turns - torch.round(turns))


def _separable(case, xyz, amp, both):
    """sum_j A_j exp(i phase), real part [H][W] or both parts [2][H][W], as products of column and row factors."""
    w, h = case["width"], case["height"]
    m = torch.arange(w, device="cuda", dtype=torch.float64)
    r = torch.arange(h, device="cuda", dtype=torch.float64)
    out = torch.zeros((2 if both else 1, h, w), device="cuda", dtype=torch.float64)
    px = lambda d, c: c[:, None] * d * d  # noqa: E731
    for a in range(0, len(amp), 8192):
        x, y, z = xyz[a:a + 8192].double().unbind(1)
        c = PITCH * PITCH / (2 * LAMBDA * z)
        tx, ty = px(m[None] - x[:, None], c), px(r[None] - y[:, None], c)
        if case.get("piston"):
            tx = tx + (z / LAMBDA)[:, None]
        if case.get("reference"):
            sx, sy, ph = REFERENCE
            tx = tx + m[None] * (PITCH * sx / LAMBDA) + ph / (2 * math.pi)
            ty = ty + r[None] * (PITCH * sy / LAMBDA)
        col, row = _angles(tx), _angles(ty)
        A = amp[a:a + 8192].double()[:, None]
        left = torch.cat([A * torch.cos(row), A * torch.sin(row)])
        cx, sx_ = torch.cos(col), torch.sin(col)
        out[0] += left.T @ torch.cat([cx, -sx_])
        if both:
            out[1] += left.T @ torch.cat([sx_, cx])
    return out if both else out[0]


def _layered(case, xyz, amp):
    w, h = case["width"], case["height"]
    m = torch.arange(w, device="cuda", dtype=torch.float64)
    r = torch.arange(h, device="cuda", dtype=torch.float64)
    out = torch.zeros((h, w), device="cuda", dtype=torch.float64)
    for z in torch.unique(xyz[:, 2]):
        here = xyz[:, 2] == z
        x, y, A = xyz[here, 0].long(), xyz[here, 1].double(), amp[here].double()
        c = PITCH * PITCH / (2 * LAMBDA * z.double())
        rows = torch.zeros((2, w, h), device="cuda", dtype=torch.float64)
        for a in range(0, len(A), 16384):
            ang = _angles(c * (r[None] - y[a:a + 16384, None]) ** 2)
            rows[0].index_add_(0, x[a:a + 16384], A[a:a + 16384, None] * torch.cos(ang))
            rows[1].index_add_(0, x[a:a + 16384], A[a:a + 16384, None] * torch.sin(ang))
        col = _angles(c * (m[:, None] - m[None]) ** 2)
        out += rows[0].T @ torch.cos(col) - rows[1].T @ torch.sin(col)
    return out


def _spherical(case, xyz, amp):
    w, h = case["width"], case["height"]
    m = torch.arange(w, device="cuda", dtype=torch.float64) * PITCH
    r = torch.arange(h, device="cuda", dtype=torch.float64) * PITCH
    out = torch.zeros((h, w), device="cuda", dtype=torch.float64)
    step = max(1, int(2e8 / (w * h)))
    for a in range(0, len(amp), step):
        x, y, z = (v[:, None, None] for v in xyz[a:a + step].double().unbind(1))
        t = torch.sqrt((m[None, None] - x * PITCH) ** 2 + (r[None, :, None] - y * PITCH) ** 2 + z * z) / LAMBDA
        t -= torch.round(t)
        out += (torch.cos(t.mul_(2 * math.pi)) * amp[a:a + step].double()[:, None, None]).sum(0)
    return out


def _fresnel(plane, z):
    """Eq. 10 on the grid: the linear convolution with exp(i pi p^2 (k^2 + l^2)/(lambda z)), by padded transforms."""
    h, w = plane.shape
    ly, lx = 2 * h, 2 * w
    chirp = lambda n, s: torch.exp(1j * _angles(PITCH * PITCH / (2 * LAMBDA * z) * s * s))  # noqa: E731
    k = lambda n: torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)  # noqa: E731
    spec = torch.fft.fft(chirp(ly, k(ly)))[:, None] * torch.fft.fft(chirp(lx, k(lx)))[None]
    pad = torch.zeros((ly, lx), device="cuda", dtype=torch.complex128)
    pad[:h, :w] = plane
    out = torch.fft.ifft2(torch.fft.fft2(pad).mul_(spec))[:h, :w]
    turns = z / LAMBDA
    front = complex(math.cos(2 * math.pi * (turns - round(turns))), math.sin(2 * math.pi * (turns - round(turns))))
    return out * (front * PITCH * PITCH / (1j * LAMBDA * z))


def _wrp_record(case, xyz, amp):
    """Each point inside its window: squared radius floor(w^2), w = d s / sqrt(1 - s^2) / p, s = lambda / (2 p)."""
    w, h = case["width"], case["height"]
    out = torch.zeros((2, h * w), device="cuda", dtype=torch.float64)
    s = LAMBDA / (2 * PITCH)
    for a in range(0, len(amp), 4096):
        x, y, z = xyz[a:a + 4096].double().unbind(1)
        d = z - Z_WRP
        w2 = torch.floor((d * s / math.sqrt(1 - s * s) / PITCH) ** 2)
        R = int(math.sqrt(float(w2.max())))
        o = torch.arange(-R, R + 1, device="cuda", dtype=torch.float64)
        r2 = o[None, :, None] ** 2 + o[None, None, :] ** 2
        m, n = x[:, None, None] + o[None, None, :], y[:, None, None] + o[None, :, None]
        inside = (r2 <= w2[:, None, None]) & (m >= 0) & (m < w) & (n >= 0) & (n < h)
        ang = _angles((PITCH * PITCH / (2 * LAMBDA * d))[:, None, None] * r2)
        A = amp[a:a + 4096].double()[:, None, None]
        at = (n * w + m).long()[inside]
        out[0].index_add_(0, at, (A * torch.cos(ang))[inside])
        out[1].index_add_(0, at, (A * torch.sin(ang))[inside])
    return torch.complex(out[0], out[1]).view(h, w)


def exact(case, seed):
    kind, inputs = case["kind"], _inputs(case, seed)
    if kind == "batch":
        return {"fields": [_separable(dict(width=w, height=h), xyz, amp, False) for xyz, amp, w, h, _, _ in inputs]}
    if kind == "fresnel":
        o = _fresnel(torch.complex(inputs[0].double(), inputs[1].double()), case["z"])
        return {"plane": torch.stack([o.real, o.imag])}
    if kind == "wrp":
        o = _fresnel(_wrp_record(case, *inputs), Z_WRP)
        return {"wave": torch.stack([o.real, o.imag]), "codes": None}
    if kind == "wave":
        return {"wave": _separable(case, *inputs, True), "codes": None}
    field = {"layered": _layered, "spherical": _spherical}.get(kind)
    field = field(case, *inputs) if field else _separable(case, *inputs, False)
    return {"field": field, "codes": None} if case.get("codes") else {"field": field}
