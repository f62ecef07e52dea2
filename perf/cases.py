"""The work that users of the framework have it do, as timed cases.

A migration user models records (rbc_model), migrates shots (rbc_rtm_shot, rbc_rtm_storage) and stacks their images
(rbc_image_stack), one shot at a time or in batches of uneven apertures (rbc_batch_rtm); an inversion user evaluates
the misfit and its gradient (fwi.fwi_misfit); an imaging user denoises single images and volumes (denoise.Denoiser)
and trains the network (rbc_cnn_forward / mse / backward).  Grids, spacings, velocities, wavelets and geometries are
those of the repository's workload presets, with shorter records where a full one would only repeat the same step.
"""
import math

import numpy as np
import torch

import paper_2204_03380_gb300 as R
from paper_2204_03380_gb300 import denoise, fwi

# spacing (m), time step (s), peak frequency (Hz), velocity range and random-boundary cap (m/s) of the presets
PHYS = {
    "small2d": dict(h=10.0, dt=1e-3, f=15.0, v_min=1500.0, v_max=3500.0, v_lo=1500.0, v_hi=4500.0, cap=3500.0),
    "survey2d": dict(h=4.0, dt=0.4e-3, f=25.0, v_min=1500.0, v_max=5500.0, v_lo=1500.0, v_hi=5500.0, cap=5500.0),
    "batch2d": dict(h=5.0, dt=0.5e-3, f=25.0, v_min=1500.0, v_max=4000.0, v_lo=1500.0, v_hi=4000.0, cap=4000.0),
    "shot3d": dict(h=10.0, dt=1e-3, f=15.0, v_min=1500.0, v_max=4500.0, v_lo=1500.0, v_hi=4500.0, cap=4500.0),
}
EPS_REL = 1e-2                 # water level of the image ratio
C = (1.6, -0.2, 8.0 / 315.0, -1.0 / 560.0)   # 8th-order second-derivative weights c1..c4
C0 = -2.0 * sum(C)


def listed():
    return [
        # modeling one record on the smallest preset (three layers, 10 m cells): launches and latency
        dict(name="model2d_small", kind="model", phys="small2d", nx=200, nz=200, nb=50, nt=1000, fs=0, step=1),
        # synthetic records for a survey: the 2-D survey preset's grid, receivers every fifth column
        dict(name="model2d_survey", kind="model", phys="survey2d", nx=2301, nz=751, nb=60, nt=1500, fs=0, step=5),
        # one migrated shot of the smallest preset, stacked
        dict(name="rtm2d_small", kind="rtm", phys="small2d", nx=200, nz=200, nb=50, nt=1000, fs=0, step=1),
        # one shot of the 240-shot survey, migrated and stacked: the benchmark's default workload
        dict(name="rtm2d_survey", kind="rtm", phys="survey2d", nx=2301, nz=751, nb=60, nt=2000, fs=0, step=5),
        # a small ragged 3-D target volume
        dict(name="rtm3d_target", kind="rtm3", phys="shot3d", nx=151, ny=110, nz=93, nb=20, nt=300, step=3),
        # the 3-D preset's grid (580 x 580 x 380 padded), the largest migration
        dict(name="rtm3d_full", kind="rtm3", phys="shot3d", nx=500, ny=500, nz=300, nb=40, nt=240, step=2),
        # migration with the wavefield kept every Nyquist stride instead of reconstructed
        dict(name="storage2d_survey", kind="storage", phys="survey2d", nx=2301, nz=751, nb=60, nt=1000, fs=0, step=5),
        # a batch of uneven apertures (400 to 1200 columns, 600 rows)
        dict(name="batch2d_uneven", kind="batch", phys="batch2d", nshots=16, wmin=400, wmax=1200, nz=600, nb=50, nt=600),
        # one misfit and gradient of the inversion preset: 4 shots on 300 x 300 cells
        dict(name="fwi2d", kind="fwi", phys="small2d", nx=300, nz=300, nb=50, nt=1000, nshots=4),
        # one image through the denoiser: the smallest call
        dict(name="denoise_image", kind="denoise", n=1, H=200, W=200),
        # a 3-D image denoised slice by slice (one slab of the 800 x 800 x 400 volume)
        dict(name="denoise_volume", kind="volume", nz=400, ny=64, nx=800),
        # one training batch of the denoiser: forward, loss, gradients (batch of 8, 512 x 512 images)
        dict(name="denoise_train", kind="train", n=8, H=512, W=512),
    ]


def draw(rng):
    def lu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["model", "rtm", "rtm", "rtm3", "storage", "batch", "fwi", "denoise", "volume", "train"])
    if kind in ("model", "rtm", "storage"):
        return dict(kind=kind, phys=rng.choice(["small2d", "survey2d"]), nx=lu(40, 2400), nz=lu(40, 1000),
                    nb=rng.randint(6, 60), nt=lu(200, 2000 if kind != "storage" else 1000), fs=int(rng.random() < 0.25),
                    step=rng.randint(1, 5))
    if kind == "rtm3":
        return dict(kind=kind, phys="shot3d", nx=lu(20, 320), ny=lu(20, 320), nz=lu(16, 200), nb=rng.randint(5, 30),
                    nt=rng.randint(60, 240), step=rng.randint(1, 4))
    if kind == "batch":
        w = lu(80, 800)
        return dict(kind=kind, phys="batch2d", nshots=rng.randint(3, 20), wmin=w, wmax=min(1200, w + lu(20, 600)),
                    nz=lu(60, 600), nb=rng.randint(8, 50), nt=lu(150, 600))
    if kind == "fwi":
        return dict(kind=kind, phys="small2d", nx=lu(60, 500), nz=lu(60, 400), nb=rng.randint(10, 50),
                    nt=lu(400, 1000), nshots=rng.randint(1, 6))
    if kind == "denoise":
        return dict(kind=kind, n=lu(1, 32), H=lu(64, 600), W=lu(64, 600))
    if kind == "volume":
        return dict(kind=kind, nz=lu(100, 400), ny=lu(8, 96), nx=lu(100, 800))
    return dict(kind=kind, n=lu(1, 8), H=lu(64, 512), W=lu(64, 512))


# ------------------------------------------------------------------- inputs --
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt=0):
    return torch.Generator().manual_seed(1_000_003 * (seed + 1) + salt)


def _uniform(g, n, lo, hi):
    return (lo + (hi - lo) * torch.rand(n, generator=g, dtype=torch.float64)).tolist()


def _velocity(ph, shape, seed, smooth=False):
    """Layers with dips and a lateral undulation (a migration model: the same as a smooth gradient), fp32."""
    g, dev = _gen(seed, 1), _device()
    nz, nx = shape[0], shape[-1]
    z = torch.arange(nz, device=dev, dtype=torch.float32).reshape((-1,) + (1,) * (len(shape) - 1))
    x = torch.arange(nx, device=dev, dtype=torch.float32).reshape((1,) * (len(shape) - 1) + (-1,))
    nl = 8
    depth = sorted(_uniform(g, nl - 1, 0.08, 0.92))
    dip, amp, ph0 = _uniform(g, nl - 1, -0.06, 0.06), _uniform(g, nl - 1, 0.0, 0.03), _uniform(g, nl - 1, 0.0, 6.28)
    lat = x / nx
    if len(shape) == 3:
        lat = lat + 0.7 * torch.arange(shape[1], device=dev, dtype=torch.float32).reshape(1, -1, 1) / shape[1]
    v = torch.zeros(shape, device=dev)
    width = 0.05 * nz if smooth else 0.35
    for d, s, a, p in zip(depth, dip, amp, ph0):
        face = nz * (d + s * (lat - 0.5) + a * torch.sin(6.28 * lat + p))
        v += torch.sigmoid((z - face) / width) if smooth else (z >= face).float()
    return (ph["v_min"] + (ph["v_max"] - ph["v_min"]) * v / (nl - 1)).contiguous()


def _ricker(ph, nt):
    t = np.arange(nt) * ph["dt"] - 1.5 / ph["f"]
    x = (math.pi * ph["f"] * t) ** 2
    return torch.tensor((1.0 - 2.0 * x) * np.exp(-x), dtype=torch.float32, device=_device())


def _record(ph, src, rec, nt, seed):
    """A record with a direct wave, a few reflections of hyperbolic moveout and weak noise: (nrec, nt + 1) fp32."""
    dev = _device()
    g = _gen(seed, 2)
    d = torch.tensor(np.linalg.norm((rec - src).astype(np.float64), axis=1) * ph["h"], dtype=torch.float32, device=dev)
    t = torch.arange(nt + 1, device=dev, dtype=torch.float32) * ph["dt"]
    out = torch.empty((len(rec), nt + 1), dtype=torch.float32, device=dev)
    gd = torch.Generator(device=dev).manual_seed(seed + 17)
    out.normal_(0.0, 1e-4, generator=gd)
    span = nt * ph["dt"]
    for k, (t0, vel, amp) in enumerate(zip(_uniform(g, 5, 0.05, 0.95), _uniform(g, 5, 1600.0, 3000.0),
                                           _uniform(g, 5, -0.02, 0.02))):
        t0 = 0.0 if k == 0 else t0 * span
        arrive = torch.sqrt(t0 ** 2 + (d / vel) ** 2) + 1.5 / ph["f"]
        u = (math.pi * ph["f"] * (t[None, :] - arrive[:, None])) ** 2
        out += (0.05 if k == 0 else amp) / (1.0 + d[:, None] / 500.0) * (1.0 - 2.0 * u) * torch.exp(-u)
    return out


def _geometry(case):
    """Grid arguments, source node and receiver nodes (padded frame) of a single-shot case."""
    nb = case["nb"]
    top = 4 if case.get("fs") else nb
    nx, ny, nz, step = case["nx"], case.get("ny", 1), case["nz"], case["step"]
    depth = top + min(1, nz - 1)
    if "ny" in case:
        xs, ys = np.arange(0, nx, step) + nb, np.arange(0, ny, step) + nb
        X, Y = np.meshgrid(xs, ys, indexing="xy")
        rec = np.stack([X.ravel(), Y.ravel(), np.full(X.size, depth)], 1).astype(np.int32)
        src = np.array([nx // 2 + nb, ny // 2 + nb, depth], np.int32)
    else:
        xs = np.arange(0, nx, step) + nb
        rec = np.stack([xs, np.zeros_like(xs), np.full_like(xs, depth)], 1).astype(np.int32)
        src = np.array([nx // 2 + nb, 0, depth], np.int32)
    return src, rec


def _grid(case, nx=None):
    ph = PHYS[case["phys"]]
    return R.make_grid(3 if "ny" in case else 2, nx or case["nx"], case.get("ny", 1), case["nz"], case["nb"], ph["h"],
                       ph["dt"], case["nt"], case.get("fs", 0))


def _interior(case, nx=None):
    return (case["nz"], case["ny"], case["nx"]) if "ny" in case else (case["nz"], nx or case["nx"])


class _Handle:
    """A context or batch that is destroyed with the state that holds it."""

    def __init__(self, h, free):
        self.h, self.free = h, free

    def __del__(self):
        self.free(self.h)


def _build(case, v, seed, nx=None):
    ph, g = PHYS[case["phys"]], _grid(case, nx)
    a = torch.empty(g.padded, dtype=torch.float32, device=_device())
    R.rbc_build_velocity(g, v, ph["v_lo"], ph["v_hi"], ph["cap"], seed + 1, 0, None, a)
    return g, a


def _batch_shots(case, seed):
    """(width, column offset, source, receivers) of every shot over a model four times the widest aperture."""
    g = _gen(seed, 3)
    nxs = 4 * case["wmax"]
    shots = []
    for s in range(case["nshots"]):
        width = int(torch.randint(case["wmin"], case["wmax"] + 1, (1,), generator=g))
        off = int(min(max(round((s + 0.5) * nxs / case["nshots"] - width / 2), 0), nxs - width))
        xs = np.arange(0, width, 2) + case["nb"]
        rec = np.stack([xs, np.zeros_like(xs), np.full_like(xs, case["nb"] + 1)], 1).astype(np.int32)
        shots.append((width, off, np.array([width // 2 + case["nb"], 0, case["nb"] + 1], np.int32), rec))
    return nxs, shots


def _fwi_inputs(case, seed):
    """True and starting interior velocity, sources, receivers and observed records of the inversion."""
    ph, nx, nz, nb, nt = PHYS[case["phys"]], case["nx"], case["nz"], case["nb"], case["nt"]
    v0, vt = _velocity(ph, (nz, nx), seed, smooth=True), _velocity(ph, (nz, nx), seed)
    xs = np.arange(0, nx, 2) + nb
    rec = np.stack([xs, np.zeros_like(xs), np.full_like(xs, nb + 1)], 1).astype(np.int32)
    srcs = [np.array([int((k + 0.5) * nx / case["nshots"]) + nb, 0, nb + 1], np.int32) for k in range(case["nshots"])]
    wav = _ricker(ph, nt)
    a = _coef(case, vt, seed).double()
    dobs = [_model64(a, wav, s, rec, nt, 1.0).float() for s in srcs]
    return v0, srcs, rec, wav, dobs


def _params(seed):
    """Network parameters as training leaves them: He-scaled weights, small biases, a small last layer."""
    g = _gen(seed, 4)
    out = []
    for l, (ci, co) in enumerate([(1, 32), (32, 32), (32, 32), (32, 32), (32, 1)]):
        out.append(torch.randn(9 * co * ci, generator=g, dtype=torch.float64) * math.sqrt(2.0 / (9 * ci)) *
                   (0.1 if l == 4 else 1.0))
        out.append(torch.randn(co, generator=g, dtype=torch.float64) * 0.05)
    return torch.cat(out).float().to(_device())


def _images(shape, seed):
    """Images scaled to unit RMS: bands along the second-last axis under noise."""
    dev = _device()
    g = torch.Generator(device=dev).manual_seed(seed + 29)
    x = torch.randn(shape, generator=g, device=dev)
    z = torch.arange(shape[-2], device=dev, dtype=torch.float32)[:, None]
    c = torch.arange(shape[-1], device=dev, dtype=torch.float32)[None, :]
    x = 0.5 * x + torch.sin(0.21 * z + 0.013 * c) * torch.sin(0.05 * z + 1.0)
    return (x / x.pow(2).mean().sqrt()).contiguous()


# --------------------------------------------------------------------- cases --
def prepare(case, seed):
    kind, dev = case["kind"], _device()
    st = dict(case=case)
    if kind in ("model", "rtm", "rtm3", "storage"):
        ph = PHYS[case["phys"]]
        src, rec = _geometry(case)
        g, a = _build(case, _velocity(ph, _interior(case), seed, smooth=kind != "model"), seed)
        st.update(g=g, src=src, rec=rec, wav=_ricker(ph, case["nt"]), ctx=_Handle(R.rbc_create(g, a), R.rbc_destroy))
        if kind == "model":
            st["seis"] = torch.empty((len(rec), case["nt"] + 1), device=dev)
        else:
            st["seis"] = _record(ph, src, rec, case["nt"], seed)
            st["num"], st["den"] = torch.empty(g.interior, device=dev), torch.empty(g.interior, device=dev)
            st["image"] = torch.zeros(g.interior, device=dev)
        if kind == "storage":
            st["k"] = R.rbc_nyquist_stride(ph["dt"], 2.5 * ph["f"])
            st["store"] = torch.empty(R.rbc_storage_bytes(g, st["k"]) // 4, device=dev)
    elif kind == "batch":
        ph = PHYS[case["phys"]]
        nxs, shots = _batch_shots(case, seed)
        v = _velocity(ph, (case["nz"], nxs), seed, smooth=True)
        a_list, arr = [], []
        for s, (width, off, src, rec) in enumerate(shots):
            a_list.append(_build(case, v[:, off:off + width].contiguous(), seed + s, width)[1])
            arr.append(dict(src=src, rec=rec, off_x=off, seis=_record(ph, src, rec, case["nt"], seed + s)))
        st.update(shots=arr, wav=_ricker(ph, case["nt"]), image=torch.zeros((case["nz"], nxs), device=dev),
                  batch=_Handle(R.rbc_batch_create(_grid(case, 1), [s[0] for s in shots], a_list),
                                R.rbc_batch_destroy))
    elif kind == "fwi":
        ph = PHYS[case["phys"]]
        v0, srcs, rec, wav, dobs = _fwi_inputs(case, seed)
        st.update(g=_grid(case), v=v0.requires_grad_(True), srcs=srcs, rec=rec, wav=wav, dobs=dobs,
                  rbc=(ph["v_lo"], ph["v_hi"], ph["cap"], seed + 1))
    elif kind == "train":
        n, H, W = case["n"], case["H"], case["W"]
        x = _images((n, H, W), seed)
        st.update(p=_params(seed), x=x, t=x + 0.3 * _images((n, H, W), seed + 1), y=torch.empty_like(x),
                  dy=torch.empty_like(x), grad=torch.empty(R.rbc_cnn_param_count(), device=dev),
                  loss=torch.empty(1, dtype=torch.float64, device=dev),
                  ws=torch.empty(R.rbc_cnn_workspace_bytes(n, H, W), dtype=torch.uint8, device=dev))
    else:
        st["net"] = denoise.Denoiser(_params(seed), device=dev)
        st["x"] = _images((case["n"], case["H"], case["W"]) if kind == "denoise" else
                          (case["nz"], case["ny"], case["nx"]), seed)
    return st


def run(st):
    kind = st["case"]["kind"]
    if kind == "model":
        R.rbc_model(st["ctx"].h, st["src"], st["wav"], st["rec"], st["seis"])
        return st["seis"]
    if kind in ("rtm", "rtm3", "storage"):
        if kind == "storage":
            R.rbc_rtm_storage(st["ctx"].h, st["src"], st["wav"], st["rec"], st["seis"], st["k"], st["store"],
                              R.RBC_ZERO_FIRST, st["num"], st["den"])
        else:
            R.rbc_rtm_shot(st["ctx"].h, st["src"], st["wav"], st["rec"], st["seis"],
                           R.RBC_REINJECT_SOURCE | R.RBC_ZERO_FIRST, st["num"], st["den"])
        st["image"].zero_()
        R.rbc_image_stack(st["g"], st["num"], st["den"], EPS_REL, 0, 0, st["g"], st["image"])
        out = dict(num=st["num"], den=st["den"], image=st["image"])
        if kind == "storage":
            out["store"] = st["store"]
        return out
    if kind == "batch":
        st["image"].zero_()
        R.rbc_batch_rtm(st["batch"].h, st["shots"], st["wav"], R.RBC_REINJECT_SOURCE, EPS_REL, st["image"])
        return st["image"]
    if kind == "fwi":
        st["v"].grad = None
        J = fwi.fwi_misfit(st["v"], st["g"], st["srcs"], st["wav"], st["rec"], st["dobs"], st["rbc"])
        J.backward()
        return dict(misfit=J.detach(), grad=st["v"].grad)
    if kind == "denoise":
        return st["net"](st["x"])
    if kind == "volume":
        return st["net"].denoise_volume(st["x"])
    st["loss"].zero_()
    st["grad"].zero_()
    R.rbc_cnn_forward(st["p"], st["x"], st["y"], st["ws"])
    R.rbc_cnn_mse(st["y"], st["t"], st["dy"], st["loss"])
    R.rbc_cnn_backward(st["p"], st["dy"], st["grad"], st["ws"])
    return dict(y=st["y"], loss=st["loss"], grad=st["grad"])


def work(case):
    """What a pass cannot do without: its inputs and outputs once, and the arithmetic of its equations."""
    kind = case["kind"]
    if kind in ("denoise", "volume", "train"):
        px = case["n"] * case["H"] * case["W"] if kind != "volume" else case["nz"] * case["ny"] * case["nx"]
        fwd = 2 * 9 * (32 + 3 * 1024 + 32) * px
        if kind == "train":   # data gradients of four layers, weight gradients of five
            return dict(bytes=12 * px + 8 * 28000, flops=fwd + 2 * 9 * (3 * 1024 + 32) * px + fwd)
        return dict(bytes=8 * px + 4 * 28000, flops=fwd)
    nt, nb, nz = case["nt"], case["nb"], case["nz"]
    if kind == "batch":
        mean = (case["wmin"] + case["wmax"]) / 2
        nodes, inner = case["nshots"] * (mean + 2 * nb) * (nz + 2 * nb), case["nshots"] * mean * nz
        recs = case["nshots"] * mean / 2
        return dict(bytes=int(4 * (nodes + recs * (nt + 1) + 4 * case["wmax"] * nz)),
                    flops=int(nt * (3 * 26 * nodes + 4 * inner)))
    if kind == "fwi":
        nodes, recs = (case["nx"] + 2 * nb) * (nz + 2 * nb), case["nx"] // 2
        return dict(bytes=int(4 * (2 * case["nx"] * nz + case["nshots"] * recs * (nt + 1))),
                    flops=int(case["nshots"] * nt * (3 * 26 + 2) * nodes))
    nodes, inner = (nz + nb + (4 if case.get("fs") else nb)) * (case["nx"] + 2 * nb), nz * case["nx"]
    per, recs = 26, (case["nx"] + case["step"] - 1) // case["step"]
    if kind == "rtm3":
        nodes, inner, per = nodes * (case["ny"] + 2 * nb), inner * case["ny"], 34
        recs *= (case["ny"] + case["step"] - 1) // case["step"]
    if kind == "model":
        return dict(bytes=4 * (nodes + nt + recs * (nt + 1)), flops=nt * per * nodes)
    ins = nodes + nt + recs * (nt + 1)
    if kind == "storage":
        k = int(1.0 / (5.0 * PHYS[case["phys"]]["f"]) / PHYS[case["phys"]]["dt"] + 1e-9)
        levels = nt // k + 1
        return dict(bytes=4 * (ins + 3 * inner + 2 * levels * inner), flops=nt * 2 * per * nodes + 4 * levels * inner)
    return dict(bytes=4 * (ins + 3 * inner), flops=nt * (3 * per * nodes + 4 * inner))


# ------------------------------------------------------------ 64-bit values --
def _sm64(seed, j):
    """splitmix64 as a counter generator (wrapping 64-bit arithmetic), uniform in [0, 1)."""
    def signed(c):
        return c - (1 << 64) if c >= 1 << 63 else c

    def shr(z, n):
        return (z >> n) & ((1 << (64 - n)) - 1)

    z = j * signed(0x9E3779B97F4A7C15) + seed
    z = (z ^ shr(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * signed(0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 11).double() * 2.0 ** -53


def _coef(case, v, seed, nx=None):
    """Padded (v dt / h)^2 with the random boundary of mode 0, rounded once to fp32."""
    ph, nb, dev = PHYS[case["phys"]], case["nb"], v.device
    top = 4 if case.get("fs") else nb
    n = list(v.shape)
    lead = [top] + [nb] * (v.dim() - 1)
    total = [n[0] + top + nb] + [m + 2 * nb for m in n[1:]]
    dist, vp = None, v.double()
    for ax in range(v.dim()):
        i = torch.arange(total[ax], device=dev)
        q = torch.where(i < lead[ax], lead[ax] - i, torch.where(i >= lead[ax] + n[ax], i - (lead[ax] + n[ax] - 1), 0 * i))
        q = q.reshape([-1 if k == ax else 1 for k in range(v.dim())])
        dist = q if dist is None else torch.maximum(dist, q)
        vp = vp.index_select(ax, (i - lead[ax]).clamp(0, n[ax] - 1))
    j = torch.arange(int(np.prod(total)), device=dev).reshape(total)
    d = dist.double()
    g, u = (nb - d) / (nb - 1), (d - 1) / (nb - 1)
    hh = torch.exp(-120.0 * u * u)
    lo, up = torch.minimum(hh, g), torch.maximum(hh, g)
    c = lo + (up - lo) * _sm64(seed + 1, 2 * j + 1)
    vr = ph["v_lo"] + (ph["v_hi"] - ph["v_lo"]) * _sm64(seed + 1, 2 * j + 2)
    vp = torch.where(dist > 0, (c * vp + (1.0 - c) * vr).clamp(max=ph["cap"]), vp)
    if case.get("fs"):
        vp[:top] = 0.0
    return ((vp * ph["dt"] / ph["h"]) ** 2).float()


class _Wave:
    """A pair of levels of one wavefield in 64 bits, zero beyond the grid."""

    def __init__(self, a):
        self.a, nd = a, a.dim()
        pad = [m + 8 for m in a.shape]
        self.cur, self.old = (torch.zeros(pad, dtype=torch.float64, device=a.device) for _ in range(2))
        self.acc, self.tmp = torch.empty_like(a), torch.empty_like(a)
        self.mid = tuple(slice(4, -4) for _ in range(nd))

    def at(self, p, ax, k):
        n = p.shape[ax] - 8
        return p[tuple(slice(4 + k, 4 + k + n) if d == ax else slice(4, -4) for d in range(p.dim()))]

    def lap(self, p):
        nd = p.dim()
        torch.mul(p[self.mid], nd * C0, out=self.acc)
        for k in range(1, 5):
            torch.add(self.at(p, 0, k), self.at(p, 0, -k), out=self.tmp)
            for ax in range(1, nd):
                self.tmp.add_(self.at(p, ax, k)).add_(self.at(p, ax, -k))
            self.acc.add_(self.tmp, alpha=C[k - 1])
        return self.acc

    def step(self):
        """old <- 2 cur - old + a lap cur, then the two levels change places."""
        self.lap(self.cur).mul_(self.a)
        o = self.old[self.mid]
        o.neg_().add_(self.cur[self.mid], alpha=2.0).add_(self.acc)
        self.cur, self.old = self.old, self.cur

    @property
    def p(self):
        return self.cur[self.mid]


def _at(nodes, nd):
    n = torch.as_tensor(np.asarray(nodes, np.int64).reshape(-1, 3), device=_device())
    return (n[:, 2], n[:, 0]) if nd == 2 else (n[:, 2], n[:, 1], n[:, 0])


def _inject(wave, idx, val):
    wave.p.index_put_(idx, val, accumulate=True)


def _model64(a, wav, src, rec, nt, scale, keep=None):
    w, s, r = _Wave(a), _at(src, a.dim()), _at(rec, a.dim())
    f = -(a[s] * scale)[None] * wav.double()[:, None]
    out = torch.empty((nt + 1, len(rec)), dtype=torch.float64, device=a.device)
    for n in range(nt + 1):
        out[n] = w.p[r]
        if keep is not None:
            keep(n, w)
        if n < nt:
            w.step()
            _inject(w, s, f[n])
    return out.t().contiguous()


def _rtm64(a, wav, src, rec, seis, nt, scale, box, k=0):
    """num, den (and, for k > 0, the levels kept every k steps) of one shot."""
    store = []

    def keep(n, w):
        if k and n % k == 0:
            store.append(w.p[box].clone())

    w, s, r = _Wave(a), _at(src, a.dim()), _at(rec, a.dim())
    f = -(a[s] * scale)[None] * wav.double()[:, None]
    for n in range(nt):
        keep(n, w)
        w.step()
        _inject(w, s, f[n])
    keep(nt, w)
    b, d = _Wave(a), seis.double().t().contiguous() * (a[r] * scale)[None]
    num = torch.zeros_like(w.p[box])
    den = torch.zeros_like(num)
    if not k:
        w.cur, w.old = w.old, w.cur        # level nt - 1 is at hand: the first step back needs no update
    for n in range(nt, -1, -1):
        if k:
            if n % k == 0:
                num.addcmul_(store[n // k], b.p[box])
                den.addcmul_(store[n // k], store[n // k])
        else:
            p = w.old[w.mid][box] if n == nt else w.p[box]
            num.addcmul_(p, b.p[box])
            den.addcmul_(p, p)
            if 0 < n < nt:
                w.step()
                _inject(w, s, f[n])
        if n > 0:
            b.step()
            _inject(b, r, d[n])
    return num, den, store


def _fwi64(a, v_box, wav, src, rec, dobs, nt, box):
    """Misfit and its gradient with respect to the interior velocity, by the discrete adjoint."""
    levels = torch.empty((nt + 1,) + a.shape, dtype=torch.float64, device=a.device)

    def keep(n, w):
        levels[n] = w.p

    res = _model64(a, wav, src, rec, nt, 1.0, keep) - dobs.double()
    s, r = _at(src, 2), _at(rec, 2)
    lam, aux = _Wave(a), _Wave(a)          # lam.cur = lambda^{n+1}, lam.old = lambda^{n+2}
    grad = torch.zeros_like(a)
    for n in range(nt, -1, -1):
        if n < nt:                         # d p^{n+1} / d a = lap p^n - f[n] delta_s
            aux.p.copy_(levels[n])
            g = aux.lap(aux.cur)
            g[s] -= wav[n].double()
            grad.addcmul_(lam.p, g)
        aux.p.copy_(lam.p).mul_(a)         # lambda^n = 2 lambda^{n+1} - lambda^{n+2} + lap(a lambda^{n+1}) + residual
        g = aux.lap(aux.cur)
        o = lam.old[lam.mid]
        o.neg_().add_(lam.p, alpha=2.0).add_(g)
        lam.cur, lam.old = lam.old, lam.cur
        _inject(lam, r, res[:, n])
    return 0.5 * res.pow(2).sum(), grad[box] * 2.0 * a[box] / v_box


def _net64(p, x):
    """The network on (n, H, W) images; parameters as the library stores them."""
    h, o = x[:, None], 0
    for l, (ci, co) in enumerate([(1, 32), (32, 32), (32, 32), (32, 32), (32, 1)]):
        w = p[o:o + 9 * ci * co].reshape(3, 3, co, ci).permute(2, 3, 0, 1)
        b = p[o + 9 * ci * co:o + 9 * ci * co + co]
        o += 9 * ci * co + co
        h = torch.nn.functional.conv2d(h, w.contiguous(), b, padding=1)
        if l < 4:
            h = torch.relu(h)
    return x + h[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("denoise", "volume"):
        p = _params(seed).double()
        with torch.no_grad():
            if kind == "volume":
                x = _images((case["nz"], case["ny"], case["nx"]), seed)
                return torch.stack([_net64(p, x[:, k:k + 1].permute(1, 0, 2).double())[0] for k in range(case["ny"])], 1)
            x = _images((case["n"], case["H"], case["W"]), seed)
            return torch.cat([_net64(p, x[k:k + 1].double()) for k in range(case["n"])])
    if kind == "train":
        n, H, W = case["n"], case["H"], case["W"]
        x = _images((n, H, W), seed)
        t = x + 0.3 * _images((n, H, W), seed + 1)
        p = _params(seed).double().requires_grad_(True)
        ys, loss = [], 0.0
        for k in range(n):
            y = _net64(p, x[k:k + 1].double())
            part = (y - t[k:k + 1].double()).pow(2).sum() / (n * H * W)
            part.backward()
            ys.append(y.detach())
            loss = loss + part.detach()
        return dict(y=torch.cat(ys), loss=loss.reshape(1), grad=p.grad)
    ph, nt, nb = PHYS[case["phys"]], case["nt"], case["nb"]
    if kind == "batch":
        nxs, shots = _batch_shots(case, seed)
        v, wav = _velocity(ph, (case["nz"], nxs), seed, smooth=True), _ricker(ph, nt)
        image = torch.zeros((case["nz"], nxs), dtype=torch.float64, device=v.device)
        for s, (width, off, src, rec) in enumerate(shots):
            a = _coef(case, v[:, off:off + width].contiguous(), seed + s).double()
            box = (slice(nb, nb + case["nz"]), slice(nb, nb + width))
            num, den, _ = _rtm64(a, wav, src, rec, _record(ph, src, rec, nt, seed + s), nt, 1.0, box)
            image[:, off:off + width] += num / (den + EPS_REL * den.max())
        return image
    if kind == "fwi":
        v0, srcs, rec, wav, dobs = _fwi_inputs(case, seed)
        a = _coef(case, v0, seed).double()
        box = (slice(nb, nb + case["nz"]), slice(nb, nb + case["nx"]))
        J, grad = 0.0, 0.0
        for s, d in zip(srcs, dobs):
            j, g = _fwi64(a, v0.double(), wav, s, rec, d, nt, box)
            J, grad = J + j, grad + g
        return dict(misfit=J, grad=grad)
    src, rec = _geometry(case)
    a = _coef(case, _velocity(ph, _interior(case), seed, smooth=kind != "model"), seed).double()
    wav = _ricker(ph, nt)
    scale = 1.0 / ph["h"] if "ny" in case else 1.0
    if kind == "model":
        return _model64(a, wav, src, rec, nt, scale)
    top = 4 if case.get("fs") else nb
    box = (slice(top, top + case["nz"]),) + tuple(slice(nb, nb + m) for m in _interior(case)[1:])
    k = R.rbc_nyquist_stride(ph["dt"], 2.5 * ph["f"]) if kind == "storage" else 0
    num, den, store = _rtm64(a, wav, src, rec, _record(ph, src, rec, nt, seed), nt, scale, box, k)
    out = dict(num=num, den=den, image=num / (den + EPS_REL * den.max()))
    if kind == "storage":
        out["store"] = torch.stack(store).reshape(-1)
    return out
