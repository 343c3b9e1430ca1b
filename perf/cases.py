"""The work a user of this library has it do, as measurable cases: imaging (2D
and 3D), the autofocus step, the linear adjoint, range compression and
conditioning, micronavigation and the interpolator's training step.

listed() gives named cases, draw() more of the same ranges, prepare() what a
program has in hand before the call, run() one pass through the public entry
points, work() what a pass cannot do without and exact() the same outputs by
plain FP64 torch.  Sizes come from the synthetic workloads (small_2d,
stripmap_2d, volume_3d, learned_2d, autofocus_2d), the tests and the benchmark.
"""
import math

import numpy as np
import torch

import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import autofocus

FC, FS, C_SOUND, BANDWIDTH, PULSE_T = 100e3, 40e3, 1500.0, 20e3, 5e-3
NU = BANDWIDTH / (2.0 * FS)     # band edge of the echoes [cycles/sample]
SPACING, SPEED = 0.1, 1.95      # along-track ping spacing [m], platform speed [m/s]
EXACT_UPDATES = 8e10            # imaging sums beyond this take FP64 torch too long
STORE = {"c64": sas.SAS_ECHO_C64, "f16": sas.SAS_ECHO_C32_F16, "bf16": sas.SAS_ECHO_C32_BF16}
DEV = "cuda"


def listed():
    return [
        # a quick look at the newest block of pings: the small_2d workload, one upload and one small image
        dict(name="image_small", kind="image", P=128, C=4, Ns=2048, nx=256, ny=256, px=0.02, t0=0.025, y0=20.0,
             store="c64", table=False, beam=0.0, motion=False, upload=True),
        # the survey image: a quarter of the stripmap workload's pings onto its full grid
        dict(name="image_strip", kind="image", P=512, C=32, Ns=16384, nx=4096, ny=4096, px=0.015, t0=0.05, y0=40.0,
             store="c64", table=False, beam=0.0, motion=False, upload=False),
        # the learned interpolator with BF16 storage on a ragged patch; fresh echoes are stored on every pass
        dict(name="image_learned", kind="image", P=250, C=24, Ns=8192, nx=1500, ny=1101, px=0.015, t0=0.04, y0=30.0,
             store="bf16", table=True, beam=0.0, motion=False, upload=True),
        # a strip with the beam's field of view (ray culling) and the receivers moving during reception
        dict(name="image_beam", kind="image", P=768, C=16, Ns=8192, nx=1600, ny=1400, px=0.015, t0=0.05, y0=40.0,
             store="c64", table=False, beam=30.0, motion=True, upload=False),
        # a near-field sub-bottom volume from a planar array with FP16 storage
        dict(name="volume", kind="volume", P=196, C=64, Ns=8192, nx=256, ny=224, nz=56, px=0.02, store="f16",
             c_sed=0.0, upload=True),
        # one gradient step of the sharpness autofocus
        dict(name="autofocus_step", kind="autofocus", P=256, C=16, Ns=8192, nx=1024, ny=1000, px=0.015, t0=0.04,
             y0=30.0),
        # image to echo: the transpose, for iterative reconstruction
        dict(name="adjoint", kind="adjoint", P=128, C=8, Ns=4096, nx=512, ny=480, px=0.015, t0=0.025, y0=20.0),
        # range compression of raw rows with the 5 ms chirp
        dict(name="matched_filter", kind="matched_filter", rows=8192, n=16384, L=200),
        # conditioning of compressed rows in place: whitening, then time-varying gain
        dict(name="condition", kind="condition", rows=16384, n=8192, gamma=0.1, alpha=0.5),
        # micronavigation: the delays between displaced phase centres of a survey leg
        dict(name="dpc_delays", kind="delays", P=256, C=32, Ns=16384, shift=8, K=120, W=128, L=8, store="c64"),
        # and the motion solution from them
        dict(name="dpc_solve", kind="solve", P=1024, C=32, shift=8, K=24, huber=0.0),
        # one optimiser step of the learned interpolator
        dict(name="train_step", kind="train", B=8192),
    ]


def draw(rng):
    def lg(lo, hi, m=1):
        return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / m)) * m)

    while True:
        kind = rng.choice(["image", "image", "image", "volume", "autofocus", "adjoint", "matched_filter", "condition",
                           "delays", "solve", "train"])
        if kind == "image":
            store = rng.choice(["c64", "c64", "f16", "bf16"])
            c = dict(P=lg(64, 1024), C=rng.choice([1, 4, 6, 8, 16, 24, 32]), Ns=lg(2048, 16384, 4), nx=lg(200, 4096),
                     ny=lg(200, 4096), px=rng.choice([0.01, 0.015, 0.02]), t0=0.05, y0=40.0, store=store,
                     table=rng.random() < 0.3, beam=rng.choice([0.0, 0.0, 0.0, 20.0, 30.0]),
                     motion=rng.random() < 0.2, upload=rng.random() < 0.5)
            ok = c["P"] * c["C"] * c["nx"] * c["ny"] <= 1.2e11
        elif kind == "volume":
            c = dict(P=lg(16, 256), C=rng.choice([16, 64]), Ns=lg(2048, 8192, 4), nx=lg(40, 400), ny=lg(40, 400),
                     nz=lg(8, 128), px=0.02, store=rng.choice(["c64", "f16", "bf16"]),
                     c_sed=rng.choice([0.0, 0.0, 0.0, 1700.0]), upload=rng.random() < 0.5)
            ok = c["P"] * c["C"] * c["nx"] * c["ny"] * c["nz"] <= 5e10
        elif kind == "autofocus":
            c = dict(P=lg(64, 512), C=rng.choice([4, 8, 16]), Ns=lg(4096, 8192, 4), nx=lg(200, 2048),
                     ny=lg(200, 2048), px=0.015, t0=0.04, y0=30.0)
            ok = c["P"] * c["C"] * c["nx"] * c["ny"] <= 1e10
        elif kind == "adjoint":
            c = dict(P=lg(32, 256), C=rng.choice([1, 4, 8, 16]), Ns=lg(2048, 8192, 4), nx=lg(100, 1024),
                     ny=lg(100, 1024), px=rng.choice([0.015, 0.02]), t0=0.025, y0=20.0)
            ok = c["P"] * c["C"] * c["nx"] * c["ny"] <= 1e9
        elif kind == "matched_filter":
            c = dict(rows=lg(64, 16384), n=lg(1000, 16384), L=lg(50, 1000))
            ok = c["rows"] * c["n"] <= 1.5e8
        elif kind == "condition":
            c = dict(rows=lg(256, 65536), n=rng.choice([1024, 2048, 4096, 8192, 16384]), gamma=0.1, alpha=0.5)
            ok = c["rows"] * c["n"] <= 1.5e8
        elif kind == "delays":
            W, L = rng.choice([64, 100, 128, 160]), rng.choice([4, 8, 12])
            c = dict(P=lg(16, 512), C=rng.choice([8, 16, 32]), Ns=lg(4096, 16384, 4), shift=rng.choice([2, 4]),
                     K=lg(8, 120), W=W, L=L, store=rng.choice(["c64", "c64", "f16"]))
            ok = c["P"] * c["C"] * c["Ns"] <= 1.4e8
        elif kind == "solve":
            c = dict(P=lg(64, 2048), C=rng.choice([8, 16, 32]), shift=rng.choice([2, 4]), K=lg(6, 32),
                     huber=0.0)
            ok = True
        else:
            c = dict(B=lg(256, 32768))
            ok = True
        if ok:
            return dict(kind=kind, **c)


# ---------------------------------------------------------------------------
# inputs, from the seed alone

def gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 1)
    return g


def randc(shape, g):
    """complex64 Gaussian, unit power"""
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), device=DEV, generator=g) * math.sqrt(0.5))


def band_rows(rows, n, g):
    """Rows of band-limited complex Gaussian samples with unit mean power: the statistics of range-compressed
    speckle echoes.  complex64 [rows, n]."""
    out = torch.empty((rows, n), dtype=torch.complex64, device=DEV)
    keep = (torch.fft.fftfreq(n, device=DEV).abs() <= NU).to(torch.float32)
    step = max(1, (1 << 26) // n)
    for r in range(0, rows, step):
        z = torch.fft.fft(randc((min(step, rows - r), n), g)) * keep
        out[r:r + step] = torch.fft.ifft(z) * math.sqrt(n / float(keep.sum()))
    return out


def strip_nav(c, seed, error=0.0):
    """A straight track with sway, heave and a yaw random walk; receivers along the hull (FP64, host)."""
    rng = np.random.default_rng(seed + 11)
    P, C = c["P"], c["C"]
    i = np.arange(P)
    pos = np.stack([i * SPACING, np.zeros(P), np.full(P, -10.0)], 1)
    t, ph = rng.uniform(20.0, 60.0, 2), rng.uniform(0.0, 2 * np.pi, 2)
    pos[:, 1] += 0.05 * np.sin(2 * np.pi * i / t[0] + ph[0])
    pos[:, 2] += 0.05 * np.sin(2 * np.pi * i / t[1] + ph[1])
    rate = 0.05 * 2 * np.pi / t * (SPEED / SPACING)
    vel = np.stack([np.full(P, SPEED), rate[0] * np.cos(2 * np.pi * i / t[0] + ph[0]),
                    rate[1] * np.cos(2 * np.pi * i / t[1] + ph[1])], 1)
    att = np.zeros((P, 3))
    att[:, 2] = np.cumsum(rng.normal(0.0, np.deg2rad(0.01), P))
    if error:
        pos += rng.normal(0.0, error, pos.shape)
    rx = np.stack([(np.arange(C) - 0.5 * (C - 1)) * 0.025, np.zeros(C), np.zeros(C)], 1)
    return dict(pos=pos, att=att, vel=vel, tx=np.zeros(3), rx=rx)


def volume_nav(c, seed):
    """Pings on a square lattice two metres above the seafloor, a planar receive array (FP64, host)."""
    P, n = c["P"], int(math.isqrt(c["C"]))
    side, i = int(math.ceil(math.sqrt(P))), np.arange(P)
    rng = np.random.default_rng(seed + 12)
    pos = np.stack([(i % side) * 0.64, (i // side) * 0.64, np.full(P, -2.0)], 1) + rng.normal(0.0, 0.02, (P, 3))
    att = np.zeros((P, 3))
    att[:, 2] = np.cumsum(rng.normal(0.0, np.deg2rad(0.01), P))
    a = (np.arange(n) - 0.5 * (n - 1)) * 0.02
    gx, gy = np.meshgrid(a, a)
    rx = np.stack([gx.ravel(), gy.ravel(), np.zeros(n * n)], 1)
    return dict(pos=pos, att=att, vel=None, tx=np.zeros(3), rx=rx)


def grid_of(c):
    """(x0, y0, z0, dx, dy, dz, nx, ny, nz): the patch abeam of the middle of the track, or under the lattice."""
    p = c["px"]
    if c["kind"] == "volume":
        mid = 0.5 * 0.64 * (math.ceil(math.sqrt(c["P"])) - 1)
        return (mid - 0.5 * c["nx"] * p, mid - 0.5 * c["ny"] * p, 0.0, p, p, p, c["nx"], c["ny"], c["nz"])
    return (0.5 * (c["P"] * SPACING - c["nx"] * p), c["y0"], 0.0, p, p, 0.0, c["nx"], c["ny"], 1)


def scene(c, seed):
    """Navigation, echo [P, C, Ns] and (with table) the tabulated interpolator of an imaging case."""
    if c["kind"] == "volume":
        nav = volume_nav(c, seed)
    else:
        nav = strip_nav(c, seed, 0.02 if c["kind"] == "autofocus" else 0.0)
    echo = None
    if c["kind"] != "adjoint":
        echo = band_rows(c["P"] * c["C"], c["Ns"], gen(seed)).reshape(c["P"], c["C"], c["Ns"])
    table = None
    if c.get("table"):
        f = torch.arange(4097, dtype=torch.float64, device=DEV) / 4096
        table = kaiser_weights(f, 8, 5.5).to(torch.float32).contiguous()
    return nav, echo, table


def sonar(c, nav):
    g = sas.Geometry(nav["pos"], nav["att"], nav["tx"], nav["rx"],
                     sas.make_signal(FC, FS, C_SOUND, c.get("t0", 0.0), c["Ns"]))
    if c.get("beam"):
        g.set_beam(math.radians(c["beam"]), 1)
    if c.get("motion"):
        g.set_velocity(nav["vel"])
    if c.get("c_sed"):
        g.set_refraction(0.3, c["c_sed"])
    return g


# ---------------------------------------------------------------------------
# micronavigation inputs

def dpc_echo(c, seed):
    """Echoes whose receiver c of ping i + 1 sees what receiver c + shift of ping i saw, delayed by the sway of
    that ping, plus noise (correlation about 0.9).  complex64 [P, C, Ns]."""
    P, C, Ns, s = c["P"], c["C"], c["Ns"], c["shift"]
    g = gen(seed)
    base = band_rows((P - 1) * s + C, Ns, g)
    rng = np.random.default_rng(seed + 13)
    step = 0.4 * rng.integers(-3, 4, P) + rng.uniform(-0.1, 0.1, P)     # delay from ping to ping [samples]
    d = torch.from_numpy(np.cumsum(step) - np.cumsum(step).mean())
    nu = torch.fft.fftfreq(Ns, dtype=torch.float64)
    out = torch.empty((P, C, Ns), dtype=torch.complex64, device=DEV)
    for i in range(P):
        ramp = torch.exp(-2j * math.pi * (nu + FC / FS) * d[i]).to(torch.complex64).to(DEV)
        z = torch.fft.ifft(torch.fft.fft(base[i * s:i * s + C]) * ramp)
        out[i] = z + 0.3 * band_rows(C, Ns, g)
    return out


def dpc_centres(c):
    lo, hi = 2 * c["W"], c["Ns"] - 2 * c["W"]
    return torch.from_numpy(np.round(np.linspace(lo, hi, c["K"])).astype(np.int32)).to(DEV)


def dpc_motion(c, seed):
    """The arrays of a motion problem: a track with sway and heave, and delays with 50 ns of noise."""
    rng = np.random.default_rng(seed + 14)
    P, C, s, K = c["P"], c["C"], c["shift"], c["K"]
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(DEV)  # noqa: E731
    i = np.arange(P)
    a = rng.uniform(0.0, 2 * np.pi, 2)
    vy, vz = 0.03 * np.sin(2 * np.pi * i / 40.0 + a[0]), 0.02 * np.sin(2 * np.pi * i / 55.0 + a[1])
    dt = np.full(P - 1, SPACING / SPEED)
    att = np.stack([rng.normal(0, 0.002, P), rng.normal(0, 0.002, P), np.cumsum(rng.normal(0, 1e-4, P))], 1)
    rx = np.stack([(np.arange(C) - 0.5 * (C - 1)) * 2 * SPACING / s, np.zeros(C), np.zeros(C)], 1)
    M = (P - 1) * (C - s) * K
    m = dict(p0=t([0.0, 0.0, -10.0]), vx=t(np.full(P, SPEED)), att=t(att), dt=t(dt), tx=t(np.zeros(3)), rx=t(rx),
             t=t(np.linspace(0.05, 0.3, K)), weight=t(rng.uniform(0.5, 1.0, M)),
             z=t(-10.0 + np.concatenate([[0.0], np.cumsum(vz[:-1] * dt)]) + rng.normal(0, 0.002, P)))
    zero = torch.zeros(P, dtype=torch.float64, device=DEV)
    m["ps"] = dpc_footprints(c, m, zero, zero)
    m["delay"] = -dpc_residual(c, m, dpc_nodes(m, t(vy), t(vz)))[0].reshape(-1) / C_SOUND + t(rng.normal(0, 5e-8, M))
    return m


# ---------------------------------------------------------------------------
# training inputs

def mlp_inputs(c, seed):
    """Mid-training parameters and moments, and a batch of (fraction, window, residual target) draws."""
    g, B = gen(seed), c["B"]
    n = lambda *s: torch.randn(s, device=DEV, generator=g)  # noqa: E731
    theta = torch.cat([3.0 * n(64), 3.0 * (2 * torch.rand(64, device=DEV, generator=g) - 1), n(4096) / 8, 0.1 * n(64),
                       0.001 / 8 * n(512), torch.zeros(8, device=DEV)])
    m, v = 1e-4 * n(4808), 1e-8 * (0.5 + torch.rand(4808, device=DEV, generator=g))
    rows = band_rows(512, 2048, g).reshape(-1)
    at = torch.randint(0, 512, (B,), device=DEV, generator=g) * 2048 + torch.randint(24, 2024, (B,), device=DEV, generator=g)
    f = torch.rand(B, device=DEV, generator=g)
    win = rows[at[:, None] + torch.arange(-3, 5, device=DEV)].contiguous()
    far = rows[at[:, None] + torch.arange(-15, 17, device=DEV)].to(torch.complex128)
    y = (kaiser_weights(f.double(), 32, 10.0) * far).sum(1) - (kaiser_weights(f.double(), 8, 4.0) * win).sum(1)
    return dict(theta=theta, m=m, v=v, f=f, win=win, y=y.to(torch.complex64), step=1000, lr=2e-3)


# ---------------------------------------------------------------------------

def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("image", "volume", "autofocus", "adjoint"):
        nav, echo, table = scene(c, seed)
        geom = sonar(c, nav)
        grid = sas.make_grid(*grid_of(c))
        s = dict(kind=kind, geom=geom, grid=grid, interp=sas.table_interp(table, 4096) if table is not None else sas.kaiser(4.0))
        if kind in ("image", "volume"):
            s["store"] = STORE[c["store"]]
            if c["upload"]:
                s["echo"] = echo
            else:
                geom.upload_echo(echo, s["store"])
        elif kind == "autofocus":
            geom.upload_echo(echo)
            s["dp"] = 1e-3 * torch.randn((c["P"], 3), device=DEV, generator=gen(seed + 5))
        else:
            s["img"] = randc((c["ny"], c["nx"]), gen(seed))
            s["shape"] = (c["P"], c["C"], c["Ns"])
        return s
    if kind == "matched_filter":
        t = torch.arange(c["L"], dtype=torch.float64, device=DEV) / FS
        T = c["L"] / FS
        rep = torch.exp(1j * math.pi * (BANDWIDTH / T) * (t - 0.5 * T) ** 2).to(torch.complex64)
        return dict(kind=kind, raw=randc((c["rows"], c["n"]), gen(seed)), rep=rep)
    if kind == "condition":
        return dict(kind=kind, c=c, rows=condition_rows(c, seed))
    if kind == "delays":
        nav = strip_nav(c, seed)
        geom = sas.Geometry(nav["pos"], nav["att"], nav["tx"], nav["rx"],
                            sas.make_signal(FC, FS, C_SOUND, 0.0, c["Ns"]))
        geom.upload_echo(dpc_echo(c, seed), STORE[c["store"]])
        return dict(kind=kind, c=c, geom=geom, centres=dpc_centres(c), M=(c["P"] - 1) * (c["C"] - c["shift"]) * c["K"])
    if kind == "solve":
        m = dpc_motion(c, seed)
        pr = sas.sas_dpc_problem(P=c["P"], C=c["C"], shift=c["shift"], K=c["K"], side=1, c=C_SOUND, lambda1=1e-4,
                                 lambda2=1e-3, huber=c["huber"], **{"d_" + k: m[v].data_ptr() for k, v in (
                                     ("p0", "p0"), ("vx", "vx"), ("att", "att"), ("dt", "dt"), ("tx_lever", "tx"),
                                     ("rx_lever", "rx"), ("t", "t"), ("delay", "delay"), ("weight", "weight"),
                                     ("z_dvl", "z"), ("ps", "ps"))})
        return dict(kind=kind, P=c["P"], arrays=m, pr=pr)
    s = mlp_inputs(c, seed)
    s.update(kind=kind, B=c["B"], loss=torch.empty(1, device=DEV), grad=torch.empty(4808, device=DEV),
             work=torch.empty(sas.sas_mlp_workspace_bytes(c["B"]), dtype=torch.uint8, device=DEV))
    return s


def run(s):
    kind = s["kind"]
    if kind in ("image", "volume"):
        if "echo" in s:
            s["geom"].upload_echo(s["echo"], s["store"])
        return s["geom"].backproject(s["grid"], s["interp"])
    if kind == "autofocus":
        # FP32 offsets as an optimiser's parameters: their gradient comes back in their type
        dp = s["dp"].detach().requires_grad_()
        img = autofocus.backproject_offsets(dp.double(), s["geom"], s["grid"], s["interp"])
        _, g = autofocus.sharpness_and_grad(img.detach())
        img.backward(gradient=2.0 * g)      # dL/dRe + i dL/dIm = 2 dL/dI*
        return [img.detach(), g, dp.grad]
    if kind == "adjoint":
        out = torch.empty(s["shape"], dtype=torch.complex64, device=DEV)
        sas.sas_backproject_adjoint(s["geom"].h, s["grid"], s["interp"], s["img"], out)
        return out
    if kind == "matched_filter":
        out = torch.empty_like(s["raw"])
        sas.sas_matched_filter(s["raw"], out.shape[0], out.shape[1], s["rep"], s["rep"].numel(), out)
        return out
    if kind == "condition":
        c, out = s["c"], torch.empty_like(s["rows"])
        wg, tg = torch.empty(c["n"], device=DEV), torch.empty(c["n"], device=DEV)
        sas.sas_whiten(s["rows"], out, c["rows"], c["n"], c["gamma"], wg)
        sas.sas_tvg(out, out, c["rows"], c["n"], c["alpha"], tg)
        return [out, wg, tg]
    if kind == "delays":
        c = s["c"]
        o = [torch.empty(s["M"], dtype=torch.float64, device=DEV) for _ in range(3)]
        sas.sas_dpc_delays(s["geom"].h, c["shift"], s["centres"], c["K"], c["W"], c["L"], *o)
        return o
    if kind == "solve":
        vy, vz = (torch.zeros(s["P"], dtype=torch.float64, device=DEV) for _ in range(2))
        loss, _ = sas.sas_dpc_solve(s["pr"], vy, vz, 50)
        return [vy, vz, loss]
    sas.sas_mlp_loss_grad(s["theta"], s["f"], s["win"], s["y"], s["B"], s["loss"], s["grad"], s["work"])
    sas.sas_mlp_adam(s["theta"], s["grad"], s["m"], s["v"], s["step"], s["lr"])
    return [s["loss"], s["grad"], s["theta"], s["m"], s["v"]]


def work(case):
    c, kind = case, case["kind"]
    if kind in ("image", "volume", "autofocus", "adjoint"):
        npx = c["nx"] * c["ny"] * c.get("nz", 1)
        upd = float(c["P"]) * c["C"] * npx
        if c.get("beam"):   # the part of the track whose beams see a pixel
            w = 2 * math.tan(math.radians(c["beam"]) / 2) * (c["y0"] + 0.5 * c["ny"] * c["px"])
            upd *= min(1.0, w / (c["P"] * SPACING))
        elem = 8 if c.get("store", "c64") == "c64" else 4
        # samples a row can give to this grid: its delay span
        span = 2 * FS / C_SOUND * math.hypot(c["nx"] * c["px"], c["ny"] * c["px"])
        echo = c["P"] * c["C"] * min(c["Ns"], span) * elem
        # FP32 operations of an update: a fused multiply-add counts two; 14 of them for the taps' polynomial,
        # 4 to rotate and add, 14 for range, delay and phase
        f = 64.0 * upd
        if kind == "autofocus":
            return dict(bytes=2 * echo + 4 * 8 * npx, flops=f + 1.6 * f)
        if kind == "adjoint":
            return dict(bytes=8 * npx + c["P"] * c["C"] * c["Ns"] * 8, flops=f)
        up = c["P"] * c["C"] * c["Ns"] * (8 + elem) if c["upload"] else 0
        return dict(bytes=echo + up + 8 * npx, flops=f)
    if kind == "matched_filter":
        return dict(bytes=16.0 * c["rows"] * c["n"], flops=10.0 * math.log2(max(2, 4 * c["L"])) * c["rows"] * c["n"])
    if kind == "condition":
        return dict(bytes=32.0 * c["rows"] * c["n"], flops=10.0 * math.log2(c["n"]) * c["rows"] * c["n"])
    if kind == "delays":
        M = (c["P"] - 1) * (c["C"] - c["shift"]) * c["K"]
        elem = 8 if c["store"] == "c64" else 4
        return dict(bytes=float(min(M * 2 * c["W"], 2 * c["P"] * c["C"] * c["Ns"])) * elem + 24.0 * M,
                    flops=8.0 * M * c["W"] * (2 * c["L"] + 1))
    if kind == "solve":
        M = (c["P"] - 1) * (c["C"] - c["shift"]) * c["K"]
        return dict(bytes=10 * 40.0 * M, flops=10 * 2 * 150.0 * M)   # about ten linearisations and losses
    return dict(bytes=c["B"] * 76.0 + 4808 * 4 * 8, flops=6.0 * 4672 * c["B"])


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, by plain torch

def kaiser_weights(f, taps, beta):
    """Normalised Kaiser-windowed sinc taps at fractions f [n] (FP64): [n, taps]."""
    k = torch.arange(1 - taps // 2, taps // 2 + 1, device=f.device, dtype=torch.float64)
    d = f[:, None] - k
    s = (1.0 - (2.0 * d / taps) ** 2).clamp_min(0.0)
    w = torch.sinc(d) * torch.special.i0(beta * torch.sqrt(s)) * (d.abs() < taps / 2)
    return w / w.sum(1, keepdim=True)


def rotation(att):
    """R of roll, pitch, yaw [P, 3] (yaw about z after pitch about y after roll about x): [P, 3, 3]."""
    (sr, sp, sy), (cr, cp, cy) = torch.sin(att).T, torch.cos(att).T
    return torch.stack([cp * cy, cy * sp * sr - cr * sy, cr * cy * sp + sr * sy,
                        cp * sy, cr * cy + sp * sr * sy, cr * sp * sy - cy * sr,
                        -sp, cp * sr, cp * cr], 1).reshape(-1, 3, 3)


def sums(c, nav, echo, weights, image=None, g=None, dp=None):
    """The imaging sums over all pings and channels: returns the image (image, g None), the adjoint's echo (image
    given) or the gradient with respect to the per-ping offsets (g given)."""
    t = lambda a: torch.from_numpy(np.asarray(a)).to(DEV)  # noqa: E731
    R, pos = rotation(t(nav["att"])), t(nav["pos"])
    if dp is not None:
        pos = pos + dp
    tx = pos + R @ t(nav["tx"])
    rx = pos[:, None] + torch.einsum("pij,cj->pci", R, t(nav["rx"]))
    x0, y0, z0, dx, dy, dz, nx, ny, nz = grid_of(c)
    ar = lambda n: torch.arange(n, dtype=torch.float64, device=DEV)  # noqa: E731
    Z, Y, X = torch.meshgrid(z0 + dz * ar(nz), y0 + dy * ar(ny), x0 + dx * ar(nx), indexing="ij")
    pts = torch.stack([X.reshape(-1), Y.reshape(-1), Z.reshape(-1)])           # [3, n]
    n, Ns, pad = pts.shape[1], c["Ns"], 8
    tab = weights                                                               # [N + 1, 8]
    dtab = (tab[1:] - tab[:-1]) * (tab.shape[0] - 1)
    N = tab.shape[0] - 1
    vel = t(nav["vel"]) if c.get("motion") else None
    tan = math.tan(math.radians(c["beam"]) / 2) if c.get("beam") else 0.0
    acc = torch.zeros(n, dtype=torch.complex128, device=DEV) if image is None and g is None else None
    grad = torch.zeros((c["P"], 3), dtype=torch.float64, device=DEV)
    out = torch.zeros((c["P"], c["C"], Ns), dtype=torch.complex128, device=DEV) if image is not None else None
    for i in range(c["P"]):
        wt = pts - tx[i][:, None]
        rt = torch.sqrt((wt * wt).sum(0))
        def sees(w):
            b = R[i].T @ w
            return (b[1] > 0) & (b[0].abs() <= tan * b[1])
        st = sees(wt) if tan else None
        if tan and not bool(st.any()):
            continue
        for ch in range(c["C"]):
            wr = pts - rx[i, ch][:, None]
            ok = st & sees(wr) if tan else None
            rr = torch.sqrt((wr * wr).sum(0))
            tau = (rt + rr) / C_SOUND
            if vel is not None:
                for _ in range(4):
                    q = wr - vel[i][:, None] * tau
                    tau = (rt + torch.sqrt((q * q).sum(0))) / C_SOUND
            u = (tau - c.get("t0", 0.0)) * FS
            j = torch.floor(u)
            f = u - j
            j = j.to(torch.int64).clamp(-pad, Ns + pad - 1)
            y = f * N
            m = y.to(torch.int64).clamp_max(N - 1)
            w = torch.lerp(tab[m], tab[m + 1], (y - m)[:, None])                # [n, 8]
            ph = torch.polar(torch.ones_like(tau), 2 * math.pi * torch.remainder(FC * tau, 1.0))
            if image is not None:
                v = (image * ph.conj())[:, None] * w
                row = torch.zeros(Ns + 4 * pad, dtype=torch.complex128, device=DEV)
                at = (j[:, None] + torch.arange(-3, 5, device=DEV) + 2 * pad).reshape(-1)
                torch.view_as_real(row).index_add_(0, at, torch.view_as_real(v.reshape(-1)))
                out[i, ch] = row[2 * pad:2 * pad + Ns]
                continue
            row = torch.nn.functional.pad(torch.view_as_real(echo[i, ch].to(torch.complex128)).T, (2 * pad, 2 * pad))
            win = torch.view_as_complex(row.T.contiguous()).unfold(0, 8, 1)[j + 2 * pad - 3]     # [n, 8]
            s = (win * w).sum(1)
            if g is None:
                acc += torch.where(ok, s * ph, 0) if tan else s * ph
                continue
            ds = (win * dtab[m]).sum(1)
            r = (g.conj() * (FS * ds + 2j * math.pi * FC * s) * ph).real
            grad[i] += -2.0 / C_SOUND * ((wt / rt + wr / rr) @ r)
    return out if image is not None else (grad if g is not None else acc.reshape(nz, ny, nx))


def fine_table(beta):
    """Kaiser taps on 2^16 fractions: linear interpolation of it is within 1e-9 of the definition."""
    return kaiser_weights(torch.arange(65537, dtype=torch.float64, device=DEV) / 65536, 8, beta)


def condition_rows(c, seed):
    """Compressed rows: band-limited speckle with white noise, fading along the row."""
    g = gen(seed)
    x = band_rows(c["rows"], c["n"], g)
    fade = torch.linspace(1.0, 0.2, c["n"], device=DEV)
    for r in range(0, c["rows"], 4096):
        x[r:r + 4096] = x[r:r + 4096] * fade + 0.1 * randc(x[r:r + 4096].shape, g)
    return x


def dpc_nodes(m, vy, vz):
    """Positions [P, 3] integrated from the velocities, with the velocities [P, 3]."""
    v = torch.stack([m["vx"], vy, vz], 1)
    p = torch.cat([m["p0"][None], m["p0"] + torch.cumsum(v[:-1] * m["dt"][:, None], 0)])
    return p, v


def dpc_footprints(c, m, vy, vz):
    p, _ = dpc_nodes(m, vy, vz)
    R, s = rotation(m["att"]), c["shift"]
    mid = p[:, None] + 0.5 * ((R @ m["tx"])[:, None] + torch.einsum("pij,cj->pci", R, m["rx"][s:]))
    mid = mid[:-1, :, None]                                              # [P-1, nc, 1, 3]
    ground = torch.sqrt(((0.5 * C_SOUND * m["t"]) ** 2 - mid[..., 2] ** 2).clamp_min(0.0))
    yaw = m["att"][:-1, 2][:, None, None]
    ps = torch.stack([mid[..., 0] - ground * torch.sin(yaw), mid[..., 1] + ground * torch.cos(yaw),
                      torch.zeros_like(ground)], -1)
    return ps.reshape(-1, 3).contiguous()


def dpc_residual(c, m, pv):
    """(path of ping i) - (path of ping i + 1) [P-1, nc, K] and its four leg vectors over their lengths."""
    p, v = pv
    R, s, K = rotation(m["att"]), c["shift"], c["K"]
    ltx, lrx = R @ m["tx"], torch.einsum("pij,cj->pci", R, m["rx"])
    ps = m["ps"].reshape(c["P"] - 1, c["C"] - s, K, 3)
    t = m["t"][:, None]
    a = (p + ltx)[:, None, None]
    b1 = (p[:-1, None] + lrx[:-1, s:])[:, :, None] + v[:-1, None, None] * t - ps
    b2 = (p[1:, None] + lrx[1:, :c["C"] - s])[:, :, None] + v[1:, None, None] * t - ps
    a1, a2 = a[:-1] - ps, a[1:] - ps
    n = [x.norm(dim=-1, keepdim=True) for x in (a1, b1, a2, b2)]
    return (n[0] + n[1] - n[2] - n[3])[..., 0], [x / y for x, y in zip((a1, b1, a2, b2), n)]


def dpc_exact(c, m):
    """Gauss-Newton on the motion loss (squares) with a dense Cholesky solve, to convergence."""
    P, K = c["P"], c["K"]
    dt, W = m["dt"], m["weight"].reshape(P - 1, c["C"] - c["shift"], K)
    n, lam1, lam2 = 2 * P, 1e-4, 1e-3
    f64 = dict(dtype=torch.float64, device=DEV)
    # velocities from the unknowns q = (positions 1 .. P-1, last velocity) per component: v = D q + d0
    D = torch.zeros((P, P), **f64)
    k = torch.arange(P - 1, device=DEV)
    D[k, k] = 1 / dt
    D[k[1:], k[1:] - 1] = -1 / dt[1:]
    D[P - 1, P - 1] = 1.0
    d0 = torch.zeros((P, 2), **f64)
    d0[0] = -m["p0"][1:] / dt[0]
    S = torch.zeros((P - 2, P), **f64)      # second differences of the velocities
    k = torch.arange(P - 2, device=DEV)
    S[k, k], S[k, k + 1], S[k, k + 2] = 1.0, -2.0, 1.0
    B = S @ D
    vy, vz = torch.zeros(P, **f64), torch.zeros(P, **f64)
    p, _ = dpc_nodes(m, vy, vz)
    q = torch.cat([p[1:, 1:], torch.stack([vy[-1:], vz[-1:]], 1)])                      # [P, 2]
    x = p[:, 0]
    loss = None
    for it in range(14):
        v = D @ q + d0
        pos = torch.cat([x[:, None], torch.cat([m["p0"][None, 1:], q[:-1]])], 1)
        r, (a1, b1, a2, b2) = dpc_residual(c, m, (pos, torch.cat([m["vx"][:, None], v], 1)))
        r = r + C_SOUND * m["delay"].reshape(r.shape)
        t = m["t"][:, None]
        # derivatives with respect to sway and heave of p_i, v_i, p_{i+1}, v_{i+1}
        J = torch.cat([a1 + b1, t * b1, -(a2 + b2), -t * b2], -1)[..., [1, 2, 4, 5, 7, 8, 10, 11]]
        J, rr, w = J.reshape(P - 1, -1, 8), r.reshape(P - 1, -1), W.reshape(P - 1, -1)
        Hl, gl = torch.einsum("pma,pm,pmb->pab", J, w, J), torch.einsum("pma,pm,pm->pa", J, w, rr)
        # scatter into (p_0 .. p_{P-1}, v_0 .. v_{P-1}) x (sway, heave), then map to q
        A = torch.zeros((4 * P, 4 * P), **f64)
        G = torch.zeros(4 * P, **f64)
        i = torch.arange(P - 1, device=DEV)
        idx = torch.stack([2 * i, 2 * i + 1, 2 * P + 2 * i, 2 * P + 2 * i + 1, 2 * i + 2, 2 * i + 3, 2 * P + 2 * i + 2,
                           2 * P + 2 * i + 3], 1)
        A.index_put_((idx[:, :, None].expand(-1, 8, 8), idx[:, None].expand(-1, 8, 8)), Hl, accumulate=True)
        G.index_put_((idx,), gl, accumulate=True)
        T = torch.zeros((4 * P, n), **f64)
        k = torch.arange(P - 1, device=DEV)
        for a in range(2):
            T[2 * (k + 1) + a, 2 * k + a] = 1.0
            T[2 * P + a::2, a::2] = D
        H, grad = T.T @ A @ T, T.T @ G
        sv, dz = S @ v, pos[:, 2] - m["z"]
        for a in range(2):
            H[a::2, a::2] += lam1 * B.T @ B
            grad[a::2] += lam1 * B.T @ sv[:, a]
        zi = 2 * k + 1
        H[zi, zi] += lam2
        grad[zi] += lam2 * dz[1:]
        loss = (w * rr * rr).sum() + lam1 * (sv * sv).sum() + lam2 * (dz * dz).sum()
        q = q - torch.cholesky_solve(grad[:, None], torch.linalg.cholesky(H))[:, 0].reshape(P, 2)
    v = D @ q + d0
    return [v[:, 0].contiguous(), v[:, 1].contiguous(), float(loss)]


def delays_exact(c, seed):
    e = dpc_echo(c, seed)
    P, s, W, L, nc = c["P"], c["shift"], c["W"], c["L"], c["C"] - c["shift"]
    n0 = dpc_centres(c).long() - W // 2
    pad = W + L
    co, fi, rho = [], [], []
    for i in range(P - 1):
        e2 = torch.nn.functional.pad(torch.view_as_real(e[i + 1, :nc]).transpose(1, 2).double(), (pad, pad))
        e1 = torch.nn.functional.pad(torch.view_as_real(e[i, s:]).transpose(1, 2).double(), (pad, pad))
        e1, e2 = torch.complex(e1[:, 0], e1[:, 1]), torch.complex(e2[:, 0], e2[:, 1])
        b = e2.unfold(1, W, 1)[:, n0 + pad]                                # [nc, K, W]
        a = e1.unfold(1, W + 2 * L, 1)[:, n0 + pad - L].unfold(2, W, 1)     # [nc, K, 2L+1 starts, W], start 2L - lag
        a = a.flip(2)                                                       # lag index t = tau + L
        Rt = torch.einsum("ckw,cktw->ckt", b, a.conj())
        mag = Rt.abs()
        best, t = mag.max(2)
        tt = t.clamp(1, 2 * L - 1) if L else t
        pick = lambda x, k: torch.gather(x, 2, k[..., None])[..., 0]  # noqa: E731
        inside = (t > 0) & (t < 2 * L)
        mm, mp = pick(mag, tt - 1), pick(mag, tt + 1)
        den = mm - 2 * best + mp
        d = torch.where(inside & (den != 0), 0.5 * (mm - mp) / den, torch.zeros_like(den))
        R0, Rm, Rp = pick(Rt, t), pick(Rt, tt - 1), pick(Rt, tt + 1)
        R = R0 + 0.5 * d * (Rp - Rm) + 0.5 * d * d * (Rp - 2 * R0 + Rm)
        co.append(((t - L + d) / FS).reshape(-1))
        fi.append((-torch.angle(R) / (2 * math.pi * FC)).reshape(-1))
        pa = pick(a.abs().square().sum(3), t)
        rho.append((best / torch.sqrt(b.abs().square().sum(2) * pa)).reshape(-1))
    return [torch.cat(co), torch.cat(fi), torch.cat(rho)]


def train_exact(c, seed):
    s = mlp_inputs(c, seed)
    th = s["theta"].double()
    half = s["theta"].half().double().requires_grad_()
    W1, b1, W2, b2, W3, b3 = torch.split(half, [64, 64, 4096, 64, 512, 8])
    x = (2.0 * s["f"] - 1.0).double()[:, None]
    gelu = torch.nn.functional.gelu
    a = gelu(gelu(x * W1 + b1) @ W2.reshape(64, 64).T + b2) @ W3.reshape(8, 64).T + b3
    r = (a * s["win"].to(torch.complex128)).sum(1) - s["y"].to(torch.complex128)
    loss = (r.real ** 2 + r.imag ** 2).mean()
    g, = torch.autograd.grad(loss, half)
    m, v = 0.9 * s["m"].double() + 0.1 * g, 0.999 * s["v"].double() + 0.001 * g * g
    k = s["step"]
    th = th - s["lr"] * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return [loss.detach().reshape(1), g, th, m, v]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("image", "volume", "autofocus", "adjoint"):
        upd = float(c["P"]) * c["C"] * c["nx"] * c["ny"] * c.get("nz", 1)
        if upd * (4 if kind == "autofocus" else 1) > EXACT_UPDATES or c.get("c_sed"):
            return None
        nav, echo, table = scene(c, seed)
        w = table.double() if table is not None else fine_table(4.0)
        if kind == "adjoint":
            return sums(c, nav, None, w, image=randc((c["ny"], c["nx"]), gen(seed)).reshape(-1).to(torch.complex128))
        if kind != "autofocus":
            return sums(c, nav, echo, w)
        dp = (1e-3 * torch.randn((c["P"], 3), device=DEV, generator=gen(seed + 5))).double()
        img = sums(c, nav, echo, w, dp=dp)
        p = img.real ** 2 + img.imag ** 2
        Dn, Nn = p.sum(), (p * p).sum()
        g = 2.0 * img * (p / Dn ** 2 - Nn / Dn ** 3)
        return [img, g, sums(c, nav, echo, w, g=g.reshape(-1), dp=dp)]
    if kind == "matched_filter":
        s = prepare(case, seed)
        rep = s["rep"].to(torch.complex128)
        n, out = c["n"], torch.empty((c["rows"], c["n"]), dtype=torch.complex128, device=DEV)
        spec = torch.fft.fft(rep, n + c["L"]).conj() / (rep.abs() ** 2).sum()
        for r in range(0, c["rows"], 1024):
            out[r:r + 1024] = torch.fft.ifft(torch.fft.fft(s["raw"][r:r + 1024].to(torch.complex128), n + c["L"]) * spec)[:, :n]
        return out
    if kind == "condition":
        x = condition_rows(c, seed).to(torch.complex128)
        X = torch.fft.fft(x)
        Pf = torch.zeros(c["n"], dtype=torch.float64, device=DEV)
        for r in range(0, c["rows"], 1024):
            Pf += X[r:r + 1024].abs().square().sum(0)
        Pf /= c["rows"]
        G = 1.0 / (c["gamma"] * Pf.mean() + Pf)
        wg = torch.sqrt(G / G.max())
        x = torch.fft.ifft(X * wg)
        del X
        med = torch.empty(c["n"], dtype=torch.float64, device=DEV)
        for k in range(0, c["n"], 256):
            p = torch.sort(x[:, k:k + 256].abs().square(), 0).values
            med[k:k + 256] = 0.5 * (p[(c["rows"] - 1) // 2] + p[c["rows"] // 2])
        tg = torch.sqrt(1.0 / (c["alpha"] * med.mean() + med))
        return [x * tg, wg, tg]
    if kind == "delays":
        return delays_exact(c, seed)
    if kind == "solve":
        return dpc_exact(c, dpc_motion(c, seed)) if c["P"] <= 1100 else None
    return train_exact(c, seed)
