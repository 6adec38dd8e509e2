"""Workloads of the library as its users run them, for timing and for comparing results.

A pass is what a program does between two looks at its flow: step one check interval, read the
residual it stops on and fetch the fields on the device.  Fields are kept in the precision of the
lattice's storage form (FP64 and FP32: density, velocity and shear rate; the FP16 forms: the
velocity, the quantity their accuracy is stated in).  Lattices step on the caller's stream, so that
a pass queues behind the one before it.

`exact` restates the method in plain torch FP64 (matrices of monomials and of the collision's basis,
pull streaming by shifts), from the same initial state.
"""
import math

import numpy as np
import torch

from paper_1908_05396_gb300 import clbm
from paper_1908_05396_gb300 import workloads as wl

U_LID = 0.05
STORED = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "f16r": torch.float16}
BYTES = {"f64": 8, "f32": 4, "f16s": 2, "f16r": 2}
FLOPS = 500  # arithmetic of one node update, about: moments, rate solve, relaxation, back-transform


def listed():
    return [
        # The paper's validation channel at its configured size: the smallest lattice anyone steps,
        # where a step costs a launch and one node's latency.
        dict(name="channel_4x64x4_f64", kind="lattice", flow="channel", nx=4, ny=64, nz=4, form="f64",
             steps=100, n=0.5, Re=20.0),
        # The smallest cavity of the serving and batching ranges, stepped alone.
        dict(name="cavity_32_f32", kind="lattice", flow="cavity", nx=32, ny=32, nz=32, form="f32",
             steps=100, n=0.8, Re=100.0),
        # The headline cavity, tuned as the README and the benchmark do it.
        dict(name="cavity_128_f32_tuned", kind="lattice", flow="cavity", nx=128, ny=128, nz=128,
             form="f32", steps=100, n=0.5, Re=100.0, tune=True),
        # The same cavity in FP64, the reference precision of every accuracy statement.
        dict(name="cavity_128_f64", kind="lattice", flow="cavity", nx=128, ny=128, nz=128, form="f64",
             steps=20, n=1.5, Re=100.0),
        # The precision study's cavity in the FP16 form that meets its bar everywhere.
        dict(name="cavity_256_f16r", kind="lattice", flow="cavity", nx=256, ny=256, nz=256,
             form="f16r", steps=20, n=0.8, Re=1000.0),
        # FP16 storage as specified, on a box whose sides are no multiple of anything.
        dict(name="cavity_161x97x130_f16s", kind="lattice", flow="cavity", nx=161, ny=97, nz=130,
             form="f16s", steps=40, n=1.2, Re=400.0),
        # FP16 storage with stochastic rounding, as the README's second example.
        dict(name="cavity_128_f16s_stochastic", kind="lattice", flow="cavity", nx=128, ny=128, nz=128,
             form="f16s", steps=40, n=0.8, Re=200.0, stochastic=True),
        # A forced, periodic, Newtonian duct in one buffer: the memory-saving option, the force path
        # and odd sizes together.
        dict(name="channel_203x90x77_f32_inplace", kind="lattice", flow="channel", nx=203, ny=90,
             nz=77, form="f32", steps=40, n=1.0, Re=50.0, in_place=True),
        # The configured batch: 64 uneven cavities, tuned, one check interval.
        dict(name="batch_64_f32_tuned", kind="batch", count=64, lo=32, hi=96, form="f32", steps=40,
             sizes=0, tune=True),
        # A burst of requests to the solve server: half cavities, half channels, results fetched.
        dict(name="serve_12_f16r", kind="serve", count=12, lo=32, hi=96, form="f16r", steps=400,
             sizes=1),
        # One check step between a caller's own buffers (fixed memory pools), dense odd-sized layout.
        dict(name="noalloc_97x65x83_f32", kind="noalloc", flow="cavity", nx=97, ny=65, nz=83,
             form="f32", n=0.7, Re=100.0),
        # Checkpoint and restart: the state from and to host memory, through the storage codec.
        dict(name="checkpoint_96_f16s", kind="checkpoint", flow="cavity", nx=96, ny=96, nz=96,
             form="f16s", n=0.8, Re=100.0),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cavity", "cavity", "cavity", "channel", "channel", "batch", "serve", "noalloc",
                       "checkpoint"])
    n = round(rng.uniform(0.5, 1.5), 3)
    if kind == "batch":
        form = rng.choice(["f32", "f16s", "f16r"])
        return dict(kind="batch", count=rng.randint(4, 40), lo=32, hi=rng.randint(48, 96), form=form,
                    steps=40, sizes=rng.randint(2, 1 << 20), tune=rng.random() < 0.5)
    if kind == "serve":
        return dict(kind="serve", count=rng.randint(4, 12), lo=32, hi=rng.randint(40, 96),
                    form=rng.choice(["f32", "f16r"]), steps=100 * rng.randint(1, 4),
                    sizes=rng.randint(2, 1 << 20))
    if kind == "noalloc":
        return dict(kind="noalloc", flow="cavity", nx=_log_uniform(rng, 24, 160),
                    ny=_log_uniform(rng, 24, 160), nz=_log_uniform(rng, 24, 160),
                    form=rng.choice(["f32", "f64"]), n=n, Re=round(rng.uniform(50, 400), 1))
    if kind == "checkpoint":
        L = _log_uniform(rng, 24, 110)
        return dict(kind="checkpoint", flow="cavity", nx=L, ny=L + rng.randint(0, 9), nz=L,
                    form=rng.choice(["f64", "f32", "f16s", "f16r"]), n=n, Re=100.0)
    form = rng.choice(["f64", "f32", "f32", "f16s", "f16s", "f16r"])
    top = 128 if form == "f64" else 224
    if kind == "cavity":
        L = _log_uniform(rng, 24, top)
        size = dict(nx=L, ny=max(16, L - rng.randint(0, 7)), nz=max(16, L - rng.randint(0, 5)))
    elif rng.random() < 0.5:  # the narrow channels of the serving trace
        size = dict(nx=8, ny=_log_uniform(rng, 32, 256), nz=8)
    else:
        H = _log_uniform(rng, 24, top)
        size = dict(nx=max(16, H - rng.randint(0, 9)), ny=H, nz=max(8, H // rng.randint(1, 4)))
    nodes = size["nx"] * size["ny"] * size["nz"]
    c = dict(kind="lattice", flow=kind, form=form, steps=100 if nodes < 3e5 else 20,
             n=n if rng.random() < 0.75 else 1.0, Re=round(rng.uniform(50, 400), 1), **size)
    if form == "f16s" and rng.random() < 0.5:
        c["stochastic"] = True
    elif form in ("f32", "f16s") and rng.random() < 0.25:
        c["in_place"] = True
    return c


def _problem(case, seed):
    """The case's flow; the seed moves its Reynolds number by up to a tenth."""
    Re = case["Re"] * float(np.random.default_rng(seed).uniform(0.9, 1.1))
    dims = (case["nx"], case["ny"], case["nz"])
    if case["flow"] == "cavity":
        return wl.cavity(case["ny"], Re, case["n"], U=U_LID, dims=dims)
    return wl.channel(case["ny"], case["n"], u_max=U_LID, Re=Re, nx=case["nx"], nz=case["nz"])


def _problems(case, seed):
    """The uneven flows of a batch or of a burst of requests: sizes from the case, Re and n from the seed."""
    size, rng = np.random.default_rng(case["sizes"]), np.random.default_rng(seed)
    out = []
    for k in range(case["count"]):
        L = int(size.integers(case["lo"], case["hi"] + 1))
        Re, n = float(rng.uniform(50.0, 300.0)), float(rng.uniform(0.6, 1.4))
        if case["kind"] == "serve" and k % 2:
            out.append(wl.channel(2 * L, n, u_max=0.02, Re=Re, nx=8, nz=8))
        else:
            out.append(wl.cavity(L, Re, n, U=U_LID))
    return out


EX = np.array([0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0])
EY = np.array([0, 0, 0, 1, -1, 0, 0, 1, 1, -1, -1, 0, 0, 0, 0, 1, -1, 1, -1])
EZ = np.array([0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, 1, -1, -1, 1, 1, -1, -1])
WT = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
OPP = [int(np.flatnonzero((EX == -EX[q]) & (EY == -EY[q]) & (EZ == -EZ[q]))[0]) for q in range(19)]


def _initial(p, seed):
    """A developing flow: the equilibrium of a few smooth random modes that vanish at the walls,
    velocities up to about the lid's, the density a tenth of a per cent around 1.001."""
    g = np.random.default_rng(seed + 7919)
    ax = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) / m for m in (p.nz, p.ny, p.nx)]
    wall = [p.face[4] != 0, p.face[2] != 0, p.face[0] != 0]

    def mode():
        v = [torch.sin(math.pi * int(g.integers(1, 4)) * a) if w
             else torch.cos(2 * math.pi * (int(g.integers(0, 3)) * a + float(g.uniform())))
             for a, w in zip(ax, wall)]
        return v[0][:, None, None] * v[1][None, :, None] * v[2][None, None, :]

    u = [sum(float(g.uniform(-0.4, 0.4)) * mode() for _ in range(4)) * U_LID for _ in range(3)]
    rho = 1.001 + 1e-3 * sum(float(g.uniform(-0.5, 0.5)) * mode() for _ in range(3))
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    f = torch.empty((19,) + rho.shape, dtype=torch.float64, device="cuda")
    for q in range(19):
        eu = float(EX[q]) * u[0] + float(EY[q]) * u[1] + float(EZ[q]) * u[2]
        f[q] = WT[q] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu)
    return f


def _lattice(case, p, stream):
    lat = clbm.Lattice(**p.kwargs(), dtype=case["form"], check_interval=case.get("steps", 100),
                       in_place=case.get("in_place", False),
                       stream=stream.cuda_stream if stream else None)
    if case.get("stochastic"):
        lat.set_rounding("stochastic")
    return lat


def prepare(case, seed):
    kind, s = case["kind"], dict(case=case)
    if kind in ("lattice", "checkpoint", "noalloc"):
        p = _problem(case, seed)
        f = _initial(p, seed)
        s["stream"] = torch.cuda.Stream()
        shape = (p.nz, p.ny, p.nx)
    if kind == "lattice":
        s["lat"] = _lattice(case, p, s["stream"])
        s["lat"].set_state(f.cpu().numpy())
        if case.get("tune"):
            s["lat"].autotune()
        s["u"] = torch.empty((3,) + shape, dtype=torch.float64, device="cuda")
        if not case["form"].startswith("f16"):
            s["rho"], s["gd"] = (torch.empty(shape, dtype=torch.float64, device="cuda") for _ in "ab")
    elif kind == "checkpoint":
        s["lat"] = _lattice(case, p, None)
        s["f"] = f.cpu().numpy()
    elif kind == "noalloc":
        dt = STORED[case["form"]]
        w = torch.tensor(WT, device="cuda")[:, None, None, None]
        s["p"], s["bufs"] = p, [(f - w).to(dt), torch.zeros((19,) + shape, dtype=dt, device="cuda")]
        s["u_prev"] = torch.zeros((3,) + shape, dtype=dt, device="cuda")
        s["stats"] = torch.zeros(4, dtype=torch.float64, device="cuda")
    elif kind == "batch":
        s["stream"] = torch.cuda.Stream()
        probs = _problems(case, seed)
        s["lats"] = [_lattice(case, p, s["stream"]) for p in probs]
        s["batch"] = clbm.Batch(case["form"], capacity=case["count"], check_interval=case["steps"],
                                stream=s["stream"].cuda_stream)
        for lat in s["lats"]:
            s["batch"].add(lat)
        if case.get("tune"):
            s["batch"].autotune()
        s["u"] = torch.empty(sum(3 * p.N for p in probs), dtype=torch.float64, device="cuda")
    else:
        s["server"] = clbm.Server(case["form"], max_active=case["count"], check_interval=100)
        s["probs"] = _problems(case, seed)
    torch.cuda.synchronize()
    return s


def run(state):
    case = state["case"]
    return {"lattice": _run_lattice, "checkpoint": _run_checkpoint, "noalloc": _run_noalloc,
            "batch": _run_batch, "serve": _run_serve}[case["kind"]](state, case)


def _run_lattice(s, case):
    lat, dt = s["lat"], STORED[case["form"]]
    lat.step(case["steps"])
    R, _ = lat.residual()
    with torch.cuda.stream(s["stream"]):
        if "rho" not in s:
            lat.fields_device(u=s["u"])
            return dict(u=s["u"].to(dt))
        lat.fields_device(s["rho"], s["u"], s["gd"])
        return dict(rho=s["rho"].to(dt), u=s["u"].to(dt), gd=s["gd"].to(dt),
                    R=np.array([R], dtype=np.float64 if dt == torch.float64 else np.float32))


def _run_checkpoint(s, case):
    s["lat"].set_state(s["f"])
    return dict(f=s["lat"].get_state())


def _run_noalloc(s, case):
    p, (src, dst) = s["p"], s["bufs"]
    with torch.cuda.stream(s["stream"]):
        rc = clbm.step_noalloc(p.nx, p.ny, p.nz, p.face, p.K, p.n, p.U_lid, p.body_force, case["form"],
                               src.data_ptr(), dst.data_ptr(), s["u_prev"].data_ptr(),
                               s["stats"].data_ptr(), stream=s["stream"].cuda_stream)
        if rc != clbm.OK:
            raise RuntimeError(clbm.last_error())
        s["bufs"] = [dst, src]
        return dict(f=dst, u=s["u_prev"], stats=s["stats"].to(dst.dtype))


def _run_batch(s, case):
    s["batch"].step(case["steps"])
    st = s["batch"].stats_all()
    at = 0
    with torch.cuda.stream(s["stream"]):
        for lat in s["lats"]:
            lat.fields_device(u=s["u"][at:at + 3 * lat.N])
            at += 3 * lat.N
        return dict(u=s["u"].to(STORED[case["form"]]), steps=st["steps"])


def _run_serve(s, case):
    srv, kept = s["server"], np.float32 if case["form"] == "f32" else np.float16
    ids = [srv.submit(**p.kwargs(), tol=0.0, max_steps=case["steps"], keep_fields=True)
           for p in s["probs"]]
    u, steps = [], []
    for rid in ids:
        steps.append(srv.wait(rid)["steps"])
        u.append(srv.fields(rid)[1].astype(kept).reshape(-1))
        srv.release(rid)
    return dict(u=np.concatenate(u), steps=np.array(steps))


def _nodes(case):
    if "nx" in case:
        return case["nx"] * case["ny"] * case["nz"]
    return sum(p.N for p in _problems(case, 0))


def work(case):
    N, b, kind = _nodes(case), BYTES[case["form"]], case["kind"]
    pops = 19 * b + (8 if case["form"] == "f16r" else 0)
    if kind == "checkpoint":
        return dict(bytes=2 * N * (19 * 8 + pops), flops=2 * 19 * N)
    if kind == "noalloc":
        return dict(bytes=N * 2 * (pops + 3 * b), flops=FLOPS * N)
    # every step reads and writes the populations; the fields read them once and write FP64
    fields = 40 if not case["form"].startswith("f16") and kind == "lattice" else 24
    return dict(bytes=N * (case["steps"] * 2 * pops + pops + fields),
                flops=FLOPS * N * (case["steps"] + 1))


# ---- the method in plain FP64 ------------------------------------------------------------------

def _tables():
    x, y, z = (torch.tensor(e, dtype=torch.float64, device="cuda") for e in (EX, EY, EZ))
    o, e2 = torch.ones_like(x), x * x + y * y + z * z
    mono = torch.stack([o, x, y, z, x * x, y * y, z * z, x * y, x * z, y * z, x * y * y, x * z * z,
                        x * x * y, y * z * z, x * x * z, y * y * z, x * x * y * y, x * x * z * z,
                        y * y * z * z])
    basis = torch.stack([x * y, x * z, y * z, x * x - y * y, x * x + y * y - 2 * z * z, 19 * e2 - 30,
                         5 * x * e2 - 9 * x, 5 * y * e2 - 9 * y, 5 * z * e2 - 9 * z,
                         x * y * y - x * z * z, y * z * z - y * x * x, z * x * x - z * y * y,
                         21 * mono[16:].sum(0) - 16 * e2 + 12,
                         3 * (mono[16] + mono[17] - 2 * mono[18]) - 2 * (2 * x * x - y * y - z * z),
                         3 * (mono[16] - mono[17]) - 2 * (y * y - z * z)], 1)
    return mono, basis


def _rate(p, rho, A, B):
    """omega and the shear rate: y = log(1/omega - 1/2) solves y = log(3 K / rho) + (n-1)/2 log(gd^2),
    gd^2 = omega^2 A + B, clamped to the library's default viscosity bounds."""
    lo, hi = math.log(3 * 5e-4), math.log(30.0)
    c = math.log(3 * p.K) - torch.log(rho)
    y = (c + 0.5 * (p.n - 1) * torch.log((A + B).clamp_min(1e-300))).clamp(lo, hi)
    for _ in range(14):
        tau = torch.exp(y)
        w = 1 / (tau + 0.5)
        g2 = (w * w * A + B).clamp_min(1e-300)
        G = y - c - 0.5 * (p.n - 1) * torch.log(g2)
        y = (y - G / (1 + (p.n - 1) * (w * w * A / g2) * tau * w)).clamp(lo, hi)
    w = 1 / (torch.exp(y) + 0.5)
    return w, torch.sqrt(w * w * A + B)


def _node(p, T, d):
    """Moments, velocity and rate of the deviations d (19, N) from rest at density 1."""
    F = p.body_force
    rho, w = 1 + d.sum(0), torch.tensor(WT, device="cuda")
    j = T[0][1:4] @ d
    u = [(j[a] + 0.5 * F[a]) / rho for a in range(3)]
    S = None
    if any(F):
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        S = torch.empty_like(d)
        for q in range(19):
            e = (float(EX[q]), float(EY[q]), float(EZ[q]))
            eF = sum(a * b for a, b in zip(e, F))
            S[q] = w[q] * (3 * eF + 9 * eF * (e[0] * u[0] + e[1] * u[1] + e[2] * u[2]) - 3 * uF)
        d = d + 0.5 * S
    D = T[0] @ d
    ux, uy, uz = u
    m = [D[7] - rho * ux * uy, D[8] - rho * ux * uz, D[9] - rho * uy * uz,
         D[4] - D[5] - rho * (ux * ux - uy * uy), D[4] - D[6] - rho * (ux * ux - uz * uz),
         D[4] + D[5] + D[6] - (rho - 1) - rho * (ux * ux + uy * uy + uz * uz)]
    A = 3 / rho ** 2 * (m[3] ** 2 - m[3] * m[4] + m[4] ** 2 + 3 * (m[0] ** 2 + m[1] ** 2 + m[2] ** 2))
    B = 1.5 / rho ** 2 * m[5] ** 2
    om, gd = _rate(p, rho, A, B)
    return d, S, D, rho, u, m, om, gd


def _collide(p, T, d):
    d, S, D, rho, (ux, uy, uz), m, om, _ = _node(p, T, d)
    third = 1 / 3
    Dxx, Dyy, Dzz, Dxy, Dxz, Dyz = D[4:10]
    Dxyy, Dxzz, Dxxy, Dyzz, Dxxz, Dyyz, Dxxyy, Dxxzz, Dyyzz = D[10:19]
    kxx, kyy, kzz = third + Dxx, third + Dyy, third + Dzz
    g4, g5, g6 = (-0.25 * om * v for v in m[:3])
    g7, g8 = -om * m[3] / 12, -om * (2 * m[4] - m[3]) / 36
    g9 = -m[5] / 126

    def row(a, kbb, Dabb, b, Dab):
        return a * kbb - Dabb + 2 * b * Dab - 2 * rho * a * b * b

    Xy, Xz = row(ux, kyy, Dxyy, uy, Dxy), row(ux, kzz, Dxzz, uz, Dxz)
    Yx, Yz = row(uy, kxx, Dxxy, ux, Dxy), row(uy, kzz, Dyzz, uz, Dyz)
    Zx, Zy = row(uz, kxx, Dxxz, ux, Dxz), row(uz, kyy, Dyyz, uy, Dyz)
    g10 = (Xy + Xz) / 8 + uy * g4 + uz * g5 + 0.75 * ux * (14 * g9 - g7 - g8)
    g13 = (Xy - Xz) / 8 + uy * g4 - uz * g5 + 0.75 * ux * (3 * g8 - g7)
    g11 = (Yx + Yz) / 8 + ux * g4 + uz * g6 + 0.75 * uy * (14 * g9 + g7 - g8)
    g14 = (Yz - Yx) / 8 + uz * g6 - ux * g4 - 0.75 * uy * (g7 + 3 * g8)
    g12 = (Zx + Zy) / 8 + ux * g5 + uy * g6 + 1.5 * uz * (g8 + 7 * g9)
    g15 = (Zx - Zy) / 8 + ux * g5 - uy * g6 + 1.5 * uz * g7
    x2, y2, z2 = ux * ux, uy * uy, uz * uz
    ax = Dxx - third * (rho - 1) - rho * x2 + 6 * g7 + 6 * g8 + 42 * g9
    ay = Dyy - third * (rho - 1) - rho * y2 - 6 * g7 + 6 * g8 + 42 * g9
    az = Dzz - third * (rho - 1) - rho * z2 - 12 * g8 + 42 * g9

    def pair(aa, ab, Daabb, a, b, Dabb, Daab, kaa, kbb, Dab):
        return (aa * ab / rho - Daabb + 2 * a * Dabb + 2 * b * Daab - a * a * kbb - b * b * kaa
                - 4 * a * b * Dab + 3 * rho * a * a * b * b)

    Wxy = pair(ax, ay, Dxxyy, ux, uy, Dxyy, Dxxy, kxx, kyy, Dxy)
    Wxz = pair(ax, az, Dxxzz, ux, uz, Dxzz, Dxxz, kxx, kzz, Dxz)
    Wyz = pair(ay, az, Dyyzz, uy, uz, Dyzz, Dyyz, kyy, kzz, Dyz)
    b16 = third * (rho - 1) + 2 * third * (ax + ay + az) + Wxy + Wxz + Wyz
    b17 = third * (2 * ax - ay - az) + Wxy + Wxz - 2 * Wyz
    b18 = third * (ay - az) + Wxy - Wxz
    p4, p5, p6 = ux * uy * g4, ux * uz * g5, uy * uz * g6
    v10, v11, v12 = ux * g10, uy * g11, uz * g12
    g16 = (b16 / 12 - 4 * third * (p4 + p5 + p6) + 0.5 * (x2 - y2) * g7
           + 0.5 * (x2 + y2 - 2 * z2) * g8 - (7 * (x2 + y2 + z2) + 8) * g9
           + 4 * third * (v10 + v11 + v12))
    g17 = (b17 / 24 - 2 * third * (p4 + p5) + 4 * third * p6 + 0.25 * (x2 - y2 - 3 * z2 - 2) * g7
           + 0.25 * (x2 - 5 * y2 + z2 - 2) * g8 + 1.75 * (y2 + z2 - 2 * x2) * g9
           + 2 * third * v10 - third * (v11 + v12) - uy * g14 + uz * g15)
    g18 = (b18 / 8 - 2 * (p4 - p5) + 0.75 * (x2 - y2 + z2 + 2 * third) * g7
           + 0.75 * (z2 - y2 - 3 * x2 - 2) * g8 + 5.25 * (z2 - y2) * g9 + v11 - v12
           + 2 * ux * g13 - uy * g14 - uz * g15)
    d = d + T[1] @ torch.stack([g4, g5, g6, g7, g8, g9, g10, g11, g12, g13, g14, g15, g16, g17, g18])
    return d if S is None else d + 0.5 * S


def _pull(p, d):
    """Stream: shift every direction, then bounce back what crossed a wall, the lid's term last."""
    out = torch.empty_like(d)
    for q in range(19):
        e = (int(EZ[q]), int(EY[q]), int(EX[q]))
        out[q] = torch.roll(d[q], e, (0, 1, 2))
        for lid in (False, True):
            for a in range(3):
                kind = p.face[2 * (2 - a) + (0 if e[a] > 0 else 1)]
                if e[a] == 0 or kind == wl.PERIODIC or (kind == wl.LID) != lid:
                    continue
                at = [slice(None)] * 3
                at[a] = 0 if e[a] > 0 else d.shape[1 + a] - 1
                term = 6 * WT[q] * (EX[q] * p.U_lid[0] + EY[q] * p.U_lid[1] + EZ[q] * p.U_lid[2])
                out[q][tuple(at)] = d[OPP[q]][tuple(at)] + (float(term) if lid else 0.0)
    return out


def _flow(p, T, d, steps):
    """(rho, u, gd) after `steps` steps from the deviations d, and the deviations."""
    shape = d.shape
    for _ in range(steps):
        d = _collide(p, T, _pull(p, d).reshape(19, -1)).reshape(shape)
    _, _, _, rho, u, _, _, gd = _node(p, T, _pull(p, d).reshape(19, -1))
    return rho.reshape(shape[1:]), torch.stack(u).reshape((3,) + shape[1:]), gd.reshape(shape[1:]), d


def exact(case, seed):
    kind = case["kind"]
    T, w = _tables(), torch.tensor(WT, device="cuda")[:, None, None, None]
    if kind in ("batch", "serve"):
        u = [_flow(p, T, torch.zeros((19, p.nz, p.ny, p.nx), dtype=torch.float64, device="cuda"),
                   case["steps"])[1].reshape(-1) for p in _problems(case, seed)]
        return dict(u=torch.cat(u), steps=None)
    p = _problem(case, seed)
    f = _initial(p, seed)
    if kind == "checkpoint":
        return dict(f=f.cpu().numpy())
    if kind == "noalloc":
        d = _pull(p, f - w)
        _, _, _, rho, u, _, _, _ = _node(p, T, d.reshape(19, -1))
        u = torch.stack(u)
        uu = (u * u).sum()
        stats = torch.stack([uu, uu, (rho - 1).sum(), torch.zeros_like(uu)])
        out = _collide(p, T, d.reshape(19, -1))
        return dict(f=out.reshape(f.shape), u=u.reshape((3,) + f.shape[1:]), stats=stats)
    rho, u, gd, _ = _flow(p, T, f - w, case["steps"])
    return dict(u=u) if case["form"].startswith("f16") else dict(rho=rho, u=u, gd=gd, R=None)
