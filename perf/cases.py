"""The work that users of this framework have it do, as cases that can be timed and checked.

Five families, each through the public binding: one frame's cube (`frame`, six arithmetic
tiers, device or host buffers), a batch of frames of an animation (`batch`), the
range-Doppler processing of a run of cubes (`doppler`), the rendering of an analytic scene
(`raycast`) and a burst of mixed requests to the server (`serve`).  The sizes are those of
the package's configs/config1..5.json, the serving mix and the tests; `draw` spreads over
the same ranges, ragged sizes among them.
"""
import math

import numpy as np
import torch

from paper_2307_09226_gb300 import _abi, device
from paper_2307_09226_gb300.synth import Radar

C_LIGHT = 299_792_458.0
LAM, MU, FS, T_B = 3.9e-3, 3.0e13, 1.0e7, 6.0e-5
FIELDS = ("range", "sigma_re", "sigma_im", "az", "el", "vel")
AZ, EL = (-math.pi / 3, math.pi / 3), (-math.pi / 6, math.pi / 6)


def _frame(name, tier, M, N, Ns, L, n_az, n_el, mask, px="f32", host=False):
    return {"name": name, "kind": "frame", "tier": tier, "M": M, "N": N, "Ns": Ns, "L": L, "n_az": n_az, "n_el": n_el,
            "mask": mask, "px": px, "host": host}


def _batch(name, tier, frames, grid, M, N, Ns, L):
    return {"name": name, "kind": "batch", "tier": tier, "frames": frames, "grid": grid, "M": M, "N": N, "Ns": Ns, "L": L}


def _doppler(name, frames, M, N, Ns, L):
    return {"name": name, "kind": "doppler", "frames": frames, "M": M, "N": N, "Ns": Ns, "L": L}


def _raycast(name, n_az, n_el, prims, px="f32"):
    return {"name": name, "kind": "raycast", "n_az": n_az, "n_el": n_el, "prims": prims, "px": px}


def _serve(name, requests, mix_seed, max_grid, most):
    return {"name": name, "kind": "serve", "requests": requests, "mix_seed": mix_seed, "max_grid": max_grid, "most": most}


def listed():
    return [
        # the smallest call in use: a 32 x 32-pixel frame with FP64 render buffers (config 1),
        # as a real-time loop on a coarse render calls it; latency and launches count
        _frame("small_fp32", "fp32", 2, 4, 64, 32, 32, 32, 0.0, px="f64"),
        # ragged everything (rows, columns and pixels off every tile) in plain 16 bits: a quick look
        _frame("ragged_bf16", "bf16", 2, 3, 96, 48, 71, 70, 0.3),
        # config 2: one 256 x 256-pixel frame, 30% background, in the plain FP32 tier
        _frame("frame_fp32", "fp32", 3, 4, 256, 128, 256, 256, 0.3),
        # config 3: the same frame in the split-precision tensor-core tier
        _frame("frame_split_fp16", "split_fp16", 3, 4, 256, 128, 256, 256, 0.3),
        # the same frame through the gridding tier
        _frame("frame_nufft", "nufft", 3, 4, 256, 128, 256, 256, 0.3),
        # the same frame from page-locked host buffers and back, waited for: the end-to-end call
        _frame("host_split_fp16", "split_fp16", 3, 4, 256, 128, 256, 256, 0.3, host=True),
        # the largest request of the serving mix
        _frame("large_split_bf16", "split_bf16", 4, 12, 512, 256, 512, 512, 0.3),
        # config 4: a walking animation of 64 frames with uneven pixel counts in one call
        _batch("walk_split_fp16", "split_fp16", 64, 256, 3, 4, 256, 128),
        # the same animation through the gridding tier
        _batch("walk_nufft", "nufft", 64, 256, 3, 4, 256, 128),
        # target estimation on the animation's 64 cubes (the Doppler-time plot)
        _doppler("walk_doppler", 64, 3, 4, 256, 128),
        # one rendered frame of a dozen primitives: the step before the synthesis
        _raycast("render", 256, 256, 12),
        # config 5: a burst of 16 requests of mixed radars, sizes and tiers on the server
        _serve("serve_burst", 16, 5, 512, 3e11),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "batch", "doppler", "raycast", "serve"])
    if kind == "frame":
        tier = rng.choice(["fp32", "bf16", "fp16", "split_bf16", "split_fp16", "nufft"])
        host = rng.random() < 0.2
        # no more path-samples than the largest listed call of the tier does in its time
        most = 9e10 if tier == "fp32" else 1.1e12
        while True:
            c = _frame("", tier, rng.randint(1, 4), rng.randint(1, 12), _log_int(rng, 32, 512), _log_int(rng, 12, 256),
                       _log_int(rng, 32, 512), _log_int(rng, 32, 512), rng.choice([0.0, 0.3, rng.uniform(0.05, 0.9)]),
                       px=rng.choice(["f32", "f32", "f64"]), host=host)
            if c["M"] * c["N"] * c["Ns"] * c["L"] * c["n_az"] * c["n_el"] <= most:
                break
    elif kind == "batch":
        c = _batch("", rng.choice(["split_fp16", "split_bf16", "nufft"]), _log_int(rng, 4, 64), _log_int(rng, 64, 256),
                   rng.randint(1, 3), 4, rng.choice([64, 128, 200, 256]), rng.choice([32, 64, 100, 128]))
    elif kind == "doppler":
        c = _doppler("", _log_int(rng, 1, 64), rng.randint(1, 3), rng.randint(1, 4), rng.choice([32, 64, 128, 256, 512]),
                     rng.choice([16, 32, 64, 128, 256]))
    elif kind == "raycast":
        c = _raycast("", _log_int(rng, 64, 600), _log_int(rng, 64, 600), _log_int(rng, 3, 100), px=rng.choice(["f32", "f32", "f64"]))
    else:
        c = _serve("", rng.randint(4, 16), rng.randint(0, 10_000), rng.choice([128, 256]), 5e10)
    del c["name"]
    return c


# ----------------------------------------------------------------------------------
# Inputs, from the seed alone
# ----------------------------------------------------------------------------------

def _radar(c):
    return Radar(M=c["M"], N=c["N"], Ns=c["Ns"], L=c["L"], lam=LAM, mu=MU, fs=FS, t_b=T_B)


def _angles(n_az, n_el):
    az = AZ[0] + (np.arange(n_az) + 0.5) * (AZ[1] - AZ[0]) / n_az
    el = EL[0] + (np.arange(n_el) + 0.5) * (EL[1] - EL[0]) / n_el
    return np.tile(az, n_el), np.repeat(el, n_az)


def _strength(rng, n, mean=0.0, sd=1.0):
    s = np.exp(rng.normal(mean, sd, n)) * np.exp(2j * np.pi * rng.random(n))
    return s.real, s.imag


def _scatter_pixels(c, seed):
    """Uniform ranges and speeds, log-normal strengths of uniform phase, a random background."""
    rng = np.random.default_rng([seed, 1])
    P = c["n_az"] * c["n_el"]
    az, el = _angles(c["n_az"], c["n_el"])
    rr = rng.uniform(0.5, 8.0, P)
    sre, sim = _strength(rng, P)
    vel = rng.uniform(-2.0, 2.0, P)
    if c["mask"] > 0:
        miss = rng.random(P) < c["mask"]
        sre[miss] = sim[miss] = 0.0
        rr[miss] = np.inf
    return (rr, sre, sim, az, el, vel)


def _walk_pixels(grid, f, seed):
    """One animation frame: a pedestrian's block of pixels before a sparse static wall."""
    rng = np.random.default_rng([seed, 2, f])
    P = grid * grid
    share = P / 65536.0
    az, el = _angles(grid, grid)
    rr = np.full(P, np.inf)
    sre, sim, vel = np.zeros(P), np.zeros(P), np.zeros(P)
    n_ped = int(rng.integers(2000, 20001) * share) + 1
    n_wall = int(rng.integers(0, 45001) * share)
    ph = 2.0 * np.pi * f / 64.0
    w = min(max(1, int(round(math.sqrt(n_ped / 2.5)))), grid)
    h = min(-(-n_ped // w), grid)
    i0 = min(max(int((40.0 * math.sin(ph) + 60.0) / 120.0 * grid) - w // 2, 0), grid - w)
    j0 = (grid - h) // 2
    ped = ((j0 + np.arange(h))[:, None] * grid + i0 + np.arange(w)[None, :]).ravel()[:n_ped]
    free = np.ones(P, bool)
    free[ped] = False
    wall = np.flatnonzero(free & (rng.random(P) < n_wall / P))
    rr[ped] = 3.0 + 2.0 * math.sin(ph + 0.7) + rng.uniform(-0.3, 0.3, ped.size)
    vel[ped] = np.clip(1.5 * math.sin(ph) + rng.uniform(-1.5, 1.5, ped.size), -3.0, 3.0)
    sre[ped], sim[ped] = _strength(rng, ped.size)
    rr[wall] = np.minimum(6.0 / (np.cos(az[wall]) * np.cos(el[wall])), 8.0)
    sre[wall], sim[wall] = _strength(rng, wall.size, -1.0, 0.5)
    return (rr, sre, sim, az, el, vel)


def _typed(px, kind):
    return tuple(np.ascontiguousarray(a, dtype=np.float64 if kind == "f64" else np.float32) for a in px)


def _upload(px):
    return {k: torch.from_numpy(a).cuda() for k, a in zip(FIELDS, px)}


def _mix(c):
    """The burst's requests: radars, grids and tiers of config 5, drawn by the case's own seed."""
    rng = np.random.default_rng([c["mix_seed"], 3])
    out = []
    while len(out) < c["requests"]:
        pick = lambda *xs: int(rng.choice(xs))
        q = {"M": pick(2, 3, 4), "N": pick(4, 8, 12), "Ns": pick(128, 256, 512), "L": pick(64, 128, 256),
             "n_az": pick(64, 128, 256, 512), "mask": 0.3, "tier": str(rng.choice(["fp32", "split_bf16"]))}
        q["n_el"] = q["n_az"]
        # a burst is many ordinary requests: one that alone outweighs the others is left to the frame cases
        if q["n_az"] <= c["max_grid"] and q["M"] * q["N"] * q["Ns"] * q["L"] * q["n_az"] ** 2 <= c["most"]:
            out.append(q)
    return out


def _cubes(c, seed):
    """Cubes of 48 moving point targets each over a little noise, computed in 64 bits."""
    g = torch.Generator(device="cpu").manual_seed(seed * 7919 + 11)
    V, Ns, L, K = c["M"] * c["N"], c["Ns"], c["L"], 48
    out = []
    for _ in range(c["frames"]):
        r = torch.rand(5, K, generator=g, dtype=torch.float64).cuda()
        amp = torch.exp(2.0 * r[0] - 1.0)
        fast = 0.25 * r[1][:, None] * torch.arange(Ns, device="cuda", dtype=torch.float64)[None, :]
        chan = (r[2][:, None] - 0.5) * torch.arange(V, device="cuda", dtype=torch.float64)[None, :] + r[3][:, None]
        slow = (r[4][:, None] - 0.5) * torch.arange(L, device="cuda", dtype=torch.float64)[None, :]
        cis = lambda x: torch.polar(torch.ones_like(x), 2.0 * math.pi * x)
        A = (amp[:, None, None] * cis(chan)[:, :, None] * cis(fast)[:, None, :]).reshape(K, V * Ns)
        x = (A.T @ cis(slow)).reshape(V, Ns, L)
        noise = torch.randn(2, V, Ns, L, generator=torch.Generator(device="cuda").manual_seed(int(1e6 * float(r[0, 0])) + seed),
                            device="cuda", dtype=torch.float32)
        out.append((x + 0.1 * torch.complex(noise[0], noise[1])).to(torch.complex64).contiguous())
    return out


def _scene(c, seed):
    """Ellipsoids, capsules and parallelograms before the radar, as an animation step gives them."""
    rng = np.random.default_rng([seed, 4])
    scene = []
    for k in range(c["prims"]):
        rr, az, el = rng.uniform(1.5, 8.0), rng.uniform(-0.87, 0.87), rng.uniform(-0.43, 0.43)
        ctr = rr * np.array([math.cos(el) * math.sin(az), math.cos(el) * math.cos(az), math.sin(el)])
        ax = np.linalg.qr(rng.normal(size=(3, 3)))[0].T
        zero = np.zeros(3)
        p = {"kind": ("plane", "capsule", "ellipsoid")[k % 3], "d": zero, "vel": rng.uniform(-2, 2, 3),
             "omega": rng.uniform(-3, 3, 3), "rho": float(rng.uniform(0.2, 1.0))}
        if p["kind"] == "ellipsoid":
            s = rng.uniform(0.2, 0.8, 3)
            p |= {"a": ctr, "b": ax[0] * s[0], "c": ax[1] * s[1], "d": ax[2] * s[2]}
        elif p["kind"] == "capsule":
            half = 0.5 * rng.uniform(0.3, 1.5)
            p |= {"a": ctr - half * ax[0], "b": ctr + half * ax[0], "c": np.array([rng.uniform(0.05, 0.3), 0.0, 0.0])}
        else:
            b, d = ax[0] * rng.uniform(0.5, 3.0), ax[1] * rng.uniform(0.5, 3.0)
            p |= {"a": ctr - 0.5 * (b + d), "b": b, "c": d}
        scene.append(p)
    return scene


# ----------------------------------------------------------------------------------
# prepare / run
# ----------------------------------------------------------------------------------

class _Server:
    """A server on a context, closed with the state that holds it."""

    def __init__(self, ctx):
        self.ctx = ctx
        self.h = _abi.rsim_server_create(ctx.h, slots=3, express_slots=5)

    def __del__(self):
        _abi.rsim_server_destroy(self.h)


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c, "ctx": device.Context(0)}
    if kind == "frame":
        px = _typed(_scatter_pixels(c, seed), c["px"])
        st["radar"] = _radar(c)
        if c["host"]:
            st["px"] = {k: torch.from_numpy(a).pin_memory() for k, a in zip(FIELDS, px)}
            st["cube"] = device.cube_tensor(st["radar"], device="cpu").pin_memory()
        else:
            st["px"] = _upload(px)
            st["cube"] = device.cube_tensor(st["radar"])
    elif kind == "batch":
        st["radar"] = _radar(c)
        st["px"] = [_upload(_typed(_walk_pixels(c["grid"], f, seed), "f32")) for f in range(c["frames"])]
        st["cubes"] = [device.cube_tensor(st["radar"]) for _ in st["px"]]
    elif kind == "doppler":
        st["radar"] = _radar(c)
        st["cubes"] = _cubes(c, seed)
        st["power"] = torch.empty((c["frames"], c["Ns"], c["L"]), dtype=torch.float32, device="cuda")
        st["v"] = torch.empty(c["frames"], dtype=torch.float32, device="cuda")
        st["peak"] = torch.empty((c["frames"], 2), dtype=torch.int32, device="cuda")
    elif kind == "raycast":
        st["scene"] = _abi.primitives_array(_scene(c, seed))
        dt = torch.float64 if c["px"] == "f64" else torch.float32
        st["out"] = {k: torch.empty(c["n_az"] * c["n_el"], dtype=dt, device="cuda") for k in FIELDS}
    else:
        st["server"] = _Server(st["ctx"])
        st["requests"] = []
        for i, q in enumerate(_mix(c)):
            radar = _radar(q)
            px = _upload(_typed(_scatter_pixels(q, seed * 1009 + i), "f32"))
            st["requests"].append((radar, px, _abi.TIERS[q["tier"]], device.cube_tensor(radar)))
    return st


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "frame" and c["host"]:
        ctx.synth_host(state["radar"], state["px"], c["tier"], cube=state["cube"])
        torch.cuda.current_stream().synchronize()  # the caller reads the cube on the host
        return state["cube"]
    if kind == "frame":
        return ctx.synth(state["radar"], state["px"], c["tier"], cube=state["cube"])
    if kind == "batch":
        return ctx.synth_batch(state["radar"], state["px"], c["tier"], cubes=state["cubes"])
    if kind == "doppler":
        _abi.rsim_range_doppler(ctx.h, state["radar"], state["cubes"], state["power"], state["v"], state["peak"])
        return {"power": state["power"], "v": state["v"], "peak": state["peak"]}
    if kind == "raycast":
        return ctx.raycast(state["scene"], c["n_az"], c["n_el"], (AZ, EL), out=state["out"])
    srv = state["server"].h
    tickets = [_abi.rsim_server_submit(srv, _abi.make_request(*r)) for r in state["requests"]]
    for t in tickets:
        _abi.check(_abi.rsim_server_wait(srv, t))
    return [r[3] for r in state["requests"]]


# ----------------------------------------------------------------------------------
# What a pass cannot do without
# ----------------------------------------------------------------------------------

def _cube_work(c, tier, valid):
    V, Ns, L = c["M"] * c["N"], c["Ns"], c["L"]
    if tier == "nufft":
        # 7 x 7 taps of a real weight times a complex strength, an FFT of the twice oversampled grid
        gx, gy = 1 << (2 * Ns - 1).bit_length(), 1 << (2 * L - 1).bit_length()
        return V * (valid * 49 * 4.0 + 5.0 * gx * gy * math.log2(gx * gy))
    return 8.0 * valid * V * Ns * L


def work(case):
    c, kind = case, case["kind"]
    if kind in ("frame", "batch"):
        V = c["M"] * c["N"]
        if kind == "frame":
            F, P, elem, valid = 1, c["n_az"] * c["n_el"], 8 if c["px"] == "f64" else 4, 1.0 - c["mask"]
        else:
            F, P, elem, valid = c["frames"], c["grid"] ** 2, 4, 33500.0 / 65536.0
        return {"bytes": F * (6.0 * elem * P + 8.0 * V * c["Ns"] * c["L"]), "flops": F * _cube_work(c, c["tier"], valid * P)}
    if kind == "doppler":
        n = c["Ns"] * c["L"]
        return {"bytes": c["frames"] * (8.0 * c["M"] * c["N"] * n + 4.0 * n),
                "flops": c["frames"] * c["M"] * c["N"] * (5.0 * n * math.log2(n) + 4.0 * n)}
    if kind == "raycast":
        P = c["n_az"] * c["n_el"]
        return {"bytes": 6.0 * (8 if c["px"] == "f64" else 4) * P + 160.0 * c["prims"], "flops": 50.0 * P * c["prims"]}
    b = f = 0.0
    for q in _mix(c):
        P = q["n_az"] * q["n_el"]
        b += 24.0 * P + 8.0 * q["M"] * q["N"] * q["Ns"] * q["L"]
        f += _cube_work(q, q["tier"], (1.0 - q["mask"]) * P)
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------------
# The same results in 64 bits
# ----------------------------------------------------------------------------------

def _cube64(c, px):
    """The sum over the valid pixels: fast-time and slow-time phasors, one matrix product per channel."""
    rr, sre, sim, az, el, vel = (torch.from_numpy(np.asarray(a, dtype=np.float64)).cuda() for a in px)
    ok = (sre != 0) | (sim != 0)
    rr, sre, sim, az, el, vel = (a[ok] for a in (rr, sre, sim, az, el, vel))
    V, Ns, L, d, ts = c["M"] * c["N"], c["Ns"], c["L"], LAM / 2.0, c["M"] * T_B
    u = torch.cos(el) * torch.sin(az)
    n = torch.arange(Ns, device="cuda", dtype=torch.float64)
    l = torch.arange(L, device="cuda", dtype=torch.float64)

    def cis(cycles):
        x = 2.0 * math.pi * (cycles - torch.round(cycles))
        return torch.complex(torch.cos(x), torch.sin(x))

    out = torch.zeros((V, Ns, L), dtype=torch.complex128, device="cuda")
    for s in range(0, rr.numel(), 65536):
        q = slice(s, s + 65536)
        D = torch.complex(sre[q], sim[q])[:, None] * cis(-2.0 * vel[q, None] / LAM * ts * l[None, :])
        for v in range(V):
            a = 2.0 * MU * (rr[q] + 0.5 * v * d * u[q]) / (C_LIGHT * FS)
            out[v] += cis(a[:, None] * n[None, :] + (v * d / LAM * u[q])[:, None]).T @ D
    return out


def _render64(c, seed):
    """First hits, Lambert strength over the squared range and closing speed, in 64 bits."""
    dev = "cuda"
    az, el = (torch.from_numpy(a).to(dev) for a in _angles(c["n_az"], c["n_el"]))
    d = torch.stack([torch.cos(el) * torch.sin(az), torch.cos(el) * torch.cos(az), torch.sin(el)], 1)
    inf = torch.full_like(az, math.inf)

    def sphere(f, u, rr):
        """Both roots of |f + t u|^2 = rr, u a unit vector; inf for a miss."""
        b = (f * u).sum(1)
        g = f - b[:, None] * u
        disc = rr - (g * g).sum(1)
        root = torch.sqrt(disc.clamp(min=0))
        return torch.where(disc >= 0, -b - root, inf), torch.where(disc >= 0, -b + root, inf)

    def first(*ts):
        best = inf
        for t in ts:
            best = torch.where((t > 0) & (t < best), t, best)
        return best

    best, s_out, w_out = inf.clone(), torch.zeros_like(az), torch.zeros_like(az)
    for p in _scene(c, seed):
        a, b, e, g, vel, om = (torch.as_tensor(p[k], dtype=torch.float64, device=dev) for k in ("a", "b", "c", "d", "vel", "omega"))
        if p["kind"] == "plane":
            nrm = torch.linalg.cross(b, e)
            t = (a @ nrm) / (d @ nrm)
            x = t[:, None] * d - a
            s, u = x @ torch.linalg.cross(e, nrm) / (nrm @ nrm), x @ torch.linalg.cross(nrm, b) / (nrm @ nrm)
            t = torch.where((t > 0) & (s >= 0) & (s <= 1) & (u >= 0) & (u <= 1), t, inf)
            normal = nrm.expand_as(d)
        elif p["kind"] == "capsule":
            ax, r = b - a, float(e[0])
            h2 = ax @ ax
            dp = d - (d @ ax / h2)[:, None] * ax
            lp = dp.norm(dim=1)
            off = -a + (a @ ax) / h2 * ax
            t1, t2 = sphere(off.expand_as(d), dp / lp[:, None], r * r)
            side = []
            for tt in (t1 / lp, t2 / lp):
                foot = (tt * (d @ ax) - a @ ax) / h2
                side.append(torch.where((foot >= 0) & (foot <= 1), tt, inf))
            t = first(*side, *sphere((-a).expand_as(d), d, r * r), *sphere((-b).expand_as(d), d, r * r))
            x = torch.where(torch.isfinite(t), t, torch.zeros_like(t))[:, None] * d - a
            normal = x - ((x @ ax) / h2).clamp(0, 1)[:, None] * ax
        else:
            W = torch.stack([b / (b @ b), e / (e @ e), g / (g @ g)], 1)
            sd = d @ W
            ls = sd.norm(dim=1)
            t1, t2 = sphere((-a @ W).expand_as(d), sd / ls[:, None], 1.0)
            t = first(t1 / ls, t2 / ls)
            x = torch.where(torch.isfinite(t), t, torch.zeros_like(t))[:, None] * d - a
            normal = (x @ W) @ W.T
        near = t < best
        tt = torch.where(near, t, torch.ones_like(t))
        x = tt[:, None] * d - a
        cos_i = (normal * d).sum(1).abs() / normal.norm(dim=1)
        speed = -((vel + torch.linalg.cross(om.expand_as(x), x)) * d).sum(1)
        best = torch.where(near, t, best)
        s_out = torch.where(near, p["rho"] * cos_i / tt ** 2, s_out)
        w_out = torch.where(near, speed, w_out)
    return {"range": best, "sigma_re": s_out, "sigma_im": torch.zeros_like(az), "az": az, "el": el, "vel": w_out}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "frame":
        return _cube64(c, _typed(_scatter_pixels(c, seed), c["px"]))
    if kind == "batch":
        return [_cube64(c, _typed(_walk_pixels(c["grid"], f, seed), "f32")) for f in range(c["frames"])]
    if kind == "doppler":
        power = torch.stack([(torch.fft.fft2(x.to(torch.complex128)).abs() ** 2).sum(0) for x in _cubes(c, seed)])
        L = c["L"]
        bins = power.flatten(1).argmax(1) % L
        signed = torch.where(bins < L // 2, bins, bins - L).to(torch.float64)
        return {"power": power, "v": -signed * LAM / (2.0 * c["M"] * T_B * L), "peak": None}
    if kind == "raycast":
        return _render64(c, seed)
    return [_cube64(q, _typed(_scatter_pixels(q, seed * 1009 + i), "f32")) for i, q in enumerate(_mix(c))]
