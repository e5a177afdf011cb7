"""The work that users of this framework have it do, as cases that can be timed.

A case names an entry point (its "kind"), the sizes of the call and the
storage types.  prepare() makes what a program has in hand before the call
(stars, cube map, tables, cameras, output buffers), run() is one call, work()
the bytes and operations it cannot do without, and exact() the same outputs
in 64 bits, written here in plain torch and numpy from the method's
definitions.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2010_08735_gb300 import bh, synth

DEV = "cuda"
MU = 4.0 / 27.0
EXPOSURE_DISC, EXPOSURE_STARS = 1.0, 0.01
# rows e_w, e_h, e_d of a camera that looks at the hole, +z up
LOOK_AT_HOLE = (0.0, 0.0, 1.0, 0.0, -1.0, 0.0, 1.0, 0.0, 0.0)


def _frame(name, kind="frame", width=1920, height=1080, r=6.0, theta=85.0, vr=0.0, vphi=0.5, r_out=12.0,
           stars=1_000_000, face=2048, cube="f16", tables="f32", particles=0, d_n=512, **more):
    return dict(name=name, kind=kind, width=width, height=height, r=r, theta=theta, vr=vr, vphi=vphi, r_out=r_out,
                stars=stars, face=face, cube=cube, tables=tables, particles=particles, d_n=d_n, **more)


def listed():
    return [
        # the smallest frame in use: a thumbnail of a static view, a few stars (latency and launch count)
        _frame("frame_256", width=256, height=256, r=10.0, theta=80.0, vphi=0.0, stars=1000),
        # the headline: one frame at a time, camera on an orbit at 0.5 c, a million stars
        _frame("frame_1080p"),
        # the largest single frame: 4K, camera falling at 0.9 c, four million stars in BF16
        _frame("frame_4k", width=3840, height=2160, r=3.2, theta=89.0, vr=-0.9, vphi=0.0, r_out=20.0,
               stars=4_000_000, face=4096, cube="bf16"),
        # the animated disc at an odd window size, with the compact (FP16) tables
        _frame("frame_animated", width=1365, height=767, r=8.0, theta=80.0, vphi=0.3, stars=200_000, cube="bf16",
               tables="f16", particles=16),
        # many cameras of mixed size rendered by one call (dataset or wall of views)
        _frame("batch_64", kind="batch", n=64, width=1920, height=1080),
        # cameras in free fall that live on the device: advance a frame's time, then render them all
        _frame("orbits_16", kind="orbits", n=16, width=1280, height=720),
        # a server's round: sixteen viewers ask for a frame each and wait for theirs
        _frame("served_16", kind="served", n=16),
        # a video writer: packed RGB frames into pinned host memory, two in flight
        _frame("host_1080p", kind="host"),
        # lens glare of a rendered frame
        dict(name="bloom_1080p", kind="bloom", width=1920, height=1080, levels=6),
        # new tables while serving: precompute, the first frame with them, and the old ones given back
        _frame("tables_512", kind="tables", width=1280, height=720, r=10.0, theta=80.0, vphi=0.0, stars=20_000,
               face=1024, particles=16),
        # a new star field: build its cube map and render the first frame
        _frame("cube_1m", kind="cube"),
        # a small star field built into the caller's own memory (plug-in hosts)
        dict(name="records_128", kind="records", stars=20_000, face=128, cube="f16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: sizes over their logarithm, odd ones among them."""
    kind = rng.choice(["frame", "frame", "frame", "batch", "orbits", "served", "host", "bloom", "tables", "cube",
                       "records"])
    width = _log_int(rng, 64, 3840)
    height = max(1, min(2160, int(width * rng.uniform(0.4, 1.2))))
    if kind == "bloom":
        return dict(kind=kind, width=min(width, 1920), height=min(height, 1080), levels=rng.randint(2, 8))
    if kind == "records":
        return dict(kind=kind, stars=_log_int(rng, 10, 20_000), face=2 ** rng.randint(3, 7),
                    cube=rng.choice(["f16", "bf16"]))
    infall = rng.random() < 0.3
    c = _frame("", kind=kind, width=width, height=height, r=round(math.exp(rng.uniform(math.log(2.5), math.log(30))), 3),
               theta=round(rng.uniform(60, 90), 2), vr=-round(rng.uniform(0.1, 0.9), 3) if infall else 0.0,
               vphi=0.0 if infall else round(rng.uniform(0.0, 0.8), 3), r_out=rng.choice([12.0, 20.0]),
               stars=_log_int(rng, 1000, 1_000_000), face=2 ** rng.randint(9, 11), cube=rng.choice(["f16", "bf16"]),
               tables=rng.choice(["f32", "f32", "f16"]), particles=rng.choice([0, 0, 16, 48]))
    del c["name"]
    if kind in ("batch", "orbits", "served"):
        c["n"] = _log_int(rng, 2, 48 if kind == "batch" else 16)
        c["width"], c["height"] = min(width, 1920), min(height, 1080)
        c["particles"] = 0
    if kind in ("host", "tables", "cube"):
        c["width"], c["height"] = min(width, 1920), min(height, 1080)
    if kind == "tables":
        c["d_n"] = 2 * rng.randint(64, 256)
        c["stars"], c["face"] = min(c["stars"], 20_000), 1024
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _stars(n, seed):
    """(n, 5) float32 on the device: directions uniform on the sphere, luminosity
    density ~ L^-1.5 on [1, 1e4], temperature log-uniform on [3000, 30000] K."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    d = torch.randn((n, 3), dtype=torch.float64, device=DEV, generator=g)
    u = torch.rand((n, 2), dtype=torch.float64, device=DEV, generator=g)
    out = torch.empty((n, 5), dtype=torch.float32, device=DEV)
    out[:, :3] = d / d.norm(dim=1, keepdim=True)
    out[:, 3] = (1.0 - u[:, 0] * (1.0 - 1e-2)) ** -2.0
    out[:, 4] = 3000.0 * 10.0 ** u[:, 1]
    return out


def _camera(case, seed):
    """The case's camera somewhere along its orbit."""
    phi = random.Random(seed).uniform(0.0, 360.0)
    return synth.camera(case["r"], case["theta"], phi, (case["vr"], 0.0, case["vphi"]), case["width"], case["height"])


def _cameras(case, seed):
    """Cameras of a batch: the sizes cycle through fractions of the case's (mixed
    windows), positions, speeds and orientations are random."""
    cams = synth.batch_cameras(case["n"], seed)
    for k, c in enumerate(cams):
        c["width"], c["height"] = _mixed_size(case, k)
    return cams


def _mixed_size(case, k):
    num, den = ((1, 6), (1, 3), (2, 3), (1, 1))[k % 4]
    return max(1, case["width"] * num // den), max(1, case["height"] * num // den)


def _orbits(case, seed):
    """Near-circular free-fall orbits (they stay in range however long they run)."""
    rng = random.Random(seed)
    out = []
    for k in range(case["n"]):
        w, h = _mixed_size(case, k)
        r0 = rng.uniform(6.0, 30.0)
        v0 = math.sqrt(1.0 / (2.0 * (r0 - 1.0))) * rng.uniform(0.97, 1.03)
        out.append(bh.bh_orbit_init(r0, math.pi / 2, v0, rng.uniform(-0.5, 0.5), LOOK_AT_HOLE, math.pi / 3, w, h))
    return out


ORBIT_DTAU, ORBIT_STEPS = 0.05, 8


def _hdr_image(case, seed):
    """A frame as the renderer gives it: smooth glow, dark sky, a few very bright stars."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    h, w = case["height"], case["width"]
    img = torch.rand((h, w, 4), device=DEV, generator=g) * 0.05
    img += torch.rand((1, 1, 4), device=DEV, generator=g) * torch.linspace(0, 1, w, device=DEV)[None, :, None]
    lit = torch.rand((h, w, 1), device=DEV, generator=g)  # one pixel in a hundred, L^-1.5 on [1, 1e4]
    img += torch.where(lit < 0.01, (lit * 99.0 + 0.01) ** -2.0, torch.zeros_like(lit))
    img[..., 3] = 1.0
    return img


def _dtype(case, key):
    return {"f32": bh.BH_F32, "f16": bh.BH_F16, "bf16": bh.BH_BF16}[case[key]]


class _State(dict):
    """What the program keeps; gives its handles back when it is dropped."""

    def __del__(self):
        if "ctx" not in self:
            return
        for key, free in (("cube", bh.bh_cubemap_free), ("tables", bh.bh_tables_free),
                          ("particles", bh.bh_disc_particles_free), ("ctx", bh.bh_destroy)):
            if self.get(key):
                free(self.pop(key))


def prepare(case, seed):
    s = _State(kind=case["kind"], case=case, stream=torch.cuda.current_stream())
    kind = case["kind"]
    if kind == "records":
        s["stars"] = _stars(case["stars"], seed)
        s["records"] = torch.empty((bh.bh_cubemap_records(case["face"]), 4), dtype=torch.int16, device=DEV)
        s["dtype"] = _dtype(case, "cube")
        return s
    s["ctx"] = ctx = bh.bh_create(torch.cuda.current_device(), 0)
    if kind == "bloom":
        s["in"] = _hdr_image(case, seed)
        s["out"] = torch.empty_like(s["in"])
        s["weights"] = bh.bh_bloom_weights(math.pi / 3, case["height"], case["levels"])
        return s
    s["shading"] = bh.make_shading(EXPOSURE_DISC, EXPOSURE_STARS)
    disc = synth.disc(3.0, case["r_out"])
    if case["particles"]:
        s["particles"] = bh.bh_disc_particles_create(ctx, _particles(case, seed))
        disc.update(particles_handle=s["particles"], time=_disc_time(seed))
    s["disc"] = bh.make_disc(disc)
    s["stars"] = _stars(case["stars"], seed)
    if kind != "cube":
        s["cube"] = bh.bh_build_star_cubemap(ctx, s["stars"], case["face"], _dtype(case, "cube"))
    if kind != "tables":
        s["tables"] = bh.bh_precompute_tables(ctx, case["d_n"], 64, 32, _dtype(case, "tables"))

    def frame(w, h, ch=4, **kw):
        return torch.zeros((h, w, ch), dtype=torch.float32, **kw)

    if kind == "batch":
        cams = _cameras(case, seed)
        s["cameras"] = [bh.make_camera(c) for c in cams]
        s["outs"] = [frame(c["width"], c["height"], device=DEV) for c in cams]
    elif kind == "orbits":
        orbits = _orbits(case, seed)
        s["orbits"] = torch.frombuffer(bytearray(bh.orbits_to_bytes(orbits)), dtype=torch.uint8).to(DEV)
        s["outs"] = [frame(o.width, o.height, device=DEV) for o in orbits]
    elif kind == "served":
        cams = [_camera(case, seed * 131 + k) for k in range(case["n"])]
        s["cameras"] = [bh.make_camera(c) for c in cams]
        s["outs"] = [frame(c["width"], c["height"], device=DEV) for c in cams]
    elif kind == "host":
        s["camera"] = bh.make_camera(_camera(case, seed))
        s["hosts"] = [frame(case["width"], case["height"], 3, pin_memory=True) for _ in range(2)]
        s["count"], s["ticket"] = 0, None
    else:
        s["camera"] = bh.make_camera(_camera(case, seed))
        s["out"] = frame(case["width"], case["height"], device=DEV)
    torch.cuda.synchronize()
    return s


def _particles(case, seed):
    return synth.disc_particles(case["particles"], seed % 100_000, 3.0, case["r_out"])


def _disc_time(seed):
    return float(seed % 1000)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    kind, st = s["kind"], s["stream"]
    if kind == "records":
        bh.bh_build_star_cubemap_noalloc(s["stars"], s["case"]["face"], s["dtype"], s["records"], st)
        return s["records"]
    ctx = s["ctx"]
    if kind == "bloom":
        bh.bh_bloom(ctx, s["in"], s["out"], s["case"]["width"], s["case"]["height"], s["weights"], st)
        return s["out"]
    disc, shading = s["disc"], s["shading"]
    if kind == "frame":
        bh.bh_render(ctx, s["tables"], s["cube"], s["camera"], disc, shading, s["out"], st)
        return s["out"]
    if kind == "batch":
        bh.bh_render_batch(ctx, s["tables"], s["cube"], s["cameras"], disc, shading, s["outs"], st)
        return s["outs"]
    if kind == "orbits":
        n = s["case"]["n"]
        bh.bh_orbits_advance(ctx, s["orbits"], n, ORBIT_DTAU, ORBIT_STEPS, st)
        bh.bh_render_orbits(ctx, s["tables"], s["cube"], n, s["orbits"], disc, shading, s["outs"], st)
        return {"frames": s["outs"], "orbits": s["orbits"].view(torch.float64).view(n, -1)[:, :7]}
    if kind == "served":
        tickets = []
        for k, cam in enumerate(s["cameras"]):
            status, ticket = bh.bh_serve_submit(ctx, s["tables"], s["cube"], k, cam, disc, shading, s["outs"][k])
            if status != bh.BH_OK:
                raise RuntimeError("a viewer's frame was refused")
            tickets.append(ticket)
        for ticket in tickets:
            while bh.bh_serve_poll(ctx, ticket, 100_000)[0] != bh.BH_OK:
                pass
        return s["outs"]
    if kind == "host":
        host = s["hosts"][s["count"] % 2]
        s["count"] += 1
        ticket = bh.bh_render_to_host_async(ctx, s["tables"], s["cube"], s["camera"], disc, shading, host, True, st)
        if s["ticket"] is not None:  # the frame before this one goes to the writer
            bh.bh_host_wait(ctx, s["ticket"])
        s["ticket"] = ticket
        return host
    if kind == "tables":
        tables = bh.bh_precompute_tables(ctx, s["case"]["d_n"], 64, 32, _dtype(s["case"], "tables"), st)
        bh.bh_render(ctx, tables, s["cube"], s["camera"], disc, shading, s["out"], st)
        bh.bh_tables_free(tables)
        return s["out"]
    cube = bh.bh_build_star_cubemap(ctx, s["stars"], s["case"]["face"], _dtype(s["case"], "cube"), st)
    bh.bh_render(ctx, s["tables"], cube, s["camera"], disc, shading, s["out"], st)
    bh.bh_cubemap_free(cube)
    return s["out"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

# per pixel of a frame: arithmetic of the method and cube-map records first touched (1080p workload)
PIXEL_FLOPS, PIXEL_RECORDS = 473, 0.43


def work(case):
    kind = case["kind"]
    if kind == "records":
        return {"bytes": 20 * case["stars"] + 8 * _records(case["face"]), "flops": 200 * case["stars"]}
    px = case["width"] * case["height"]
    if kind == "bloom":
        return {"bytes": 32 * px, "flops": px * (3 + 6 * 3 * case["levels"] + 16 * 3)}
    if kind in ("batch", "orbits"):
        sizes = [_mixed_size(case, k) for k in range(case["n"])]
        px = sum(w * h for w, h in sizes)
    elif kind == "served":
        px *= case["n"]
    nbytes = px * (12 if kind == "host" else 16) + 8 * min(PIXEL_RECORDS * px, case["stars"])
    flops = px * PIXEL_FLOPS
    if kind == "cube":
        nbytes += 20 * case["stars"] + 8 * _records(case["face"])
        flops += 200 * case["stars"]
    if kind == "tables":
        texels = case["d_n"] ** 2 + 64 * 32
        nbytes += texels * 28 + 16 * 64 * 32 * 64
        flops += texels * 2 * 16 * 10 + 64 * 32 * 64 * 95 * 10
    return {"bytes": int(nbytes), "flops": int(flops)}


def _records(face):
    n = 0
    while face:
        n += 6 * face * face
        face >>= 1
    return n


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind == "records":
        return None
    if kind == "bloom":
        return _bloom64(_hdr_image(case, seed).double(), _bloom_weights64(math.pi / 3, case["height"], case["levels"]))
    scene = _scene64(case, seed)
    if kind == "batch":
        return [_render64(scene, c) for c in _cameras(case, seed)]
    if kind == "orbits":
        states = [_orbit_advance64(o, ORBIT_DTAU, ORBIT_STEPS) for o in _orbits(case, seed)]
        return {"frames": [_render64(scene, _orbit_camera64(o)) for o in states],
                "orbits": torch.tensor([[o[k] for k in ("t", "r", "psi", "rdot", "e", "l", "chi")] for o in states],
                                       dtype=torch.float64)}
    if kind == "served":
        return [_render64(scene, _camera(case, seed * 131 + k)) for k in range(case["n"])]
    img = _render64(scene, _camera(case, seed))
    return img[..., :3].cpu().contiguous() if kind == "host" else img


def _scene64(case, seed):
    """Tables and cube map in 64 bits, rounded to the storage types the case asks for."""
    D, U, DT, UT = _tables64(case["d_n"], 64, 32)
    if case["tables"] == "f16":
        D, U = (torch.from_numpy(a.cpu().numpy().astype(np.float16).astype(np.float64)).to(DEV) for a in (D, U))
    else:
        D, U = D.float().double(), U.float().double()
    C, disc_table = _colour64()
    scene = dict(D=D, U=U, DT=DT.float().double(), UT=UT.float().double(), C=C, disc_table=disc_table,
                 cube=_cube64(_stars(case["stars"], seed), case["face"], case["cube"]), r_in=3.0, r_out=case["r_out"],
                 t_peak=1e4, rho=0.5, time=_disc_time(seed),
                 particles=_particles(case, seed) if case["particles"] else None)
    return scene


def _gl(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.tensor(x, device=DEV), torch.tensor(w, device=DEV)


def _integral(f, a, b, n=128):
    """Gauss-Legendre of f over [a, b], elementwise."""
    x, w = _gl(n)
    out = torch.empty_like(b)
    fa, fb, fo = a.reshape(-1), b.reshape(-1), out.reshape(-1)
    step = 1 << 17
    for k in range(0, fo.numel(), step):
        sl = slice(k, k + step)
        m, h = 0.5 * (fa[sl] + fb[sl]), 0.5 * (fb[sl] - fa[sl])
        fo[sl] = (f(m[:, None] + h[:, None] * x, sl) * w).sum(1) * h
    return out


class _Scatter:
    """Rays with e^2 < mu: u = u_a - w^2, (du/dphi)^2 = w^2 q(w), w = c sinh t."""

    def __init__(self, eta, e):
        s = torch.asin(torch.sqrt(eta))
        th = (0.5 * math.pi - 2.0 * s) / 3.0
        self.e, self.ua = e, 1.0 / 3.0 + 2.0 / 3.0 * torch.sin(th)
        self.A = 4.0 * self.ua * torch.cos(math.pi / 12.0 + 0.5 * th) * torch.sin(s / 3.0)
        self.B = 2.0 * torch.sin(th)
        self.c = torch.where(self.ua > 0.6, torch.sqrt(self.A / self.B.clamp_min(0.5)), torch.ones_like(self.A))

    def q(self, w):
        return self.A + self.B * w * w - w ** 4

    def integral(self, w0, time):
        """Angle (or regularised time) from infinity to u_a - w0^2."""
        A, B, c, e = (torch.broadcast_to(v, w0.shape).reshape(-1) for v in (self.A, self.B, self.c, self.e))

        def f(t, sl):
            w = c[sl, None] * torch.sinh(t)
            q = A[sl, None] + B[sl, None] * w * w - w ** 4
            g = 2.0 * c[sl, None] * torch.cosh(t) / torch.sqrt(q)
            return g / (e[sl, None] + w * torch.sqrt(q)) if time else g

        return _integral(f, torch.asinh(w0 / self.c), torch.broadcast_to(torch.asinh(torch.sqrt(self.ua) / self.c),
                                                                        w0.shape))


def _plunge(se, e, ta, tb, time):
    """Rays with e^2 > mu: u = 2/3 + v, v = se sinh t."""
    fse, fe = (torch.broadcast_to(v, tb.shape).reshape(-1) for v in (se, e))

    def f(t, sl):
        g = torch.sqrt(1.0 + fse[sl, None] * torch.sinh(t) * torch.tanh(t) ** 2)
        return 1.0 / (g * (fe[sl, None] + fse[sl, None] * torch.cosh(t) * g)) if time else 1.0 / g

    return _integral(f, torch.broadcast_to(ta, tb.shape), tb)


def _tables64(n, ne, nphi):
    f64 = dict(dtype=torch.float64, device=DEV)
    x = torch.arange(n, **f64) / (n - 1)
    y = (torch.arange(n, **f64) / (n - 1))[:, None]
    D, DT = torch.empty((n, n), **f64), torch.empty((n, n), **f64)
    a = 0.5 - x[None, : n // 2]
    sc = _Scatter(torch.exp(-50.0 * a * a), torch.sqrt(-MU * torch.expm1(-50.0 * a * a)))
    w0 = torch.sqrt(sc.ua) * (1.0 - y)
    D[:, : n // 2] = sc.integral(w0, False) - torch.atan2(sc.ua - w0 * w0, w0 * torch.sqrt(sc.q(w0)))
    DT[:, : n // 2] = sc.integral(w0, True)
    a = x[None, n // 2:] - 0.5
    e2 = MU / -torch.expm1(-50.0 * a * a)
    em = e2 * torch.exp(-50.0 * a * a)
    z = y * (math.sqrt(2.0 / 3.0) + math.sqrt(1.0 / 3.0)) - math.sqrt(2.0 / 3.0)
    v = z * z.abs() + 0.0 * em
    se = torch.sqrt(em)
    ta, tb = torch.asinh(-2.0 / 3.0 / se), torch.asinh(v / se)
    D[:, n // 2:] = _plunge(se, torch.sqrt(e2), ta, tb, False) - torch.atan2(2.0 / 3.0 + v,
                                                                          torch.sqrt(em + v * v * (v + 1.0)))
    DT[:, n // 2:] = _plunge(se, torch.sqrt(e2), ta, tb, True)

    # U(e, phi): phi(u) inverted by bisection
    xi = torch.arange(ne, **f64) / (ne - 1)
    e2 = (1.0 / xi.clamp_min(1e-9) - 1.0) / 6.0
    phi = 3.0 * (torch.arange(nphi, **f64) / (nphi - 1))[:, None] * (1.0 + e2) / (1.0 + 6.0 * e2 ** 1.5)
    U, UT = torch.zeros((nphi, ne), **f64), torch.zeros((nphi, ne), **f64)
    low = (e2 < MU) & (e2 > 0) & (xi > 0)
    if low.any():
        e2l, ph = e2[low], phi[:, low]
        sc = _Scatter(1.0 - e2l / MU, torch.sqrt(e2l))
        phia = sc.integral(torch.zeros_like(ph), False)
        past = ph > phia
        tgt = torch.where(past, 2.0 * phia - ph, ph)
        lo, hi = torch.zeros_like(ph), torch.sqrt(sc.ua) + 0.0 * ph
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            right = sc.integral(mid, False) > tgt
            lo, hi = torch.where(right, mid, lo), torch.where(right, hi, mid)
        w = 0.5 * (lo + hi)
        u = sc.ua - w * w
        R = sc.integral(w, True)
        Ra = sc.integral(torch.zeros_like(ph), True)
        ok = u > 0
        us = torch.where(ok, u, torch.full_like(u, 0.5))
        refl = (2.0 * Ra - 2.0 / sc.ua + 2.0 * torch.log(sc.ua / (1.0 - sc.ua)) - R + 2.0 / us
                - 2.0 * torch.log(us / (1.0 - us)))
        R = torch.where(past, torch.where(ok, refl, torch.zeros_like(R)), R)
        zero = ph <= 0
        U[:, low], UT[:, low] = torch.where(zero, 0 * u, u), torch.where(zero, 0 * u, R)
    high = (e2 >= MU) & (xi > 0)
    if high.any():
        e2h, ph = e2[high], phi[:, high]
        se, e = torch.sqrt(e2h - MU), torch.sqrt(e2h)
        ta, tb = torch.asinh(-2.0 / 3.0 / se) + 0.0 * ph, torch.asinh(1.0 / 3.0 / se) + 0.0 * ph
        gone = ph >= _plunge(se, e, ta, tb, False)
        lo, hi = ta, tb
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            left = _plunge(se, e, ta, mid, False) < ph
            lo, hi = torch.where(left, mid, lo), torch.where(left, hi, mid)
        t = 0.5 * (lo + hi)
        u, R = 2.0 / 3.0 + se * torch.sinh(t), _plunge(se, e, ta, t, True)
        zero = ph <= 0
        U[:, high] = torch.where(gone, torch.ones_like(u), torch.where(zero, 0 * u, u))
        UT[:, high] = torch.where(gone | zero, 0 * R, R)
    U[1:, xi == 0] = 1.0
    return D, U, DT, UT


# --- colour (5 nm trapezoid, 360 to 830 nm)

def _observer():
    lam = torch.arange(360.0, 831.0, 5.0, dtype=torch.float64, device=DEV)

    def lobe(m, s1, s2):
        return torch.exp(-0.5 * ((lam - m) / torch.where(lam < m, torch.full_like(lam, s1), torch.full_like(lam, s2))) ** 2)

    cmf = torch.stack([1.056 * lobe(599.8, 37.9, 31.0) + 0.362 * lobe(442.0, 16.0, 26.7) - 0.065 * lobe(501.1, 20.4, 26.2),
                       0.821 * lobe(568.8, 46.9, 40.5) + 0.286 * lobe(530.9, 16.3, 31.1),
                       1.217 * lobe(437.0, 11.8, 36.0) + 0.681 * lobe(459.0, 26.0, 13.8)], 1)
    w = torch.full_like(lam, 5.0)
    w[0] = w[-1] = 2.5
    return lam, cmf * w[:, None]


def _blackbody(T):
    lam, cmf = _observer()
    out = []
    for t in T.reshape(-1).split(1 << 18):
        out.append((1.0 / (lam ** 5 * torch.expm1(1.4387769e7 / (lam * t[:, None])))) @ cmf)
    return torch.cat(out).reshape(T.shape + (3,))


def _colour64():
    f64 = dict(dtype=torch.float64, device=DEV)

    def uv(x, y, z):
        d = x + 15.0 * y + 3.0 * z
        return 4.0 * x / d, 6.0 * y / d

    locus = 1000.0 * 40.0 ** (torch.arange(4096, **f64) / 4095.0)
    lu, lv = uv(*_blackbody(locus).unbind(1))
    x = 0.15 + 0.60 * (torch.arange(64, **f64) + 0.5) / 64
    y = (0.15 + 0.35 * (torch.arange(32, **f64) + 0.5) / 32)[:, None]
    cu, cv = uv(x / y, torch.ones_like(x / y), (1.0 - x - y) / y)
    T = locus[((cu[..., None] - lu) ** 2 + (cv[..., None] - lv) ** 2).argmin(2)]
    Dop = 2.0 ** (-4.0 + 8.0 * (torch.arange(64, **f64) + 0.5) / 64)
    C = _blackbody(Dop[:, None, None] * T) / _blackbody(T).sum(2)[None, :, :, None]
    bb = _blackbody(2.0 ** (8.0 + 12.0 * (torch.arange(1024, **f64) + 0.5) / 1024))
    table = torch.stack([torch.log(bb[:, 1]), bb[:, 0] / bb[:, 1], bb[:, 2] / bb[:, 1]], 1)
    return C.float().double(), table.float().double()


def _srgb():
    px, py = np.array([0.64, 0.30, 0.15]), np.array([0.33, 0.60, 0.06])
    P = np.stack([px / py, np.ones(3), (1.0 - px - py) / py])
    W = np.array([0.3127 / 0.3290, 1.0, (1.0 - 0.3127 - 0.3290) / 0.3290])
    inv = np.linalg.inv(P)
    return inv / (inv @ W)[:, None]


# --- star cube map: colour sums and mean positions per texel, all levels

def _round_to(v, dtype):
    """v to the nearest half (at most 65504) or bfloat16 value, ties to even."""
    bits, least = (11, -13) if dtype == "f16" else (8, -125)
    _, e = torch.frexp(v)
    ulp = torch.ldexp(torch.ones_like(v), e.clamp_min(least) - bits)
    v = torch.round(v / ulp) * ulp
    return v.clamp_max(65504.0) if dtype == "f16" else v


def _face_coords(d):
    """GL cube face, its coordinates and the major axis, of directions (n, 3)."""
    x, y, z = d.unbind(-1)
    ax, ay, az = x.abs(), y.abs(), z.abs()
    isx, isy = (ax >= ay) & (ax >= az), ay >= az
    face = torch.where(isx, torch.where(x >= 0, 0, 1), torch.where(isy, torch.where(y >= 0, 2, 3), torch.where(z >= 0, 4, 5)))
    return face


def _face_axes(face, d):
    """(sc, tc, ma) of vectors d on the given faces (linear in d)."""
    x, y, z = d.unbind(-1)
    pick = lambda *v: torch.stack(v, -1).gather(-1, face[..., None])[..., 0]  # noqa: E731
    return pick(-z, z, x, x, x, -x), pick(-y, -y, z, -z, -y, -y), pick(x, -x, y, -y, z, -z)


def _cube64(stars, N, dtype):
    d = stars[:, :3].double()
    bb = _blackbody(stars[:, 4].double())
    xyz = (stars[:, 3:4].double() * bb / ((bb[:, 0] + bb[:, 1]) + bb[:, 2])[:, None]).float().double()
    q = torch.round(xyz * 2.0 ** 20).long()
    face = _face_coords(d)
    sc, tc, ma = _face_axes(face, d)
    S, T = ((sc / ma + 1.0) * 0.5) * N, ((tc / ma + 1.0) * 0.5) * N
    i, j = S.floor().clamp(0, N - 1), T.floor().clamp(0, N - 1)
    s16, t16 = (((a - b) * 65536.0).floor().clamp(0, 65535).long() for a, b in ((S, i), (T, j)))
    at = (face * N + j.long()) * N + i.long()
    nt = 6 * N * N
    sums = [torch.zeros(nt, dtype=torch.int64, device=DEV).index_add_(0, at, v) for v in q.unbind(1)]
    ps, pt = (torch.zeros(nt, dtype=torch.int64, device=DEV).index_add_(0, at, q[:, 1] * v) for v in (s16, t16))

    def byte(v, y):
        return torch.where(y > 0, (v * 256.0).floor().clamp_max(255.0), torch.full_like(v, 128.0))

    y = sums[1].double()
    ys = y.clamp_min(1.0)
    ps, pt = (byte((v.double() / ys + 0.5) / 65536.0, sums[1]) for v in (ps, pt))
    levels, n, L = [], N, 0
    while True:
        scale = 2.0 ** (20 + 2 * L)
        levels.append(torch.stack([_round_to(v.double() / scale, dtype).float() for v in sums] + [ps.float(), pt.float()], 1))
        if n == 1:
            return dict(levels=levels, N=N)
        quad = lambda v: v.view(6, n // 2, 2, n // 2, 2)  # noqa: E731
        y, p, t = quad(sums[1]).double(), quad(ps), quad(pt)
        off = torch.arange(2.0, dtype=torch.float64, device=DEV)
        ns = (y * ((off + (p + 0.5) / 256.0) * 0.5)).sum((2, 4)).reshape(-1)
        nn = (y * ((off[:, None, None] + (t + 0.5) / 256.0) * 0.5)).sum((2, 4)).reshape(-1)
        sums = [quad(v).sum((2, 4)).reshape(-1) for v in sums]
        ys = sums[1].double().clamp_min(1.0)
        ps, pt = byte(ns / ys, sums[1]), byte(nn / ys, sums[1])
        n, L = n // 2, L + 1


# --- the pixels

def _bilinear(t, fx, fy, xlo, xhi):
    """Table t[j, i] at texel coordinates, x clamped to [xlo, xhi]."""
    fx = torch.minimum(torch.maximum(fx.nan_to_num(), xlo.double()), xhi.double())
    fy = fy.nan_to_num().clamp(0, t.shape[0] - 1)
    i0, j0 = fx.long(), fy.long()
    i1, j1 = torch.minimum(i0 + 1, xhi), (j0 + 1).clamp_max(t.shape[0] - 1)
    tx, ty = fx - i0, fy - j0
    lo = t[j0, i0] + tx * (t[j0, i1] - t[j0, i0])
    hi = t[j1, i0] + tx * (t[j1, i1] - t[j1, i0])
    return lo + ty * (hi - lo)


def _render64(scene, cam):
    W, H = cam["width"], cam["height"]
    out = torch.empty((H, W, 4), dtype=torch.float64, device=DEV)
    out[..., 3] = 1.0
    rows = max(2, (1 << 20) // (W + (W & 1)) // 2 * 2)
    M = torch.tensor(_srgb(), device=DEV)
    for y0 in range(0, H, rows):
        y1 = min(H, y0 + rows)
        xyz = _rows64(scene, cam, y0, y1 + ((y1 - y0) & 1))
        out[y0:y1, :, :3] = (xyz @ M.T)[: y1 - y0, :W]
    return out


def _rows64(scene, cam, ya, yb):
    f64 = dict(dtype=torch.float64, device=DEV)
    W, H = cam["width"], cam["height"]
    W2 = W + (W & 1)
    # camera frame: static basis, boost, orientation
    st, ct, sp, cp = math.sin(cam["theta"]), math.cos(cam["theta"]), math.sin(cam["phi"]), math.cos(cam["phi"])
    u = 1.0 / cam["r"]
    er, et, ep = (np.array(v) for v in ((st * cp, st * sp, ct), (ct * cp, ct * sp, -st), (-sp, cp, 0.0)))
    v = np.array(cam["v"], dtype=np.float64)
    beta = float(np.linalg.norm(v))
    gamma = 1.0 / math.sqrt(1.0 - beta * beta)
    vh = v / beta if beta > 0 else np.zeros(3)
    O = np.array(cam["orient"], dtype=np.float64).reshape(3, 3)
    R = np.stack([math.sqrt(1.0 - u) * er, et, ep], 1)
    f = 0.5 * H / math.tan(0.5 * cam["fov_y"])
    px = torch.arange(W2, **f64) + 0.5 - 0.5 * W
    py = 0.5 * H - (torch.arange(ya, yb, **f64) + 0.5)
    q = torch.stack(torch.broadcast_tensors(px[None, :], py[:, None], torch.tensor(-f, **f64)), -1)
    q = q / q.norm(dim=-1, keepdim=True)
    qs = q @ torch.tensor(O, **f64)  # on the boosted static axes
    vt = torch.tensor(vh, **f64)
    par = qs @ vt
    dpar = gamma * (par - beta)
    ds = (qs - par[..., None] * vt) + dpar[..., None] * vt
    dcam = gamma * (1.0 + beta * dpar / ds.norm(dim=-1))
    d = ds @ torch.tensor(R.T, **f64)
    x = torch.tensor(er, **f64)
    c = torch.linalg.cross(x.expand_as(d), d)
    cn = c.norm(dim=-1)
    cosd = d @ x
    delta = torch.atan2(cn, cosd)
    z = c / cn[..., None].clamp_min(1e-300)
    y = torch.linalg.cross(z, x.expand_as(z))
    t = torch.stack([-z[..., 1], z[..., 0], torch.zeros_like(cn)], -1)
    tn = t.norm(dim=-1)
    sign = torch.where((t * y).sum(-1) < 0, -1.0, 1.0)
    t = t * (sign / tn.clamp_min(1e-300))[..., None]
    alpha = torch.atan2((t * y).sum(-1), t @ x)

    # the ray's class and its deflection
    D, U = scene["D"], scene["U"]
    n = D.shape[0]
    udot = -u * cosd / cn.clamp_min(1e-300)
    em = udot ** 2 - (u - 2.0 / 3.0) ** 2 * (u + 1.0 / 3.0)
    e2 = MU + em
    low = em < 0
    dead = low & (u > 2.0 / 3.0)
    half = torch.full_like(em, 0, dtype=torch.long) + n // 2
    xlo, xhi = torch.where(low, 0, half), torch.where(low, half - 1, n - 1)
    lg = torch.where(low, torch.log((-em / MU).clamp_min(1e-300)), torch.log((em / e2).clamp_min(1e-300)))
    off = torch.sqrt((-lg).clamp_min(0.0) / 50.0)
    fx = torch.where(low, 0.5 - off, 0.5 + off) * (n - 1)
    eta = (-em / MU).clamp(0.0, 1.0)
    ua = 1.0 / 3.0 + 2.0 / 3.0 * torch.sin((0.5 * math.pi - 2.0 * torch.asin(torch.sqrt(eta))) / 3.0)
    g = ua + u - ua * ua - ua * u - u * u
    om = torch.where(g > 0, udot ** 2 / (ua * g), 1.0 - u / ua)
    root = math.copysign(math.sqrt(abs(u - 2.0 / 3.0)), u - 2.0 / 3.0)
    top = math.sqrt(2.0 / 3.0) + math.sqrt(1.0 / 3.0)
    yv = torch.where(low, 1.0 - torch.sqrt(om.clamp_min(0.0)), torch.full_like(om, (math.sqrt(2.0 / 3.0) + root) / top))
    Dl = _bilinear(D, fx, yv * (n - 1), xlo, xhi)
    last = torch.full_like(fx, n - 1.0)
    Da = torch.where(low, _bilinear(D, fx, last, xlo, xhi), 0.0 * fx)
    phia = torch.where(low, Da + 0.5 * math.pi, torch.full_like(Da, math.inf))
    out_ = udot > 0
    captured = dead | (out_ & ~low)
    turn = torch.where(out_, torch.where(low, 2.0 * Da - Dl, 0.0 * Dl), Dl)

    # disc crossings
    ne, nphi = U.shape[1], U.shape[0]
    uxf = (1.0 / (1.0 + 6.0 * e2)) * (ne - 1)
    yk = (1.0 + 6.0 * e2 ** 1.5) / (3.0 * (1.0 + e2)) * (nphi - 1)
    zero, wide = torch.zeros_like(half), torch.full_like(half, ne - 1)

    def at(tab, ph):
        return _bilinear(tab, uxf, ph * yk, zero, wide)

    def coord_time(Rt, uu):
        return Rt - 1.0 / uu + torch.log(uu / (1.0 - uu))

    s = torch.where(out_, 1.0, -1.0)
    phi = Dl + torch.where(out_, math.pi - (delta - alpha), delta - alpha)
    uic, uoc = 1.0 / scene["r_in"], 1.0 / scene["r_out"]
    valid = (tn > 1e-12) & ~dead
    hits = []
    ph2 = 2.0 * phia - phi
    for k, ph in enumerate((phi, torch.where(low & out_, ph2, torch.zeros_like(phi)))):
        turns = torch.floor(ph / math.pi)
        p0 = ph - math.pi * turns
        hu = at(U, p0)
        ok = valid & (p0 < phia) & (hu >= uoc) & (hu <= uic)
        ok = ok & (torch.where(out_, hu > u, hu < u) if k == 0 else low & out_)
        hits.append((ok, torch.where(ok, hu, torch.full_like(hu, 0.2)), p0, turns.long() & 1))
    y_peak = _disc_light(scene, torch.tensor(math.log2(scene["t_peak"]), **f64))[..., 1]
    L = torch.zeros(em.shape + (3,), **f64)
    trans = torch.ones_like(em)
    fmax = (12.0 / 49.0) ** 3 * (1.0 - math.sqrt(36.0 / 49.0))
    dpre = dcam / math.sqrt(1.0 - u)
    for k, (ok, hu, p0, odd) in enumerate(hits):
        rho = torch.full_like(hu, scene["rho"])
        if scene["particles"] is not None:
            tcam = coord_time(_bilinear(scene["DT"], fx, yv * (n - 1), xlo, xhi), torch.full_like(fx, u))
            th = coord_time(at(scene["UT"], p0), hu)
            if k == 0:
                delay = s * (th - tcam)
            else:
                delay = 2.0 * coord_time(_bilinear(scene["DT"], fx, last, xlo, xhi), ua) - tcam - th
            sg = torch.where(odd == 1, -1.0, 1.0)
            rho = _particle_density(scene, rho, delay, 1.0 / hu, torch.atan2(sg * t[..., 1], sg * t[..., 0]))
        dop = dpre * torch.sqrt(2.0 - 3.0 * hu) / (math.sqrt(2.0) + hu ** 1.5 * z[..., 2] / torch.sqrt(e2))
        fu = hu ** 3 * (1.0 - torch.sqrt(3.0 * hu))
        lgT = torch.log2(dop) + 0.25 * torch.log2((fu / fmax).clamp_min(1e-300)) + math.log2(scene["t_peak"])
        lit = ok & (fu > 0) & (lgT >= 8.0)
        light = _disc_light(scene, lgT) * (trans * rho * EXPOSURE_DISC / y_peak)[..., None]
        L = L + torch.where(lit[..., None], light, 0.0 * light)
        trans = torch.where(ok, trans * (1.0 - rho), trans)

    # escape direction, its derivatives within 2 x 2 quads, and the star light
    b = d / d.norm(dim=-1, keepdim=True)
    nrm = torch.linalg.cross(z, b)
    dp = torch.cos(turn)[..., None] * b + torch.sin(turn)[..., None] * nrm
    dp = torch.where(captured[..., None], 0.0 * dp, dp)
    h2 = em.shape[0]
    quad = captured.view(h2 // 2, 2, W2 // 2, 2)
    dark = quad.any(3, keepdim=True).any(1, keepdim=True).expand_as(quad).reshape(em.shape)

    def diffs(a):
        a = a.view(h2 // 2, 2, W2 // 2, 2, 3)
        w = (a - a.flip(3)).reshape(h2, W2, 3)
        h = (a - a.flip(1)).reshape(h2, W2, 3)
        return w, h

    dw, dh = diffs(dp)
    qw, qh = diffs(q)
    cd = torch.linalg.cross(dw, dh).norm(dim=-1)
    sky = ~dark & (cd > 0)
    omega = torch.linalg.cross(qw, qh).norm(dim=-1)[sky] / cd[sky]
    xyz = _sky64(scene, dp[sky], dw[sky], dh[sky])
    tot = xyz.sum(-1)
    has = tot > 0
    chroma = xyz / torch.where(has, tot, torch.ones_like(tot))[:, None]
    cc = _c_lookup(scene["C"], chroma[:, 0], chroma[:, 1], torch.log2(dpre[sky]))
    star = cc * (tot * omega * EXPOSURE_STARS * trans[sky])[:, None]
    L[sky] += torch.where(has[:, None], star, 0.0 * star)
    return L


def _disc_light(scene, lgT):
    tab = scene["disc_table"]
    f = ((lgT - 8.0) / 12.0 * 1024 - 0.5).nan_to_num().clamp(0, 1023)  # NaN where there is no crossing
    k0 = f.long()
    k1, t = (k0 + 1).clamp_max(1023), (f - k0)[..., None]
    v = tab[k0] + t * (tab[k1] - tab[k0])
    Y = torch.exp(v[..., :1])
    return torch.cat([Y * v[..., 1:2], Y, Y * v[..., 2:3]], -1)


def _particle_density(scene, rho, delay, hr, hphi):
    total = torch.zeros_like(hr)
    for u1, u2, phi0 in np.asarray(scene["particles"], dtype=np.float64):
        u3, ub = 1.0 - u1 - u2, 0.5 * (u1 + u2)
        a, b = 1.0, math.sqrt(1.0 - (u2 - u1) / (u3 - u1))  # K by the arithmetic-geometric mean
        for _ in range(40):
            a, b = 0.5 * (a + b), math.sqrt(a * b)
        K = math.pi / (2.0 * a)
        ph = math.sqrt(0.5 * ub ** 3) * (scene["time"] - delay) + phi0
        ang = torch.remainder(hphi - ph, 2.0 * math.pi)
        uu = u1 + (u2 - u1) * torch.sin(math.pi / (4.0 * K) * math.sqrt(u3 - u1) * (ang + ph)) ** 2
        d2 = (ang / math.pi - 1.0) ** 2 + (hr - 1.0 / uu) ** 2
        total = total + torch.where(d2 < 1.0, (1.0 - d2) ** 2, 0.0 * d2)
    return (rho * total).clamp_max(1.0)


def _sky64(scene, dp, dw, dh):
    """Star light gathered over each footprint: tent-weighted sum of the records."""
    cube = scene["cube"]
    N, top = cube["N"], len(cube["levels"]) - 1
    face = _face_coords(dp)
    sc, tc, ma = _face_axes(face, dp)
    sw, tw, mw = _face_axes(face, dw)
    sh, th, mh = _face_axes(face, dh)
    hN = 0.5 * N
    sr, tr = sc / ma, tc / ma
    S, T = (sr + 1.0) * hN, (tr + 1.0) * hN
    J = [hN / ma * v for v in (sw - sr * mw, sh - sr * mh, tw - tr * mw, th - tr * mh)]
    hs, ht = J[0].abs() + J[1].abs(), J[2].abs() + J[3].abs()
    level = torch.ceil(torch.log2((0.25 * torch.maximum(hs, ht)).clamp_min(1e-300))).clamp(0, top).long()
    out = torch.zeros((dp.shape[0], 3), dtype=torch.float64, device=DEV)
    for L in torch.unique(level).tolist():
        m = level == L
        NL, k = N >> L, 2.0 ** -L
        rec = cube["levels"][L]
        cS, cT, a, b_ = S[m] * k, T[m] * k, hs[m] * k, ht[m] * k
        a11, a12, a21, a22 = (v[m] * k for v in J)
        det = a11 * a22 - a12 * a21
        good = torch.isfinite(cS + cT + a + b_) & (det * det > 1e-12 * ((a11 * a11 + a21 * a21) * (a12 * a12 + a22 * a22)))
        inv = 1.0 / torch.where(good, det, torch.ones_like(det))
        i0, i1 = (cS - a).floor().clamp_min(0).long(), (cS + a).floor().clamp_max(NL - 1).long()
        j0, j1 = (cT - b_).floor().clamp_min(0).long(), (cT + b_).floor().clamp_max(NL - 1).long()
        base = face[m] * NL * NL
        acc = torch.zeros((cS.numel(), 3), dtype=torch.float64, device=DEV)
        if not cS.numel():
            continue
        for dj in range(max(0, int((j1 - j0).max()) + 1)):
            for di in range(max(0, int((i1 - i0).max()) + 1)):
                sel = (good & (j0 + dj <= j1) & (i0 + di <= i1)).nonzero()[:, 0]
                if not sel.numel():
                    continue
                i, j = i0[sel] + di, j0[sel] + dj
                r = rec[base[sel] + j * NL + i].double()
                lit = (r[:, 0] + r[:, 1] + r[:, 2]) > 0
                sel, i, j, r = sel[lit], i[lit], j[lit], r[lit]
                x = i + (r[:, 3] + 0.5) / 256.0 - cS[sel]
                y = j + (r[:, 4] + 0.5) / 256.0 - cT[sel]
                w = (a22[sel] * x - a12[sel] * y) * inv[sel]
                h = (a11[sel] * y - a21[sel] * x) * inv[sel]
                wt = (1.0 - w.abs()).clamp_min(0.0) * (1.0 - h.abs()).clamp_min(0.0)
                acc[sel] += wt[:, None] * r[:, :3]
        out[m] = acc * 4.0 ** L
    return out


def _c_lookup(C, x, y, lgD):
    f = [((x - 0.15) / 0.60 * 64 - 0.5).clamp(0, 63), ((y - 0.15) / 0.35 * 32 - 0.5).clamp(0, 31),
         ((lgD + 4.0) / 8.0 * 64 - 0.5).clamp(0, 63)]
    f = [v.nan_to_num() for v in f]
    lo = [v.long() for v in f]
    out = 0.0
    for k in range(8):
        w, at = 1.0, []
        for a, bit in zip((0, 1, 2), (k & 1, k >> 1 & 1, k >> 2 & 1)):
            frac = f[a] - lo[a]
            w = w * (frac if bit else 1.0 - frac)
            at.append((lo[a] + bit).clamp_max((63, 31, 63)[a]))
        out = out + w[:, None] * C[at[2], at[1], at[0]]
    return out


# --- free-fall orbits

def _orbit_advance64(o, dtau, steps):
    s = {k: getattr(o, k) for k in ("t", "r", "psi", "rdot", "e", "l", "chi", "fov_y", "width", "height")}
    s["orient"] = np.array(o.orient[:]).reshape(3, 3)
    h, l2 = dtau / steps, s["l"] ** 2

    def rhs(y):
        u = 1.0 / y[1]
        return np.array([s["e"] / (1.0 - u), y[3], s["l"] * u * u, 0.5 * (2.0 * l2 * u ** 3 - 3.0 * l2 * u ** 4 - u * u)])

    y = np.array([s["t"], s["r"], s["psi"], s["rdot"]])
    for _ in range(steps):
        k1 = rhs(y)
        k2 = rhs(y + 0.5 * h * k1)
        k3 = rhs(y + 0.5 * h * k2)
        k4 = rhs(y + h * k3)
        y = y + h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    s["t"], s["r"], s["psi"], s["rdot"] = (float(v) for v in y)
    return s


def _orbit_camera64(s):
    psi, chi, u = s["psi"], s["chi"], 1.0 / s["r"]
    th = math.acos(math.cos(psi) * math.sin(chi))
    ph = math.atan2(math.sin(psi), math.cos(chi) * math.cos(psi))
    a = math.sin(chi) * math.cos(th) * math.cos(ph) + math.cos(chi) * math.sin(th)
    b = -math.sin(chi) * math.sin(ph)
    vpsi = s["l"] * u * math.sqrt(1.0 - u) / s["e"]
    o = s["orient"]
    orient = np.stack([o[:, 0], a * o[:, 1] - b * o[:, 2], b * o[:, 1] + a * o[:, 2]], 1)
    return dict(r=s["r"], theta=th, phi=ph, v=(s["rdot"] / s["e"], -b * vpsi, a * vpsi), orient=orient,
                fov_y=s["fov_y"], width=s["width"], height=s["height"])


# --- bloom

def _bloom_weights64(fov_y, height, levels):
    """Share of the point spread function's energy in each octave of radius."""
    s = c = 0.02

    def energy(a, b):
        e0 = lambda t: -2.61e6 * math.pi * s * s * math.exp(-(t / s) ** 2)  # noqa: E731
        e1 = lambda t: 2 * math.pi * 20.91 * (-1 / (t + c) + c / (2 * (t + c) ** 2))  # noqa: E731
        e2 = lambda t: 2 * math.pi * 72.37 * (math.log(t + c) + c / (t + c))  # noqa: E731
        return 0.384 * (e0(b) - e0(a)) + 0.478 * (e1(b) - e1(a)) + 0.138 * (e2(b) - e2(a))

    a = math.degrees(fov_y) / height
    edge = [0.0] + [a * 2.0 ** (k + 0.5) for k in range(levels + 1)]
    total = energy(0.0, edge[-1])
    return [energy(edge[k], edge[k + 1]) / total for k in range(levels + 1)]


def _bloom64(img, weights):
    H, W, _ = img.shape
    out = weights[0] * img[..., :3]
    D = img[..., :3].permute(2, 0, 1)[None]
    taps = torch.exp(-0.5 * torch.arange(-3.0, 4.0, dtype=torch.float64, device=DEV) ** 2)
    taps = taps / taps.sum()
    for k in range(1, len(weights)):
        D = torch.nn.functional.pad(D, (0, D.shape[3] & 1, 0, D.shape[2] & 1), mode="replicate")
        D = 0.25 * (D[..., ::2, ::2] + D[..., ::2, 1::2] + D[..., 1::2, ::2] + D[..., 1::2, 1::2])
        h, w = D.shape[2:]
        ix = (torch.arange(w, device=DEV)[:, None] + torch.arange(-3, 4, device=DEV)).clamp(0, w - 1)
        iy = (torch.arange(h, device=DEV)[:, None] + torch.arange(-3, 4, device=DEV)).clamp(0, h - 1)
        B = (D[:, :, :, ix] * taps).sum(-1)
        B = (B[:, :, iy, :] * taps[:, None]).sum(3)[0].permute(1, 2, 0)

        def axis(n, m):
            u = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * 2.0 ** -k - 0.5
            f = u.floor()
            return f.long().clamp(0, m - 1), (f.long() + 1).clamp(0, m - 1), u - f

        x0, x1, tx = axis(W, w)
        y0, y1, ty = axis(H, h)
        rows = B[:, x0] + tx[None, :, None] * (B[:, x1] - B[:, x0])
        out = out + weights[k] * (rows[y0] + ty[:, None, None] * (rows[y1] - rows[y0]))
    return torch.cat([out, torch.ones_like(out[..., :1])], -1)
