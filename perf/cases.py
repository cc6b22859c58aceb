"""Performance cases of the ray tracer: what a user has it do, through its
public entry points, with the inputs drawn from a seed.

A case is a dict of plain values:
  call       "single"  one osr.trace / osr.render_disk call per pass
             "batch"   one osr.trace_batch call over `count` renders
             "plan"    one BatchPlan.launch over `count` renders (the plan is kept)
             "states"  one osr.trace_states call (explicit initial data)
  metric     "kerr" or "q"
  precision  "fp64", "df64" or "mixed";  integrator "ck45" or "dp45";  tol
  a / q      spin or quadrupole parameter;  incl  inclination in degrees
  scene      "sky", "disk" (Keplerian), "disk_l0" (constant l0), or "both"
             (sky and disk renders in turn, batches only)
  nx, ny     pixels of a render;  in a batch with side_max > 0 the sides are
             spread over [side_min, side_max] instead
  count      renders of a batch;  ranges  each entry is a pixel range of its
             render (a round of the render server)
  persistent a single call on a persistent grid (with a workspace)
  n, mass    particles of a "states" case

listed() holds the cases by name, draw() gives more of the same ranges,
prepare() makes a case's inputs from a seed, run() is one pass, work() counts
what a pass cannot do without, and exact() integrates the same rays with plain
torch in 64 bits.
"""
import math
import random

import numpy as np
import torch

import paper_2202_00086_gb300 as osr

PRECISION = {"fp64": osr.FP64, "df64": osr.DF64, "mixed": osr.MIXED}
INTEGRATOR = {"ck45": osr.RKCK45, "dp45": osr.RKDP45}
R_OBS = 1000.0


def _case(**kw):
    c = dict(call="single", metric="kerr", precision="fp64", integrator="ck45", tol=1e-10,
             a=0.9, q=0.0, incl=60.0, scene="sky", nx=0, ny=0, count=1, side_min=0, side_max=0,
             ranges=False, persistent=False, n=0, mass=0.0)
    c.update(kw)
    return c


def listed():
    return [
        # the first render of a new user: the 64 x 64 Schwarzschild shadow with every default
        # (the smallest call: it lasts as long as its slowest ray)
        _case(name="schwarzschild_64", a=0.0, incl=85.0, nx=64, ny=64),
        # an interactive preview while a camera is being set up, ragged size, in double-float
        _case(name="preview_df64", precision="df64", nx=161, ny=119),
        # one lensing image of a near-extremal hole with the defaults (FP64, plain launch)
        _case(name="kerr_render", a=0.998, nx=768, ny=768),
        # the shadow / Einstein-ring figure: 12 cameras in one replayed plan, FP64 (the
        # headline workload at a smaller side)
        _case(name="kerr_set_plan", call="plan", count=12, nx=320, ny=320),
        # the same figure in double-float, at a larger side
        _case(name="kerr_set_df64", call="plan", precision="df64", count=12, nx=512, ny=512),
        # the Keplerian disk figure in double-float
        _case(name="disk_df64", precision="df64", a=0.0, incl=80.0, scene="disk", nx=1024,
              ny=1024),
        # a panel of the constant-l0 disk figure with the integrator that the paper prefers
        _case(name="disk_l0_dp45", integrator="dp45", a=0.5, incl=85.0, scene="disk_l0", nx=640,
              ny=320),
        # a q-metric shadow in FP64, odd sizes, on a persistent grid
        _case(name="qmetric_fp64", metric="q", q=0.5, incl=90.0, nx=333, ny=257,
              persistent=True),
        # a q-metric image at the loose tolerance of the served stream
        _case(name="qmetric_mixed", metric="q", precision="mixed", tol=1e-8, q=0.1, incl=30.0,
              nx=1024, ny=1024),
        # a batch of uneven renders, sky and disk in turn (a parameter study), double-float
        _case(name="uneven_df64", call="batch", precision="df64", scene="both", count=16,
              side_min=128, side_max=1024),
        # one round of the render server for loose-tolerance renders: pixel ranges, MIXED
        _case(name="served_round_mixed", call="plan", precision="mixed", tol=1e-8, scene="both",
              count=10, side_min=256, side_max=1024, ranges=True),
        # unit-mass particles from explicit initial data, FP64
        _case(name="particles_fp64", call="states", mass=1.0, n=100003),
    ]


# Rays of the largest drawn case, so that none costs more than the largest listed one.
MAX_RAYS = {("kerr", "fp64"): 700_000, ("kerr", "df64"): 2_500_000, ("kerr", "mixed"): 8_000_000,
            ("q", "fp64"): 300_000, ("q", "df64"): 1_200_000, ("q", "mixed"): 6_000_000}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    precision = rng.choice(["fp64", "df64", "mixed"])
    metric = rng.choice(["kerr", "kerr", "kerr", "q"])
    c = _case(precision=precision, metric=metric,
              integrator=rng.choice(["ck45", "ck45", "dp45"]),
              tol=rng.choice([1e-8, 1e-7] if precision == "mixed" else [1e-10, 1e-10, 1e-9, 1e-8]),
              a=round(rng.uniform(0.0, 0.998), 4) if metric == "kerr" else 0.0,
              q=round(rng.uniform(-0.5, 0.5), 3) if metric == "q" else 0.0,
              incl=round(rng.uniform(5.0, 90.0), 2))
    top = MAX_RAYS[metric, precision]
    call = rng.choice(["single", "single", "batch", "plan", "states"])
    if call == "states" and metric == "kerr":
        c.update(call=call, mass=1.0, n=_log_int(rng, 1_000, min(top, 1_000_000)))
        return c
    scenes = ["sky"] if metric == "q" else ["sky", "disk", "disk_l0"]
    if call in ("batch", "plan"):
        count = _log_int(rng, 2, 32)
        side = math.sqrt(top / count)  # of the largest render
        lo = _log_int(rng, 32, max(33.0, side / 3))
        c.update(call=call, count=count, side_min=lo, side_max=_log_int(rng, lo + 1, max(lo + 2, side)),
                 scene=rng.choice(scenes if metric == "q" else scenes + ["both"]),
                 ranges=bool(call == "plan" and rng.random() < 0.5))
        return c
    rays = _log_int(rng, 2_000, top)
    aspect = math.exp(rng.uniform(-0.7, 0.7))
    nx = max(16, int(math.sqrt(rays * aspect)))
    c.update(scene=rng.choice(scenes), nx=nx, ny=max(16, rays // nx),
             persistent=bool(rng.random() < 0.4))
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _renders(case, seed):
    """The renders of a case: their sizes follow from the case alone, their
    cameras from the seed (small changes of spin, inclination and extent around
    the case's, or the 4 x 3 grid of the Kerr figure for its set)."""
    sizes, rng = random.Random("%s" % sorted(case.items())), random.Random(seed)
    out = []
    for k in range(case["count"]):
        nx, ny = case["nx"], case["ny"]
        if case["side_max"]:
            nx = ny = _log_int(sizes, case["side_min"], case["side_max"])
        a, q, incl = case["a"], case["q"], case["incl"]
        if case["call"] != "single":
            a = (0.0, 0.5, 0.9, 0.998)[k % 4] if case["metric"] == "kerr" else 0.0
            q = (-0.5, 0.1, 0.5)[k % 3] if case["metric"] == "q" else 0.0
            incl = (17.0, 60.0, 90.0)[(k // 4) % 3]
        a *= 1.0 - 0.02 * rng.random()
        q *= 1.0 - 0.02 * rng.random()
        incl = min(90.0, incl * (1.0 - 0.02 * rng.random()))
        zoom = 1.0 + 0.02 * rng.random()
        scene = ("sky", "disk")[k % 2] if case["scene"] == "both" else case["scene"]
        half = (8.0 if a or q else 10.0) if scene == "sky" else 25.0
        r = dict(a=a, q=q if case["metric"] == "q" else None, incl=incl, nx=nx, ny=ny,
                 extent=(-half * zoom, half * zoom, -half * zoom * ny / nx, half * zoom * ny / nx),
                 disk=scene != "sky", l0=2.8 if scene == "disk_l0" else None, r_in=0.0,
                 r_out=20.0, tol=case["tol"], first=0, n=nx * ny)
        if r["disk"]:
            r["r_in"] = 6.0 if a == 0.0 else osr.isco(a)
        if case["ranges"]:  # a chunk of the render, as the server deals them out
            r["n"] = max(1, int(nx * ny * sizes.uniform(0.3, 1.0)))
            r["first"] = int(sizes.random() * (nx * ny - r["n"] + 1))
        out.append(r)
    return out


def _particles(case, seed):
    """Unit-mass particles leaving r = 30 in Kerr: E = 1.2, L and theta uniform,
    outward p_r on the mass shell (host arrays)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, a, r = case["n"], case["a"], 30.0
    th, L = rng.uniform(0.3, np.pi - 0.3, n), rng.uniform(-4.0, 4.0, n)
    E = np.full(n, 1.2)
    s2 = np.sin(th) ** 2
    sig, dlt = r * r + a * a * (1.0 - s2), r * r - 2.0 * r + a * a
    big = (r * r + a * a) ** 2 - a * a * dlt * s2
    gtt, gtp = -big / (sig * dlt), -2.0 * a * r / (sig * dlt)
    gpp, grr = (dlt - a * a * s2) / (sig * dlt * s2), dlt / sig
    rest = -1.0 - (gtt * E * E - 2.0 * gtp * E * L + gpp * L * L)
    st = np.zeros((n, 6))
    st[:, 1], st[:, 2], st[:, 4] = r, th, np.sqrt(np.maximum(rest, 0.0) / grr)
    return st, E, L


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.call = case["call"]
    s.opts = dict(tol=case["tol"], precision=PRECISION[case["precision"]],
                  integrator=INTEGRATOR[case["integrator"]],
                  cell_phase_deg=10.0 * random.Random(seed + 1).random())
    if s.call == "states":
        st, E, L = _particles(case, seed)
        s.a = case["a"]
        s.states, s.E, s.L = (torch.from_numpy(v).cuda() for v in (st, E, L))
        return s
    renders = _renders(case, seed)
    cams = [osr.Camera(r["a"], R_OBS, r["incl"], r["extent"], r["nx"], r["ny"], q=r["q"])
            for r in renders]
    if s.call == "single":
        s.render, s.cam = renders[0], cams[0]
        if case["persistent"]:
            s.opts.update(persistent=True, workspace=torch.empty(
                osr.workspace_bytes(1), dtype=torch.uint8, device="cuda"))
        return s
    # batches write into one buffer per field; a render's outputs are slices of it
    fields = osr.DISK_FIELDS if any(r["disk"] for r in renders) else osr.SHADOW_FIELDS
    s.out = osr.alloc_outputs(sum(c.n_rays for c in cams), fields=fields)
    for t in s.out.values():
        t.zero_()
    s.requests, at = [], 0
    for r, cam in zip(renders, cams):
        s.requests.append(dict(camera=cam, disk=r["disk"], r_in=r["r_in"], r_out=r["r_out"],
                               l0=r["l0"], tol=r["tol"], first_ray=r["first"], n_rays=r["n"],
                               out={f: t[at:at + cam.n_rays] for f, t in s.out.items()}))
        at += cam.n_rays
    s.opts["workspace"] = torch.empty(osr.workspace_bytes(len(cams)), dtype=torch.uint8,
                                      device="cuda")
    if s.call == "plan":
        s.plan = osr.BatchPlan(len(cams), spacetime=osr.SPACETIME_QMETRIC
                               if case["metric"] == "q" else osr.SPACETIME_KERR, **s.opts)
    return s


def run(s):
    if s.call == "states":
        return osr.trace_states(s.a, R_OBS, s.states, s.E, s.L, mass2=1.0, **s.opts)
    if s.call == "plan":
        s.plan.launch(s.requests)
        return s.out
    if s.call == "batch":
        osr.trace_batch(s.requests, **s.opts)
        return s.out
    if s.render["disk"]:
        return osr.render_disk(s.cam, s.render["r_in"], s.render["r_out"], l0=s.render["l0"],
                               **s.opts)
    return osr.trace(s.cam, **s.opts)


# ---------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------
# Attempts per ray (accepted, rejected and surface location) at tol 1e-10, and their growth
# with the tolerance (a fifth-order step: tol^-1/5).
ATTEMPTS = {"sky": 345.0, "disk": 267.0, "states": 82.0}
# Operations of one attempt: six evaluations of Hamilton's equations in separated form and the
# sums of the step (the q-metric evaluation counted with its four transcendentals as one each).
FLOPS = {"kerr": 6 * 59 + 258, "q": 6 * 75 + 258}


def work(case):
    if case["call"] == "states":
        rays = [("states", case["n"])]
    else:
        rays = [("disk" if r["disk"] else "sky", r["n"]) for r in _renders(case, 0)]
    per = {"sky": 42, "disk": 66, "states": 42 + 64}  # bytes written (and read) per ray
    scale = (case["tol"] / 1e-10) ** -0.2
    return {"bytes": sum(per[k] * n for k, n in rays),
            "flops": sum(ATTEMPTS[k] * scale * FLOPS[case["metric"]] * n for k, n in rays)}


# ---------------------------------------------------------------------------
# The same rays in plain torch, 64 bits
# ---------------------------------------------------------------------------
CK = dict(
    a=[[], [1 / 5], [3 / 40, 9 / 40], [3 / 10, -9 / 10, 6 / 5],
       [-11 / 54, 5 / 2, -70 / 27, 35 / 27],
       [1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096]],
    b=[37 / 378, 0, 250 / 621, 125 / 594, 0, 512 / 1771],
    e=[-277 / 64512, 0, 6925 / 370944, -6925 / 202752, -277 / 14336, 277 / 7084])
DP = dict(
    a=[[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
       [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
       [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
       [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]],
    b=[35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0],
    e=[71 / 57600, 0, -71 / 16695, 71 / 1920, -17253 / 339200, 22 / 525, -1 / 40])


def _rhs_kerr(y, p):
    r, th, _, pr, pth = y
    s, c = torch.sin(th), torch.cos(th)
    a, E, L = p["a"], p["E"], p["L"]
    sig, dlt = r * r + (a * c) ** 2, r * (r - 2.0) + a * a
    P, W = (r * r + a * a) * E - a * L, L / s - a * E * s
    u = P / dlt
    N = dlt * pr * pr + pth * pth + W * W - P * u
    h2 = N / sig  # 2H
    k = torch.stack([dlt * pr, pth, W / s + a * u,
                     r * h2 - (r - 1.0) * (pr * pr + u * u) + 2.0 * r * E * u,
                     c * (W * (L / (s * s) + a * E) - a * a * s * h2)]) / sig
    return k, h2


def _rhs_q(y, p):
    r, th, _, pr, pth = y
    s, c = torch.sin(th), torch.cos(th)
    q, E, L = p["q"], p["E"], p["L"]
    k = q * (2.0 + q)
    D, f = r * (r - 2.0), 1.0 - 2.0 / r
    X = 1.0 + s * s / D
    fq, Xk = f ** q, X ** k
    Ht = -E * E / (f * fq)
    grr, gth, gph = f * fq * Xk, fq * Xk / (r * r), fq / (r * r * s * s)
    Hr, Hth, Hph = grr * pr * pr, gth * pth * pth, gph * L * L
    dlnf, dlnX = 2.0 / D, -s * s * (2.0 * r - 2.0) / (D * D * X)
    dpr = -0.5 * ((1.0 + q) * dlnf * (Hr - Ht) + k * dlnX * (Hr + Hth)
                  + (q * dlnf - 2.0 / r) * (Hth + Hph))
    dpth = -0.5 * (k * 2.0 * s * c / (D * X) * (Hr + Hth) - 2.0 * c / s * Hph)
    return torch.stack([grr * pr, gth * pth, gph * L, dpr, dpth]), Ht + Hr + Hth + Hph


def _attempt(rhs, T, y, h, p):
    ks = []
    for row in T["a"]:
        x = y
        for w, k in zip(row, ks):
            if w:
                x = x + (w * h) * k
        k, h2 = rhs(x, p)
        if not ks:
            twoH = h2
        ks.append(k)
    o, d = y, torch.zeros_like(y)
    for b, e, k in zip(T["b"], T["e"], ks):
        if b:
            o = o + (b * h) * k
        if e:
            d = d + (e * h) * k
    return o, d, twoH


def _rays(renders):
    """Initial data of every traced pixel, per ray: y (5, n) and the parameters."""
    ys, ps = [], []
    for m in renders:
        idx = torch.arange(m["first"], m["first"] + m["n"], device="cuda")
        a, q, r, th = m["a"], m["q"], R_OBS, m["incl"] * math.pi / 180.0
        s, c = math.sin(th), math.cos(th)
        if q is None:
            sig, dlt = r * r + (a * c) ** 2, r * r - 2.0 * r + a * a
            g_tp = -2.0 * a * r * s * s / sig
            g_pp = s * s * ((r * r + a * a) ** 2 - a * a * dlt * s * s) / sig
            g_th, g_rr, inv_at = sig, sig / dlt, math.sqrt(dlt * s * s / g_pp)
            r_h = 1.0 + math.sqrt(1.0 - a * a)
        else:
            f, X, k = 1.0 - 2.0 / r, 1.0 + s * s / (r * r - 2.0 * r), q * (2.0 + q)
            g_tp, g_pp = 0.0, f ** -q * r * r * s * s
            g_th, g_rr = f ** -q * r * r * X ** -k, f ** (-1.0 - q) * X ** -k
            inv_at, r_h, a = math.sqrt(f ** (1.0 + q)), 2.0, 0.0
        x0, x1, y0, y1 = m["extent"]
        x = x0 + ((idx % m["nx"]).double() + 0.5) * (x1 - x0) / m["nx"]
        z = y0 + ((idx // m["nx"]).double() + 0.5) * (y1 - y0) / m["ny"]
        one = torch.ones_like(x)
        ys.append(torch.stack([r * one, th * one, 0.0 * one,
                               -torch.sqrt(g_rr * (1.0 - (x * x + z * z) / (r * r))),
                               z * math.sqrt(g_th) / r]))
        ps.append(dict(a=a * one, q=(q or 0.0) * one, l0=(m["l0"] or 0.0) * one,
                       E=inv_at + x * g_tp / (r * math.sqrt(g_pp)), L=-x * math.sqrt(g_pp) / r,
                       cap=1.01 * r_h * one, r_in=m["r_in"] * one, r_out=m["r_out"] * one,
                       disk=torch.full_like(x, m["disk"], dtype=torch.bool)))
    return torch.cat(ys, 1), {k: torch.cat([p[k] for p in ps]) for k in ps[0]}


def _integrate(rhs, T, y, p, tol, H0):
    """Every ray to its end, one attempt per ray and turn; surfaces by 52
    halvings of the last step. Returns (end state, max |H|, on the disk)."""
    n = y.shape[1]
    end, maxH = torch.empty_like(y), torch.zeros_like(y[0])
    hit = torch.zeros(n, dtype=torch.bool, device=y.device)
    esc, half_pi = 1.1 * R_OBS, 0.5 * math.pi
    st = dict(p, y=y, h=torch.full_like(y[0], 0.01 * R_OBS), i=torch.arange(n, device=y.device),
              surf=torch.zeros_like(y[0], dtype=torch.int8), left=torch.zeros_like(y[0]),
              lo=torch.zeros_like(y[0]), hi=torch.zeros_like(y[0]), yF=y, yE=y,
              hE=torch.zeros_like(y[0]), H=torch.zeros_like(y[0]), done=torch.zeros_like(hit))

    def side(surf, o, cap):  # > 0 before the surface
        return torch.where(surf == 1, torch.cos(o[1]), torch.where(surf == 2, o[0] - cap,
                                                                   esc - o[0]))

    for turn in range(20000):
        if turn % 16 == 0:
            d = st["done"]
            if bool(d.any()):
                i = st["i"][d]
                end[:, i], maxH[i], hit[i] = st["yF"][:, d], st["H"][d], st["surf"][d] == 1
                st = {k: v[..., ~d] for k, v in st.items()}
            if not st["i"].numel():
                break
        y, surf, cap = st["y"], st["surf"], st["cap"]
        loc = surf > 0
        h = torch.where(loc, 0.5 * (st["lo"] + st["hi"]), torch.minimum(st["h"], 0.1 * y[0]))
        o, d, twoH = _attempt(rhs, T, y, h, st)
        act = ~loc & ~st["done"]
        st["H"] = torch.where(act, torch.maximum(st["H"], (0.5 * twoH - H0).abs()), st["H"])
        err = (d.abs() / (tol * (1.0 + torch.maximum(y.abs(), o.abs())))).amax(0)
        ok = act & (err <= 1.0)
        grow = torch.where(err <= 1.0, (0.9 * err ** -0.2).clamp(0.2, 5.0),
                           (0.9 * err ** -0.25).clamp(min=0.1))
        st["h"] = torch.where(act, h * grow, st["h"])
        # surface location: halve the step, keep the state at its upper end
        same = loc & ((side(surf, o, cap) > 0) == (side(surf, y, cap) > 0)) \
            & (side(surf, o, cap) != 0)
        up = loc & ~same
        st["lo"] = torch.where(same, h, st["lo"])
        st["hi"] = torch.where(up, h, st["hi"])
        st["yF"] = torch.where(up, o, st["yF"])
        st["left"] = torch.where(loc, st["left"] - 1.0, st["left"])
        over = loc & (st["left"] <= 0) & ~st["done"]
        miss = over & (surf == 1) & ~((st["yF"][0] >= st["r_in"]) & (st["yF"][0] <= st["r_out"]))
        st["done"] = st["done"] | (over & ~miss)
        # the end of an accepted step, or of one whose crossing missed the disk
        z = torch.where(miss, st["yE"], o)
        st["yE"] = torch.where(ok, o, st["yE"])
        c0, c1 = half_pi - y[1], half_pi - o[1]
        eq = ok & st["disk"] & (((c0 > 0) & (c1 <= 0)) | ((c0 < 0) & (c1 >= 0)))
        test = (ok & ~eq) | miss
        capt, escd = test & (z[0] < cap), test & (z[0] > esc) & ~(z[0] < cap)
        new = eq | capt | escd
        kind = torch.where(eq, 1, torch.where(capt, 2, 3)).to(torch.int8)
        st["surf"] = torch.where(new, kind, torch.where(miss, 0, surf).to(torch.int8))
        step = torch.where(miss, st["hE"], h)
        st["hE"] = torch.where(ok, h, st["hE"])
        st["lo"] = torch.where(new, 0.0, st["lo"])
        st["hi"] = torch.where(new, step, st["hi"])
        st["yF"] = torch.where(new, z, st["yF"])
        st["left"] = torch.where(new, 52.0, st["left"])
        st["y"] = torch.where(test & ~capt & ~escd, z, y)
    else:
        raise RuntimeError("rays left after %d attempts" % turn)
    return end, maxH, hit


MAX_EXACT = 4_000_000  # rays that plain torch integrates in under 20 seconds


def exact(case, seed):
    rhs = _rhs_q if case["metric"] == "q" else _rhs_kerr
    T, H0 = (DP if case["integrator"] == "dp45" else CK), 0.0
    if case["call"] == "states":
        st, E, L = (torch.from_numpy(v).cuda() for v in _particles(case, seed))
        y, zero, H0, total, at = st.T[1:].contiguous(), torch.zeros_like(E), -0.5, case["n"], None
        p = dict(a=case["a"] + zero, q=zero, l0=zero, E=E, L=L, r_in=zero, r_out=zero,
                 cap=1.01 * (1.0 + math.sqrt(1.0 - case["a"] ** 2)) + zero, disk=zero > 0.0)
    else:
        renders = _renders(case, seed)
        if sum(r["n"] for r in renders) > MAX_EXACT:
            return None
        y, p = _rays(renders)
        total, at, begin = sum(r["nx"] * r["ny"] for r in renders), [], 0
        for r in renders:
            at.append(torch.arange(begin + r["first"], begin + r["first"] + r["n"], device="cuda"))
            begin += r["nx"] * r["ny"]
        at = torch.cat(at)
    end, maxH, hit = _integrate(rhs, T, y, p, case["tol"], H0)
    # gas on circular orbits: u^t from its normalisation, g = 1 / (u^t (E - Omega L))
    r, a, l0 = end[0], p["a"], p["l0"]
    gtt, gtp, gpp = -(1.0 - 2.0 / r), -2.0 * a / r, r * r + a * a + 2.0 * a * a / r
    om = torch.where(l0 != 0.0, -(gtp + l0 * gtt) / (gpp + l0 * gtp), 1.0 / (r ** 1.5 + a))
    norm = -gtt - 2.0 * om * gtp - om * om * gpp
    g = torch.where(hit & (norm > 0.0), norm.clamp(min=0.0).sqrt() / (p["E"] - om * p["L"]), 0.0)
    vals = dict(r=r, theta=end[1], phi=end[2], g=g, intensity=g ** 3 / (r * r),
                r_hit=torch.where(hit, r, 0.0))
    if case["precision"] == "fp64":  # elsewhere max |H| is that of the arithmetic's own rounding
        vals["max_abs_H"] = maxH
    disk = case["scene"] != "sky" and case["call"] != "states"
    out = {}
    for f in (osr.DISK_FIELDS if disk else osr.SHADOW_FIELDS):
        v = vals.get(f)
        if v is not None and at is not None and total != v.numel():
            v = torch.zeros(total, dtype=torch.float64, device="cuda").index_copy(0, at, v)
        out[f] = v
    return out
