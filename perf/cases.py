"""What the library is measured on: its public entry points over the range of sizes, scenes and
options that its users run, from one small plane to the full synthetic city.

A case is a dict of plain values.  ``op`` names the entry points that ``run`` goes through:

  solve   recv_order + gbs_solve: receivers in, field out, tracing included
  sum     gbs_sum over a trace the program keeps
  train   gbs_field forward, a least-squares loss, and its gradients (autograd)
  grad    gbs_sum_backward over a trace the program keeps
  batch   Batch.submit: several sources as one replayed unit
  trace   Trace + segments: the ray tracer and its segment list
  synth   synthesize: time signals from per-frequency fields

Scenes: ``plane`` (ground only), ``city`` (8 x 8 boxes over 500 m on the ground), ``big``
(32 x 32 boxes over 2 km).  Receivers: a ``grid`` map at ear height, or ``scatter``ed points.
``cull`` is the tile pre-cull switch, ``precision`` 32 or 64, ``losses`` air absorption and a
porous ground, ``window`` line (planes: the unfolded images) or segment.  ``prepare`` draws the
scene, the source, the receivers and the coefficients from the seed (the tracer's scene is one
city, moved and scaled, so that every seed gives as many segments).
"""
import math

import numpy as np
import torch

from paper_2501_13382_gb300 import gbt as G
from paper_2501_13382_gb300 import inputs as I
from paper_2501_13382_gb300.autograd import gbs_field

C_AIR = 343.0
CUTOFF = 16.0


def _case(op, scene, rays, refl, path, recv, n, half, bands, f_lo, f_hi, **more):
    d = dict(op=op, scene=scene, rays=rays, refl=refl, path=float(path), recv=recv, n=n,
             half=float(half), bands=bands, f_lo=float(f_lo), f_hi=float(f_hi), cull=False,
             precision=32, losses=False, sources=1, samples=0)
    d.update(more)
    return d


def listed():
    cases = [
        # one interactive update: a source over a plane, a small map, one band
        _case("solve", "plane", 1024, 2, 200, "grid", 64, 50, 1, 500, 500,
              name="solve_plane_small"),
        # the open-plane map in six octave bands, with the library's default options
        _case("sum", "plane", 65536, 3, 1000, "grid", 256, 500, 6, 125, 4000,
              name="sum_plane_6_bands"),
        # scattered listeners at different heights (no grid, a ragged count), pre-cull on
        _case("sum", "plane", 32768, 3, 1000, "scatter", 9973, 300, 3, 250, 2000, cull=True,
              name="sum_plane_scatter_cull"),
        # the full city noise map, pre-cull on: trace, lists, sum
        _case("solve", "city", 1 << 20, 8, 1000, "grid", 512, 250, 1, 1000, 1000, cull=True,
              name="solve_city_1m_rays_cull"),
        # a coarser city map by someone who leaves the options at their defaults
        _case("solve", "city", 65536, 8, 1000, "grid", 200, 250, 2, 500, 1000,
              name="solve_city_64k_rays"),
        # a city map in eight bands with the atmosphere and a porous ground
        _case("sum", "city", 131072, 8, 1000, "grid", 192, 250, 8, 125, 4000, cull=True,
              losses=True, name="sum_city_8_bands_losses_cull"),
        # one step of fitting reflection coefficients, source weights and beam widths
        _case("train", "city", 262144, 6, 1000, "grid", 128, 250, 4, 250, 2000, cull=True,
              name="train_city_4_bands_cull"),
        # the gradient alone, default options, fewer receivers (a set of microphones)
        _case("grad", "city", 65536, 6, 1000, "scatter", 4000, 250, 4, 250, 2000,
              name="grad_city_4_bands"),
        # several sources of uneven ray counts, eight bands, replayed as one unit
        _case("batch", "city", 65536, 8, 1000, "grid", 128, 250, 8, 125, 4000, cull=True,
              sources=8, name="batch_city_8_sources_cull"),
        # a reference field in FP64 to compare others with
        _case("sum", "plane", 16384, 3, 1000, "grid", 128, 500, 2, 500, 2000, precision=64,
              name="sum_plane_fp64"),
        # the tracer on a large mesh, for a program that keeps the segment list
        _case("trace", "big", 262144, 8, 1000, "grid", 1, 1000, 1, 1000, 1000,
              name="trace_12k_triangles"),
        # time signals for a map of listeners from six bands
        _case("synth", "plane", 0, 0, 0, "grid", 256, 500, 6, 125, 4000, samples=2048,
              name="synth_6_bands"),
    ]
    return cases


def _log_int(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi], odd half of the time."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.5:
        v |= 1
    return max(lo, min(hi, v))


def draw(rng):
    op = rng.choice(["solve", "sum", "sum", "train", "grad", "batch", "sum64", "trace", "synth"])
    bands = rng.choice([1, 1, 2, 3, 4, 5, 6, 7, 8])
    f_lo = 125.0 * 2.0 ** rng.uniform(0.0, 2.0)
    f_hi = f_lo if bands == 1 else min(4000.0, f_lo * 2.0 ** rng.uniform(1.0, 4.0))
    scene = rng.choice(["plane", "city"])
    refl = rng.randint(1, 3) if scene == "plane" else rng.randint(3, 8)
    grid = rng.random() < 0.7
    cull = rng.random() < 0.5
    n = _log_int(rng, 24, 200) if grid else _log_int(rng, 500, 40000)
    recv = "grid" if grid else "scatter"
    half = rng.uniform(60.0, 250.0)
    path = rng.uniform(200.0, 1000.0)
    rays = _log_int(rng, 1000, 200000)
    if op == "trace":
        return _case("trace", rng.choice(["plane", "city", "big"]), _log_int(rng, 1000, 262144),
                     rng.randint(1, 8), path, "grid", 1, half, 1, 1000, 1000)
    if op == "synth":
        return _case("synth", "plane", 0, 0, 0, "scatter", _log_int(rng, 100, 65536), half,
                     bands, f_lo, f_hi, samples=_log_int(rng, 64, 2048))
    if op == "sum64":
        return _case("sum", scene, _log_int(rng, 500, 8192 if scene == "plane" else 2048), refl,
                     path, "scatter", _log_int(rng, 200, 16384), half, min(bands, 3), f_lo, f_hi,
                     precision=64)
    if op == "batch":
        return _case("batch", "city", _log_int(rng, 4096, 65536), refl, path, "grid",
                     _log_int(rng, 24, 128), half, bands, f_lo, f_hi, cull=cull,
                     sources=rng.randint(2, 8))
    if op in ("train", "grad"):
        return _case(op, "city", _log_int(rng, 2000, 131072), refl, path, recv,
                     _log_int(rng, 16, 64) if grid else _log_int(rng, 200, 4000), half,
                     min(bands, 4), f_lo, f_hi, cull=cull)
    return _case(op, scene, rays, refl, path, recv, n, half, bands, f_lo, f_hi, cull=cull,
                 losses=(op == "sum" and rng.random() < 0.3))


# ---------------------------------------------------------------- inputs --

def _scene(case, rng):
    """Triangles (T, 3, 3), facet and material per triangle and gamma per material (0: ground)."""
    if case["scene"] == "plane":
        return (np.zeros((0, 3, 3)), np.zeros(0, np.int32), np.zeros(0, np.int32),
                rng.uniform(0.85, 1.0, 1).astype(np.float32))
    side, extent = (8, 500.0) if case["scene"] == "city" else (32, 2000.0)
    nb, cell = side * side, extent / side
    w = rng.uniform(20.0, 60.0, (nb, 2))
    h = rng.uniform(10.0, 60.0, nb)
    at = -extent / 2 + cell * (np.stack([np.arange(nb) % side, np.arange(nb) // side], 1) + 0.5)
    at = at + rng.uniform(-1.0, 1.0, (nb, 2)) * np.maximum(0.0, (cell - w) / 2 - 1.25)
    lo, hi = at - w / 2, at + w / 2
    # corner q of a box: x from bit 0, y from bit 1, z from bit 2
    q = np.arange(8)
    x = np.where(q & 1, hi[:, :1], lo[:, :1])
    y = np.where(q & 2, hi[:, 1:], lo[:, 1:])
    z = np.where(q & 4, h[:, None], 0.0)
    corner = np.stack([x, y, z], 2)
    quads = np.array([[0, 2, 6, 4], [1, 5, 7, 3], [0, 4, 5, 1], [2, 3, 7, 6], [0, 1, 3, 2],
                      [4, 6, 7, 5]])
    tri = np.concatenate([quads[:, [0, 1, 2]], quads[:, [0, 2, 3]]], 1).reshape(12, 3)
    return (corner[:, tri].reshape(-1, 3, 3), np.arange(6 * nb, dtype=np.int32).repeat(2),
            (1 + np.arange(nb) % 8).astype(np.int32).repeat(12),
            np.concatenate([[1.0], rng.uniform(0.6, 0.95, 8)]).astype(np.float32))


def _beam_b(rays, freq):
    """Beam parameter whose 1/e half-width at 100 m is the fan spacing there, else 100 m."""
    k = 2.0 * math.pi * freq / C_AIR
    a = 0.5 * k * (4.0 * math.pi / rays) * 1e4
    return 2e4 / (a + math.sqrt(a * a - 4e4)) if a > 200.0 else 100.0


def _inputs(case, seed):
    """Everything of a case as host arrays, from the seed alone."""
    rng = np.random.default_rng([seed, 13382])
    moved = rng if case["op"] != "trace" else np.random.default_rng(13382)
    d = {"scene": _scene(case, moved), "path": case["path"]}
    n_src = case["sources"]
    pos = np.zeros((n_src, 3))
    pos[:, :2] = moved.uniform(-1.0, 1.0, (n_src, 2))
    if case["scene"] != "plane":      # cell corners are streets
        pos[1:, :2] += 62.5 * rng.integers(-3, 4, (n_src - 1, 2))
    pos[:, 2] = moved.uniform(1.5, 8.0, n_src)
    if case["op"] == "trace":         # one scene, moved and scaled: the segment count stays
        shift, size = np.append(rng.uniform(-50.0, 50.0, 2), 0.0), rng.uniform(0.9, 1.1)
        d["scene"] = (size * (d["scene"][0] + shift), *d["scene"][1:])
        pos, d["path"] = size * (pos + shift), size * case["path"]
    rays = [case["rays"]] * n_src
    if n_src > 1:                     # uneven: log-uniform from a sixteenth up
        rays = [max(64, int(case["rays"] * 2.0 ** u)) for u in rng.uniform(-4.0, 0.0, n_src)]
    d["pos"], d["rays"] = pos, rays
    h = case["half"]
    if case["recv"] == "grid":
        g = np.linspace(-h, h, case["n"]) if case["n"] > 1 else np.zeros(1)
        off = rng.uniform(-0.5, 0.5, 2)
        xx, yy = np.meshgrid(g + off[0], g + off[1], indexing="xy")
        d["recv"] = np.stack([xx.ravel(), yy.ravel(), np.full(xx.size, 1.5)], 1).astype(np.float32)
    else:
        d["recv"] = (rng.uniform(-1.0, 1.0, (case["n"], 3)) * [h, h, 9.5]
                     + [0.0, 0.0, 11.0]).astype(np.float32)
    nf = case["bands"]
    d["freqs"] = [case["f_lo"] * (case["f_hi"] / case["f_lo"]) ** (i / max(nf - 1, 1))
                  for i in range(nf)]
    d["b"] = [[_beam_b(max(r, 1), f) for f in d["freqs"]] for r in rays]
    d["absorption"] = d["sigma"] = None
    if case["losses"]:
        d["absorption"] = [5.7e-4 * (f / 1000.0) ** 1.5 for f in d["freqs"]]   # Np/m
        d["sigma"] = np.zeros(len(d["scene"][3]), np.float32)
        d["sigma"][0] = 200.0                                                   # kPa s m^-2
    nr = len(d["recv"])
    if case["op"] in ("train", "grad"):
        d["weight"] = (4.0 * math.pi / case["rays"]
                       * rng.uniform(0.8, 1.2, case["rays"])).astype(np.float32)
        d["target"] = (1e-3 * rng.standard_normal((nf, nr, 2))).astype(np.float32).view(np.complex64)[..., 0]
    if case["op"] == "synth":
        d["field"] = rng.standard_normal((nf, nr, 2)).astype(np.float32).view(np.complex64)[..., 0]
        d["amp"] = [complex(a, b) for a, b in rng.uniform(-1.0, 1.0, (nf, 2))]
        d["t0"], d["dt"] = float(rng.uniform(0.0, 2.0)), 1.0 / 16000.0
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    dev = lambda a: None if a is None else torch.as_tensor(a, device="cuda")  # noqa: E731
    tri, face, mat, gamma = d["scene"]
    st = {"case": case, "freqs": d["freqs"], "recv": dev(d["recv"]), "gamma": dev(gamma),
          "window": G.WINDOW_LINE if case["scene"] == "plane" else G.WINDOW_SEGMENT}
    if case["op"] == "synth":
        st.update(field=dev(d["field"]), amp=d["amp"], t0=d["t0"], dt=d["dt"])
        return st
    scene = G.Scene(I.Scene(C_AIR, True, 0.0, 0, tri, mat, face, gamma))
    src = [I.Source(p, r, case["refl"], d["path"]) for p, r in zip(d["pos"], d["rays"])]
    st.update(scene=scene, sources=src, b=d["b"], absorption=d["absorption"],
              sigma=dev(d["sigma"]))
    if case["op"] in ("solve", "trace"):
        return st
    st["traces"] = [G.Trace(scene, s) for s in src]
    st["order"] = G.recv_order(st["recv"])
    if case["op"] in ("train", "grad"):
        st["weight"], st["target"] = dev(d["weight"]), dev(d["target"])
    if case["op"] == "train":
        st["leaves"] = [st["gamma"].clone().requires_grad_(), st["weight"].clone().requires_grad_(),
                        torch.tensor(d["b"][0], dtype=torch.float64, device="cuda").requires_grad_()]
    if case["op"] == "batch":
        st["batch"] = G.Batch([dict(trace=t, recv=st["recv"], freqs=st["freqs"], beam_b=b,
                                    gamma=st["gamma"], order=st["order"])
                               for t, b in zip(st["traces"], st["b"])],
                              window=st["window"], tile_cull=case["cull"])
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "solve":
        return G.gbs_solve(st["scene"], st["sources"][0], st["recv"], st["freqs"], st["b"][0],
                           st["gamma"], order=G.recv_order(st["recv"]), window=st["window"],
                           tile_cull=case["cull"])
    if op == "sum":
        return G.gbs_sum(st["traces"][0], st["recv"], st["freqs"], st["b"][0], st["gamma"],
                         order=st["order"], window=st["window"], tile_cull=case["cull"],
                         precision=G.PRECISION_F64 if case["precision"] == 64 else G.PRECISION_F32,
                         absorption=st["absorption"], flow_resistivity=st["sigma"])
    if op == "train":
        gamma, weight, b = st["leaves"]
        p = gbs_field(st["traces"][0], st["recv"], st["freqs"], b, gamma, ray_weight=weight,
                      order=st["order"], window=st["window"], tile_cull=case["cull"])
        loss = (p - st["target"]).abs().pow(2).sum()
        return (p.detach(), *torch.autograd.grad(loss, [gamma, weight, b]))
    if op == "grad":
        return G.gbs_sum_backward(st["traces"][0], st["recv"], st["freqs"], st["b"][0],
                                  st["gamma"], st["target"], ray_weight=st["weight"],
                                  order=st["order"], window=st["window"], tile_cull=case["cull"])
    if op == "batch":
        st["batch"].submit()
        return st["batch"].outputs
    if op == "trace":
        return G.Trace(st["scene"], st["sources"][0]).segments()
    return G.synthesize(st["field"], st["freqs"], st["amp"], st["t0"], st["dt"], case["samples"])


# --------------------------------------------------- what cannot be avoided --

def _paths(case):
    """Segments per ray, and beam paths that meet a receiver (both typical of the scene)."""
    return (1.5, 2.0) if case["scene"] == "plane" else (3.0, 4.0)


def work(case):
    """Bytes: each input and output once (segments as FP64 origin, direction, length and start).
    Operations: 57 per kept (receiver, segment, band) and 12 per band of its adjoint, with the
    count of the beams that reach a receiver at 200 m estimated from the fan and the beam width;
    a ray-segment takes about 60 through its hierarchy and reflection."""
    nr = case["n"] ** 2 if case["recv"] == "grid" else case["n"]
    nf = case["bands"]
    if case["op"] == "synth":
        return {"bytes": 8.0 * nf * nr + 4.0 * nr * case["samples"],
                "flops": 4.0 * nf * nr * case["samples"]}
    per_ray, paths = _paths(case)
    rays = case["rays"] * (1.0 if case["sources"] == 1 else 0.34 * case["sources"])
    seg = per_ray * rays
    if case["op"] == "trace":
        return {"bytes": 81.0 * seg, "flops": 60.0 * seg}
    kept = 0.0
    for i in range(nf):
        f = case["f_lo"] * (case["f_hi"] / case["f_lo"]) ** (i / max(nf - 1, 1))
        b = _beam_b(case["rays"], f)
        share = 0.5 * CUTOFF * (1.0 + (b / 200.0) ** 2) / (2.0 * math.pi * f / C_AIR * b)
        kept += nr * paths * rays * min(1.0, share)
    work_bytes = (64.0 if case["op"] != "solve" else 0.0) * seg + 12.0 * nr + 8.0 * nf * nr * case["sources"]
    flops = 57.0 * kept
    if case["op"] == "solve":
        flops += 60.0 * seg
    if case["op"] == "train":
        flops += (57.0 + 12.0) * kept
        work_bytes += 8.0 * rays + 8.0 * nf * nr
    if case["op"] == "grad":
        flops += 12.0 * kept
        work_bytes += 8.0 * rays
    return {"bytes": work_bytes, "flops": flops}


# ------------------------------------------------------- the same in 64 bits --

def _trace64(case, d, k):
    """Segments of source k in ray order: origin, direction, length, start, ray, table of the
    materials of the reflections before it (-1 padded) and their cosines of incidence."""
    tri = torch.as_tensor(d["scene"][0], dtype=torch.float64, device="cuda")
    face = torch.as_tensor(d["scene"][1], device="cuda").long()
    mat = torch.as_tensor(d["scene"][2], device="cuda").long()
    n_rays, n_refl = d["rays"][k], case["refl"]
    i = torch.arange(n_rays, dtype=torch.float64, device="cuda")
    z = 1.0 - (2.0 * i + 1.0) / n_rays
    phi = i * (math.pi * (3.0 - math.sqrt(5.0)))
    r = torch.sqrt(1.0 - z * z)
    t = torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], 1)
    o = torch.as_tensor(d["pos"][k], dtype=torch.float64, device="cuda").expand(n_rays, 3).clone()
    s0 = torch.zeros(n_rays, dtype=torch.float64, device="cuda")
    last = torch.full((n_rays,), -1, dtype=torch.long, device="cuda")
    ids = torch.arange(n_rays, device="cuda")
    mats = torch.full((n_rays, max(n_refl, 1)), -1, dtype=torch.long, device="cuda")
    cosines = torch.zeros((n_rays, max(n_refl, 1)), dtype=torch.float64, device="cuda")
    if len(tri):
        v0, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
        nrm = torch.linalg.cross(e1, e2)
        normal = nrm / nrm.norm(dim=1, keepdim=True)
    got = []
    step = max(1, (1 << 26) // max(1, len(tri)))
    for depth in range(n_refl + 1):
        tg = (0.0 - o[:, 2]) / t[:, 2]
        ok = (last != -2) & (t[:, 2] != 0) & (tg > 1e-9)
        best = torch.where(ok, tg, torch.inf)
        prim = torch.where(ok, 0, -1)
        for a in range(0, len(o) if len(tri) else 0, step):
            oo, tt, sl = o[a:a + step], t[a:a + step], slice(a, a + step)
            # plane hit, then barycentric coordinates in the triangle's own plane
            den = tt @ nrm.T
            hit = ((v0 * nrm).sum(1) - oo @ nrm.T) / den
            ray, idx = ((hit > 1e-9) & (hit < best[sl, None])
                        & (face[None, :] != last[sl, None])).nonzero(as_tuple=True)
            h = hit[ray, idx]
            w = oo[ray] + h[:, None] * tt[ray] - v0[idx]
            nn = (nrm[idx] ** 2).sum(1)
            u = (torch.linalg.cross(w, e2[idx]) * nrm[idx]).sum(1) / nn
            v = (torch.linalg.cross(e1[idx], w) * nrm[idx]).sum(1) / nn
            inside = (u >= 0) & (v >= 0) & (u + v <= 1)
            ray, idx, h = ray[inside], idx[inside], h[inside]
            near = best[sl].clone().scatter_reduce_(0, ray, h, "amin")
            win = h == near[ray]
            first = torch.full((len(oo),), 1 << 40, dtype=torch.long, device="cuda")
            first.scatter_reduce_(0, ray[win], idx[win] + 1, "amin")
            prim[sl] = torch.where(first < (1 << 40), first, prim[sl])
            best[sl] = near
        remaining = d["path"] - s0
        ends = (prim < 0) | (best >= remaining)
        length = torch.where(ends, remaining, best)
        got.append((ids, torch.full_like(ids, depth), o, t, length, s0, mats.clone(), cosines.clone()))
        if depth == n_refl:
            break
        go = ~ends
        ids, o, t, best, prim, s0 = ids[go], o[go], t[go], best[go], prim[go], s0[go]
        mats, cosines = mats[go], cosines[go]
        nv = torch.zeros_like(o)
        nv[:, 2] = 1.0
        last = torch.full_like(ids, -2)
        hit_mat = torch.zeros_like(ids)
        if len(tri):
            on = prim > 0
            nv[on] = normal[prim[on] - 1]
            last[on] = face[prim[on] - 1]
            hit_mat[on] = mat[prim[on] - 1]
        o = o + best[:, None] * t
        dn = (t * nv).sum(1)
        t = t - 2.0 * dn[:, None] * nv
        s0 = s0 + best
        mats[:, depth], cosines[:, depth] = hit_mat, dn.abs()
    cat = [torch.cat(c) for c in zip(*got)]
    at = torch.argsort(cat[0] * (n_refl + 2) + cat[1])
    return [c[at] for c in cat]


def _amplitude(mats, gamma, weight):
    """W times the product of gamma over the reflections (differentiable)."""
    g = torch.cat([gamma, torch.ones(1, dtype=gamma.dtype, device="cuda")])
    return weight * g[torch.where(mats < 0, len(gamma), mats)].prod(1)


def _porous(mats, cosines, sigma, freq):
    """Product of the plane-wave reflection factors over the porous reflections."""
    s = torch.as_tensor(sigma, dtype=torch.float64, device="cuda")
    sg = torch.where(mats < 0, 0.0, s[mats.clamp(min=0)])
    x = freq / torch.where(sg > 0, sg, 1.0)
    zc = torch.complex(1.0 + 9.08 * x ** -0.75, 11.9 * x ** -0.73) * cosines
    return torch.where(sg > 0, (zc - 1.0) / (zc + 1.0), torch.ones_like(zc)).prod(1)


def _pairs(case, seg, x, freqs, b):
    """Candidate (receiver, segment) pairs in blocks: indices, s and n^2, within the window and
    the widest beam's cutoff."""
    _, _, o, t, length, s0, _, _ = seg
    line = case["scene"] == "plane"
    kb = min(2.0 * math.pi * f / C_AIR * v for f, v in zip(freqs, b))
    b2 = max(v * v for v in b)
    xx = (x * x).sum(1)
    step = max(1, (1 << 27) // len(x))
    for a in range(0, len(o), step):
        oo, tt = o[a:a + step], t[a:a + step]
        sl = x @ tt.T - (oo * tt).sum(1)
        s = sl + s0[a:a + step]
        n2 = xx[:, None] - 2.0 * (x @ oo.T) + (oo * oo).sum(1) - sl * sl
        keep = kb * n2 <= 2.0 * CUTOFF * (s * s + b2) * 1.000001 + 1e-6
        del n2, s
        keep &= (sl > -1e-6) if not line else (sl + s0[a:a + step] > -1e-6)
        if not line:
            keep &= sl < length[a:a + step] + 1e-6
        r, j = keep.nonzero(as_tuple=True)
        del sl, keep
        j += a
        w = x[r] - o[j]
        sl = (w * t[j]).sum(1)
        n2 = torch.linalg.cross(w, t[j]).square().sum(1)
        s = sl + s0[j]
        ok = (s >= 0) if line else (sl >= 0) & (sl < length[j])
        yield r[ok], j[ok], s[ok], n2[ok]


def _beam(s, n2, f, b):
    """One beam without its amplitude, on the pairs within its cutoff (their mask first)."""
    k = 2.0 * math.pi * f / C_AIR
    ok = k * n2 * b <= 2.0 * CUTOFF * (s * s + b * b)
    s, n2 = s[ok], n2[ok]
    e = torch.complex(s, torch.full_like(s, -b))
    return ok, s, n2, e, k * b / (8.0 * math.pi ** 2) * torch.exp(1j * k * (s + n2 / (2.0 * e))) / e


def _field64(case, d, k):
    seg = _trace64(case, d, k)
    x = torch.as_tensor(d["recv"], dtype=torch.float64, device="cuda")
    gamma = torch.as_tensor(d["scene"][3], dtype=torch.float64, device="cuda")
    weight = 4.0 * math.pi / d["rays"][k]
    if "weight" in d:
        weight = torch.as_tensor(d["weight"], dtype=torch.float64, device="cuda")[seg[0]]
    amp = _amplitude(seg[6], gamma, weight)
    p = torch.zeros((case["bands"], len(x)), dtype=torch.complex128, device="cuda")
    loss = [amp.to(torch.complex128)] * case["bands"]
    if case["losses"]:
        loss = [amp * _porous(seg[6], seg[7], d["sigma"], f) for f in d["freqs"]]
    for r, j, s, n2 in _pairs(case, seg, x, d["freqs"], d["b"][k]):
        for f in range(case["bands"]):
            ok, s_f, _, _, c = _beam(s, n2, d["freqs"][f], d["b"][k][f])
            c = c * loss[f][j[ok]]
            if case["losses"]:
                c = c * torch.exp(-d["absorption"][f] * s_f)
            p[f].real.index_add_(0, r[ok], c.real)
            p[f].imag.index_add_(0, r[ok], c.imag)
    return p


def _grads64(case, d, g):
    """Gradients in gamma, the ray weights and b of a loss with dL/dp = g."""
    seg = _trace64(case, d, 0)
    x = torch.as_tensor(d["recv"], dtype=torch.float64, device="cuda")
    gamma = torch.as_tensor(d["scene"][3], dtype=torch.float64, device="cuda").requires_grad_()
    weight = torch.as_tensor(d["weight"], dtype=torch.float64, device="cuda").requires_grad_()
    big_g = torch.zeros(len(seg[0]), dtype=torch.float64, device="cuda")
    amp = _amplitude(seg[6], gamma, weight[seg[0]])
    db = torch.zeros(case["bands"], dtype=torch.float64, device="cuda")
    for r, j, s, n2 in _pairs(case, seg, x, d["freqs"], d["b"][0]):
        for f in range(case["bands"]):
            b = d["b"][0][f]
            k = 2.0 * math.pi * d["freqs"][f] / C_AIR
            ok, s_f, n2_f, e, c = _beam(s, n2, d["freqs"][f], b)
            gc = g[f][r[ok]].conj() * c
            big_g.index_add_(0, j[ok], gc.real)
            dlog = 1.0 / b + 1j / e - k * n2_f / (2.0 * e * e)
            db[f] += ((gc * dlog).real * amp.detach()[j[ok]]).sum()
    return (*torch.autograd.grad((amp * big_g).sum(), [gamma, weight]), db)


def exact(case, seed):
    nr = case["n"] ** 2 if case["recv"] == "grid" else case["n"]
    if nr * case["rays"] * _paths(case)[0] > 6e10:
        return None
    d = _inputs(case, seed)
    op = case["op"]
    if op == "synth":
        t = d["t0"] + np.arange(case["samples"]) * d["dt"]
        p = torch.as_tensor(d["field"], device="cuda").to(torch.complex128)
        ph = torch.as_tensor(np.array(d["amp"])[None, :]
                             * np.exp(-2j * np.pi * np.outer(t, d["freqs"])), device="cuda")
        return ph.real @ p.real - ph.imag @ p.imag
    if op == "trace":
        ids, depth, o, t, length, s0, _, _ = _trace64(case, d, 0)
        return {"n_segments": None, "ray_off": None, "o": o, "t": t, "L": length, "s0": s0,
                "ray": None, "depth": None, "bmat": None, "hit": None}
    if op == "batch":
        return [_field64(case, d, k) for k in range(case["sources"])]
    if op == "grad":
        return _grads64(case, d, torch.as_tensor(d["target"], device="cuda").to(torch.complex128))
    p = _field64(case, d, 0)
    if op == "train":
        g = 2.0 * (p - torch.as_tensor(d["target"], device="cuda").to(torch.complex128))
        return (p, *_grads64(case, d, g))
    return p
