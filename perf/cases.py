"""The work this framework is measured on, each case through its public entry points.

A case is a dict of plain values; ``kind`` says which entry points one pass calls:

  calls      scene update, trace, synthesis, point cloud as separate calls
  frame      ``Forward``: new vertices, then one replay of the captured step
  trace      scene update and trace (path records out)
  synth      ``synthesize`` of given path records (split or FP64 phase, static or moving)
  synth_bwd  ``synthesize_bwd`` of given path records
  points     ``pointcloud`` of a given IF cube
  recon      ``Reconstruction``: one replayed iteration (image loss) from given vertices
  grad       ``Simulator``: image loss and its gradient, separate calls

Inputs are seeded and made here: superquadrics or icospheres over a ground plane, the
77 GHz radars of the paper's Section 4, path records of a sphere over a ground plane in
closed form, cubes of point scatterers.  ``exact`` evaluates the same model in FP64 torch
(brute-force nearest hits, term-by-term sums, direct transforms).
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2311_13182_gb300 as sbr
from paper_2311_13182_gb300.autograd import Simulator
from paper_2311_13182_gb300.recon import Reconstruction

C0 = 299_792_458.0
F0, BW, TC, TREP = 77e9, 4e9, 40e-6, 40e-6
DEV = "cuda"
F64, C128 = torch.float64, torch.complex128


def listed():
    return [
        # the smallest scene of the repository (320 triangles, 64 x 64 rays, one chirp), simulated
        # call by call: launches and latency
        dict(name="calls_sphere320_64", kind="calls", mesh="sphere", tris=320, G=64, K=2, tx=1, ns=256, nc=1),
        # the headline forward step: 20,002 triangles, a million rays, 12 antennas x 128 chirps x
        # 256 samples to a point cloud, geometry moving from frame to frame
        dict(name="frame_superquadric20k_1024", kind="frame", mesh="superquadric", tris=20000, G=1024, K=3, tx=3,
             ns=256, nc=128),
        # the largest serving request: about 200,000 triangles, four million rays (an odd grid)
        dict(name="trace_superquadric200k_1999", kind="trace", mesh="superquadric", tris=200000, G=1999, K=3, tx=1,
             materials=False, jitter=False),
        # synthesis of a MIMO frame's paths (12 antennas, 128 equal chirps)
        dict(name="synth_mimo256", kind="synth", scene="ground", dist=2.0, G=700, K=3, tx=3, ns=256, nc=128,
             mode="split", moving=False),
        # long range, long chirps: 4096 samples at 10 m over a 2048 x 2048 ray grid
        dict(name="synth_range4096", kind="synth", scene="sphere", dist=10.0, G=2048, K=2, tx=1, ns=4096, nc=1,
             mode="split", moving=False),
        # the FP64 carrier phase at 20 m (a megaray grid)
        dict(name="synth_fp64_1024", kind="synth", scene="sphere", dist=20.0, G=1023, K=2, tx=1, ns=1024, nc=1,
             mode="fp64", moving=False),
        # a moving object over a static ground: every one of 128 chirps from its own delays
        dict(name="synth_moving128", kind="synth", scene="ground", dist=2.0, G=700, K=3, tx=3, ns=256, nc=128,
             mode="split", moving=True),
        # the adjoint of a MIMO frame's synthesis (dL/dlength and dL/dA of every path and antenna)
        dict(name="synth_bwd_mimo256", kind="synth_bwd", scene="ground", dist=2.0, G=700, K=3, tx=3, ns=256, nc=128),
        # the point cloud of one long chirp (4096 range cells x 64 angles)
        dict(name="points_range4096", kind="points", array="line", tx=1, ns=4096, nc=1, theta=64, elev=1),
        # the point cloud of the elevated (AWR1843-like) array: 4 x 32 angle rows
        dict(name="points_elevated256", kind="points", array="elevated", tx=3, ns=256, nc=128, theta=32, elev=4),
        # one iteration of mesh reconstruction: 2562-vertex template, 4096 rays
        dict(name="recon_icosphere5k_64", kind="recon", mesh="sphere", tris=5120, G=64, K=2, tx=1, ns=256, nc=1),
        # a reconstruction step of a serving request: 20,000 triangles, half a million rays (an odd grid)
        dict(name="grad_superquadric20k_723", kind="grad", mesh="superquadric", tris=20000, G=723, K=2, tx=1, ns=256,
             nc=1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["calls", "frame", "trace", "synth", "synth", "synth_bwd", "points", "recon", "grad"])
    c = dict(kind=kind)
    if kind in ("calls", "frame", "trace", "grad"):
        top = 1999 if kind == "trace" else 1024
        c.update(mesh=rng.choice(["sphere", "superquadric"]), G=int(_log(rng, 33, top)), K=rng.choice([2, 3]),
                 tx=rng.choice([1, 3]) if kind != "grad" else 1)
        c["tris"] = rng.choice([320, 1280, 5120, 20480]) if c["mesh"] == "sphere" else \
            int(_log(rng, 1000, 200000 if kind == "trace" else 60000))
    if kind == "trace":
        c.update(materials=rng.random() < 0.4, jitter=rng.random() < 0.3)
    if kind in ("calls", "frame", "grad"):
        c.update(ns=rng.choice([128, 256, 512]), nc=rng.choice([1, 16, 128]) if c["tx"] == 3 else 1)
    if kind in ("synth", "synth_bwd"):
        mode = rng.choice(["split", "split", "fp64"]) if kind == "synth" else "split"
        moving = kind == "synth" and mode == "split" and rng.random() < 0.3
        c.update(scene=rng.choice(["sphere", "ground"]), dist=round(rng.uniform(1.0, 20.0), 2), K=2, tx=rng.choice([1, 3]))
        c["ns"] = rng.choice([128, 256, 512] if moving else [64, 128, 256, 512, 1024, 2048, 4096])
        if c["ns"] < 512:
            c["dist"] = round(min(c["dist"], 3.0), 2)
        c["nc"] = rng.choice([1, 16, 128]) if c["ns"] <= 512 else 1
        top = 1023 if mode == "fp64" else 700 if moving or c["tx"] == 3 else 2048
        if c["ns"] > 1024:
            top = min(top, 700)
        c["G"] = int(_log(rng, 33, top))
        if kind == "synth":
            c.update(mode=mode, moving=moving)
    if kind == "points":
        elev = rng.choice([1, 1, 2, 4])
        c.update(array="elevated" if elev > 1 else "line", tx=3 if elev > 1 else rng.choice([1, 3]),
                 ns=rng.choice([64, 128, 256, 512, 1024, 4096]), theta=rng.choice([16, 32, 64]), elev=elev)
        c["nc"] = rng.choice([1, 16, 64, 128]) if c["ns"] <= 512 else 1
    if kind == "recon":
        c.update(mesh="sphere", tris=rng.choice([1280, 5120, 20480]), G=int(_log(rng, 33, 180)), K=2, tx=1,
                 ns=rng.choice([128, 256, 512]), nc=1)
    return c


# ---- inputs -----------------------------------------------------------------


def _radar(c):
    lam = C0 / F0
    if c.get("array") == "elevated":
        tx = np.array([[0, 0, 0], [lam, 0.5 * lam, 0], [2 * lam, 0, 0]], dtype=np.float64)
    else:
        tx = np.array([[2 * lam * t, 0, 0] for t in range(c["tx"])], dtype=np.float64)
    rx = np.array([[0.5 * lam * r, 0, 0] for r in range(4)], dtype=np.float64)
    return SimpleNamespace(f0=F0, bandwidth=BW, chirp_time=TC, chirp_rep=TREP, n_samples=c.get("ns", 256),
                           n_chirps=c.get("nc", 1), n_tx=len(tx), n_rx=4, n_virt=4 * len(tx), tx=tx, rx=rx)


def _cfar(c):
    return SimpleNamespace(n_theta=c.get("theta", 64), guard=2, train=8, alpha=10.0 ** 1.2, floor_rel=1e-4, beta=0.5,
                           w_min=0.01, k_max=2000, n_elev=c.get("elev", 1))


def _grid(center, radius, G, jitter=None):
    """G x G cell-centre (or jittered) directions over the cone from the origin onto a sphere."""
    d = np.asarray(center, dtype=np.float64)
    dist = float(np.linalg.norm(d))
    axis = d / dist
    u = np.cross([0.0, 1.0, 0.0], axis)
    u /= np.linalg.norm(u)
    v = np.cross(axis, u)
    v /= np.linalg.norm(v)
    return SimpleNamespace(G=G, origin=np.zeros(3), axis=axis, u_axis=u, v_axis=v,
                           tan_half=math.tan(math.asin(radius / dist)), jitter=jitter, n_rays=G * G)


@functools.lru_cache(maxsize=8)
def _icosphere(tris):
    t = (1.0 + 5.0 ** 0.5) / 2.0
    verts = np.array([(-1, t, 0), (1, t, 0), (-1, -t, 0), (1, -t, 0), (0, -1, t), (0, 1, t), (0, -1, -t), (0, 1, -t),
                      (t, 0, -1), (t, 0, 1), (-t, 0, -1), (-t, 0, 1)], dtype=np.float64)
    verts /= np.linalg.norm(verts, axis=1, keepdims=True)
    faces = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                      (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5),
                      (2, 4, 11), (6, 2, 10), (8, 6, 7), (9, 8, 1)], dtype=np.int64)
    while len(faces) < tris:
        edges = np.sort(np.concatenate([faces[:, [0, 1]], faces[:, [1, 2]], faces[:, [2, 0]]]), axis=1)
        uniq, inv = np.unique(edges, axis=0, return_inverse=True)
        mid = verts[uniq].sum(1)
        mid /= np.linalg.norm(mid, axis=1, keepdims=True)
        m = len(verts) + inv.reshape(3, -1)
        verts = np.concatenate([verts, mid])
        a, b, d = faces.T
        faces = np.concatenate([np.stack(x, 1) for x in ((a, m[0], m[2]), (b, m[1], m[0]), (d, m[2], m[1]), tuple(m))])
    return verts, faces.astype(np.int32)


def _rotation(rng):
    q = rng.standard_normal(4)
    w, x, y, z = q / np.linalg.norm(q)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                     [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                     [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])


def _superquadric(rng, tris):
    """Seeded superquadric (latitude-longitude mesh with pole fans), about ``tris`` triangles, at 1-3 m."""
    m = max(4, int(round(math.sqrt(tris / 2.0))))
    e1, e2 = rng.uniform(0.3, 2.0, size=2)
    a = rng.uniform(0.1, 0.5, size=3)
    rot, z = _rotation(rng), rng.uniform(1.0, 3.0)
    eta = -0.5 * np.pi + np.pi * np.arange(1, m + 1) / (m + 1)
    om = -np.pi + 2 * np.pi * np.arange(m) / m
    spow = lambda x, e: np.sign(x) * np.abs(x) ** e  # noqa: E731
    ce, se = spow(np.cos(eta), e1)[:, None], spow(np.sin(eta), e1)[:, None]
    ring = np.stack(np.broadcast_arrays(a[0] * ce * spow(np.cos(om), e2), a[1] * ce * spow(np.sin(om), e2), a[2] * se), -1)
    v = np.concatenate([ring.reshape(-1, 3), [[0, 0, -a[2]], [0, 0, a[2]]]]) @ rot.T + [0.0, 0.0, z]
    idx = np.arange(m * m).reshape(m, m)
    nxt = np.roll(idx, -1, axis=1)
    p00, p01, p10, p11 = idx[:-1].ravel(), nxt[:-1].ravel(), idx[1:].ravel(), nxt[1:].ravel()
    S, N = np.full(m, m * m), np.full(m, m * m + 1)
    f = np.concatenate([np.stack([p00, p01, p11, p00, p11, p10], 1).reshape(-1, 3), np.stack([S, nxt[0], idx[0]], 1),
                        np.stack([N, idx[-1], nxt[-1]], 1)])
    return v, f.astype(np.int32)


def _mesh(c, seed):
    """(vertices float32, faces int32, ray grid) of a case's scene."""
    rng = np.random.default_rng([seed, c["tris"], c["G"]])
    if c["mesh"] == "sphere":
        unit, f = _icosphere(c["tris"])
        center = np.array([0.0, 0.0, rng.uniform(0.9, 1.1)])
        v = unit @ _rotation(rng).T * 0.2 * (1 + 0.002 * rng.uniform(-1, 1, (len(unit), 1))) + center
        radius = 0.2
    else:
        v, f = _superquadric(rng, c["tris"])
        lo, hi = v.min(0), v.max(0)
        center = 0.5 * (lo + hi)
        radius = float(np.sqrt(((v - center) ** 2).sum(1)).max())
        g = 2.0 * np.array([[-1, 0, -1], [1, 0, -1], [1, 0, 1], [-1, 0, 1]]) + [center[0], lo[1], center[2]]
        f = np.concatenate([f, np.array([[0, 1, 2], [0, 2, 3]], np.int32) + len(v)])
        v = np.concatenate([v, g])
    jit = rng.random((c["G"] ** 2, 2), dtype=np.float32) if c.get("jitter") else None
    return v.astype(np.float32), f.astype(np.int32), _grid(center, radius, c["G"], jit)


EPS = [4.0 - 0.5j, 9.0 - 2.0j, 0j]  # two lossy dielectrics and a perfect conductor


def _materials(c, seed, nt):
    return np.random.default_rng([seed, 7]).integers(0, len(EPS), nt).astype(np.int32)


def _dirs(grid):
    """Launch directions [R, 3] and solid-angle weights [R] of a grid, FP64 on the device."""
    G = grid.G
    i = torch.arange(G * G, device=DEV)
    row, col = (i // G).to(F64), (i % G).to(F64)
    if grid.jitter is None:
        jx = jy = 0.5
    else:
        j = torch.from_numpy(grid.jitter).to(DEV).to(F64)
        jx, jy = j[:, 0], j[:, 1]
    a, b = grid.tan_half * (2 * (col + jx) / G - 1), grid.tan_half * (2 * (row + jy) / G - 1)
    t = lambda x: torch.from_numpy(np.asarray(x, np.float64)).to(DEV)  # noqa: E731
    w = t(grid.axis) + a[:, None] * t(grid.u_axis) + b[:, None] * t(grid.v_axis)
    inv = 1.0 / w.norm(dim=1)
    return w * inv[:, None], (2 * grid.tan_half / G) ** 2 * inv ** 3


def _paths(c):
    """Paths of a record set: a few less than the scene's rays give, the same number for every seed."""
    return int(c["G"] ** 2 * 0.75)


def _records(c, seed):
    """Path records of a sphere (with ``scene`` "ground" over a 4 x 4 m ground plane) in closed
    form, FP64, in ray order: lengths L [V, P], strengths A [V, P], rates dL/dt [V, P]."""
    rng = np.random.default_rng([seed, c["G"]])
    radar = _radar(c)
    ground = c["scene"] == "ground"
    r = 0.2 if not ground else 0.35
    center = np.array([0.0, 0.0, c["dist"] * (1 + 0.02 * rng.uniform(-1, 1))])
    y0 = -r * rng.uniform(1.0, 1.3)
    grid = _grid(center, r * (1.15 if ground else 1.0), c["G"])
    d, om = _dirs(grid)
    t = lambda x: torch.from_numpy(np.asarray(x, np.float64)).to(DEV)  # noqa: E731
    cen, vel = t(center), t([0.5, 0.0, 2.0 * rng.uniform(0.5, 1.0)])
    zero = torch.zeros_like(d)

    def sphere(o, d):
        oc = o - cen
        b = (oc * d).sum(1)
        disc = b * b - (oc * oc).sum(1) + r * r
        s = -b - disc.clamp_min(0).sqrt()
        return torch.where((disc > 0) & (s > 1e-6), s, torch.full_like(s, math.inf))

    def plane(o, d):
        if not ground:
            return torch.full((len(o),), math.inf, dtype=F64, device=DEV)
        s = (y0 - o[:, 1]) / torch.where(d[:, 1].abs() < 1e-12, torch.full_like(s0, 1e-12), d[:, 1])
        h = o + d * s[:, None]
        ok = (s > 1e-6) & (h[:, 0].abs() < 2) & ((h[:, 2] - center[2]).abs() < 2)
        return torch.where(ok, s, torch.full_like(s, math.inf))

    s0 = torch.zeros(len(d), dtype=F64, device=DEV)
    o = zero
    alive = torch.ones(len(d), dtype=torch.bool, device=DEV)
    interior, sign, rate_in = s0, 1.0, s0
    first = prev = vprev = vfirst = None
    Ls, As, Rs, ok = [], [], [], []
    tx, rx = t(radar.tx), t(radar.rx)
    for k in range(c["K"]):
        ts, tp = sphere(o, d), plane(o, d)
        s = torch.minimum(ts, tp)
        alive = alive & torch.isfinite(s)
        s = torch.where(alive, s, torch.ones_like(s))
        h = o + d * s[:, None]
        on = ts <= tp
        n = torch.where(on[:, None], (h - cen) / r, t([0.0, 1.0, 0.0]))
        v = torch.where(on[:, None], vel, zero)
        if k == 0:
            first, vfirst = h, v
        else:
            leg = (h - prev).norm(dim=1)
            u = (h - prev) / leg[:, None]
            interior = interior + leg
            rate_in = rate_in + (v * u).sum(1) - (vprev * u).sum(1)
        cosv = (d * n).sum(1).abs()
        L, A, R = [], [], []
        for a in tx:
            e = first - a
            lin0 = e.norm(dim=1)
            rt = (vfirst * e).sum(1) / lin0 + rate_in
            for b in rx:
                q = b - h
                lout = q.norm(dim=1)
                lin = lin0 + interior
                L.append(lin + lout)
                A.append(sign * om * cosv / (4 * math.pi * lin * lout))
                R.append(rt - (v * q).sum(1) / lout)
        Ls.append(torch.stack(L))
        As.append(torch.stack(A))
        Rs.append(torch.stack(R))
        ok.append(alive)
        d = d - 2 * (d * n).sum(1, keepdim=True) * n
        o, prev, vprev, sign = h, h, v, -sign
    m = torch.stack(ok, 1).reshape(-1)  # ray-major, bounce-minor
    pick = lambda xs: torch.stack(xs, 2).reshape(radar.n_virt, -1)[:, m][:, :_paths(c)]  # noqa: E731
    return pick(Ls), pick(As), pick(Rs)


def _pack(L, A):
    """The synthesis record of each (antenna, path): phi0, delta_hi, delta_lo, A (float32)."""
    def make(ns):
        phi = F0 / C0 * L
        phi = phi - phi.round()
        dl = BW / (C0 * ns) * L
        dl = dl - dl.round()
        dhi = (dl * 4096).round() / 4096
        return torch.stack([phi, dhi, dl - dhi, A], -1).float()
    return make


def _cube(c, seed):
    """IF cube [V, C, N_s] of clustered point scatterers over a noise floor, complex128."""
    radar = _radar(c)
    g = torch.Generator(device=DEV).manual_seed(seed)
    rnd = lambda *s: torch.rand(*s, generator=g, dtype=F64, device=DEV)  # noqa: E731
    ns, nc, n = radar.n_samples, radar.n_chirps, 120
    rmax = ns * C0 / (2 * BW)
    rng0 = (0.08 + 0.7 * rnd(6, 1)) * rmax + 0.25 * (rnd(6, n // 6) - 0.5)
    u0 = 1.4 * (rnd(6, 1) - 0.5) + 0.25 * (rnd(6, n // 6) - 0.5)
    w0 = 0.8 * (rnd(6, 1) - 0.5) + 0.1 * (rnd(6, n // 6) - 0.5)
    vr, amp = 6 * (rnd(6, 1) - 0.5) + 0 * u0, 1e-3 * (0.1 + rnd(6, n // 6))
    r, u, w, vr, amp = (x.reshape(-1) for x in (rng0, u0, w0, vr, amp))
    lam = C0 / (F0 + BW / 2)
    x = torch.tensor([[a[0] + b[0], a[1] + b[1]] for a in radar.tx for b in radar.rx], dtype=F64, device=DEV)
    e = lambda p: torch.polar(torch.ones_like(p), 2 * math.pi * p)  # noqa: E731
    ant = e(-(x[:, :1] * u + x[:, 1:] * w) / lam)                                      # [V, n]
    sam = e(2 * BW / (C0 * ns) * r[:, None] * torch.arange(ns, device=DEV))            # [n, Ns]
    dop = e(2 * (F0 + BW / 2) / C0 * TREP * vr[:, None] * torch.arange(nc, device=DEV))  # [n, C]
    cube = torch.einsum("vp,pc,pn->vcn", ant * (amp * e(2 * F0 / C0 * r)), dop, sam)
    noise = torch.randn(*cube.shape, 2, generator=g, dtype=F64, device=DEV)
    return cube + 2e-5 * torch.view_as_complex(noise)


# ---- the model in FP64 torch --------------------------------------------------


def _nearest(v, f, o, d, skip):
    """Nearest two-sided hit (triangle or -1) of each ray against every triangle, FP64."""
    a, b, q = v[f[:, 0]], v[f[:, 1]], v[f[:, 2]]
    e1, e2 = b - a, q - a
    N = torch.linalg.cross(e1, e2)
    un_m = torch.cat([e2, -torch.linalg.cross(e2, a)], 1).T.contiguous()   # of (o x d, d)
    vn_m = torch.cat([-e1, -torch.linalg.cross(a, e1)], 1).T.contiguous()
    aN = (a * N).sum(1)
    ids = torch.arange(len(f), device=DEV)
    out = torch.full((len(o),), -1, dtype=torch.int64, device=DEV)
    step = max(1, (1 << 26) // len(f))
    for s in range(0, len(o), step):
        oo, dd = o[s:s + step], d[s:s + step]
        md = torch.cat([torch.linalg.cross(oo, dd), dd], 1)
        det = -(dd @ N.T)
        inv = 1.0 / torch.where(det.abs() < 1e-12, torch.full_like(det, math.nan), det)
        u, w = (md @ un_m).mul_(inv), (md @ vn_m).mul_(inv)
        t = (oo @ N.T).sub_(aN).mul_(inv)
        ok = (u >= 0) & (w >= 0) & (u.add_(w) <= 1) & (t > 1e-9) & (ids != skip[s:s + step, None])
        t = torch.where(ok, t, torch.full_like(t, math.inf))
        best, k = t.min(1)
        out[s:s + step] = torch.where(torch.isfinite(best), k, torch.full_like(k, -1))
    return out


def _hit(v, f, tri, o, d):
    """Plane hit of the given triangles: (t, point, |cos|, reflected direction)."""
    a, b, q = v[f[tri, 0]], v[f[tri, 1]], v[f[tri, 2]]
    N = torch.linalg.cross(b - a, q - a)
    n = N / N.norm(dim=1, keepdim=True)
    den = (N * d).sum(1)
    t = (N * (a - o)).sum(1) / den
    dn = (n * d).sum(1, keepdim=True)
    return t, o + d * t[:, None], dn.abs()[:, 0], d - 2 * dn * n


def _bounces(v, f, grid, K):
    """Triangle sequence [R, K] (-1: none) and distances [R, K] of the specular trace."""
    d, _ = _dirs(grid)
    R = len(d)
    o = torch.zeros_like(d)
    tri = torch.full((R, K), -1, dtype=torch.int64, device=DEV)
    ts = torch.zeros(R, K, dtype=F64, device=DEV)
    live = torch.arange(R, device=DEV)
    skip = torch.full((R,), -1, dtype=torch.int64, device=DEV)
    for k in range(K):
        got = _nearest(v, f, o, d, skip)
        m = got >= 0
        live, o, d, got = live[m], o[m], d[m], got[m]
        t, o, _, d = _hit(v, f, got, o, d)
        tri[live, k], ts[live, k], skip = got, t, got
    return tri, ts


def _lengths(v, f, tri, d, om, radar):
    """Lengths and strengths ([V, P] each) of the rays' paths with the triangles held fixed."""
    tx, rx = (torch.from_numpy(x).to(DEV) for x in (radar.tx, radar.rx))
    o, first, prev = torch.zeros_like(d), None, None
    interior, sign = 0.0, 1.0
    L, A = [], []
    for k in range(tri.shape[1]):
        m = tri[:, k] >= 0
        tri, o, d, om = tri[m], o[m], d[m], om[m]
        _, h, cosv, dn = _hit(v, f, tri[:, k], o, d)
        if k:
            first, prev = first[m], prev[m]
            interior = (interior[m] if k > 1 else 0.0) + (h - prev).norm(dim=1)
        else:
            first = h
        lin = (first[None] - tx[:, None]).norm(dim=2)[:, None] + interior        # [T, 1, P]
        lout = (h[None] - rx[:, None]).norm(dim=2)[None]                         # [1, R, P]
        L.append((lin + lout).flatten(0, 1))
        A.append((sign * om * cosv / (4 * math.pi * lin * lout)).flatten(0, 1))
        o, d, prev, sign = h, dn, h, -sign
    return torch.cat(L, 1), torch.cat(A, 1)


def _polar(x):
    x = 2 * math.pi * (x - x.detach().round())
    return torch.complex(x.cos(), x.sin())


def _sum(phi, delta, A, ns):
    """sum_p A e^{j 2 pi (phi + n delta)}, n < ns, per row of the [V, P] inputs (complex128)."""
    b = 1 << ((ns.bit_length() - 1) // 2)
    na = torch.arange(ns // b, device=DEV, dtype=F64) * b
    nb = torch.arange(b, device=DEV, dtype=F64)
    step = max(1, (1 << 24) // max(b, ns // b))
    rows = []
    for i in range(phi.shape[0]):
        acc = 0
        for s in range(0, phi.shape[1], step):
            p, q, a = phi[i, s:s + step], delta[i, s:s + step], A[i, s:s + step]
            U = _polar(p[:, None] + q[:, None] * na) * a[:, None]
            W = _polar(q[:, None] * nb)
            acc = acc + U.T @ W
        rows.append(acc.reshape(-1))
    return torch.stack(rows)


def _model_cube(v, f, tri, grid, radar):
    d, om = _dirs(grid)
    L, A = _lengths(v, f, tri, d, om, radar)
    return _sum(F0 / C0 * L, BW / (C0 * radar.n_samples) * L, A, radar.n_samples)[:, None].expand(
        -1, radar.n_chirps, -1)


def _power(cube, radar, c):
    """Range-angle power map [angle rows, N_s] of a complex cube [V, C, N_s]."""
    cf = _cfar(c)
    X = torch.fft.fft(torch.fft.fft(cube, dim=2), dim=1)
    lam = C0 / (F0 + BW / 2)
    x = torch.tensor([[a[0] + b[0], a[1] + b[1]] for a in radar.tx for b in radar.rx], dtype=F64, device=DEV)
    u = -1 + 2 * torch.arange(cf.n_theta, device=DEV, dtype=F64) / cf.n_theta
    w = (2 * torch.arange(cf.n_elev, device=DEV, dtype=F64) + 1 - cf.n_elev) / cf.n_elev
    ph = (x[:, 0] * u[None, :, None] + x[:, 1] * w[:, None, None]) / lam
    Y = torch.einsum("rv,vcn->rcn", _polar(ph).reshape(-1, len(x)), X)
    return (Y.real ** 2 + Y.imag ** 2).sum(1)


def _target(c, seed):
    """Target image of a reconstruction: the map of another seeded shape, a 64 x 64 ray sample of it."""
    small = dict(c, G=64, tris=min(c["tris"], 5120))
    v, f, grid = _mesh(small, seed + 1_000_003)
    v, f = torch.from_numpy(v).to(DEV).to(F64), torch.from_numpy(f).to(DEV).long()
    radar = _radar(c)
    tri, _ = _bounces(v, f, grid, c["K"])
    return _power(_model_cube(v, f, tri, grid, radar), radar, c).float()


def _image_grad(c, seed, lap):
    """Image loss (+ lap x uniform Laplacian) and its gradient to the vertices, FP64."""
    vn, fn, grid = _mesh(c, seed)
    v, f = torch.from_numpy(vn).to(DEV).to(F64), torch.from_numpy(fn).to(DEV).long()
    radar, T = _radar(c), _target(c, seed).to(F64)
    tri, _ = _bounces(v, f, grid, c["K"])
    cube = _model_cube(v, f, tri, grid, radar).clone().requires_grad_(True)
    loss = ((_power(cube, radar, c) - T) ** 2).mean()
    loss.backward()
    gsum = cube.grad.sum(1)  # static scene: equal chirps
    v = v.requires_grad_(True)
    d, om = _dirs(grid)
    ns = radar.n_samples
    for s in range(0, len(d), 1 << 15):
        L, A = _lengths(v, f, tri[s:s + (1 << 15)], d[s:s + (1 << 15)], om[s:s + (1 << 15)], radar)
        if L.shape[1]:
            (_sum(F0 / C0 * L, BW / (C0 * ns) * L, A, ns) * gsum.conj()).real.sum().backward()
    total = loss.detach()
    if lap:
        e = torch.cat([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]])
        e = torch.unique(torch.cat([e, e.flip(1)]), dim=0)
        deg = torch.zeros(len(v), dtype=F64, device=DEV).index_add_(0, e[:, 0], torch.ones(len(e), dtype=F64, device=DEV))
        mean = torch.zeros_like(v).index_add(0, e[:, 0], v[e[:, 1]]) / deg[:, None]
        term = lap * ((v - mean) ** 2).sum(1).mean()
        term.backward()
        total = total + term.detach()
    return {"loss": total.reshape(1), "grad": v.grad}


# ---- the cases ------------------------------------------------------------------


def prepare(case, seed):
    c, k = case, case["kind"]
    radar, cfar = _radar(c), _cfar(c)
    s = SimpleNamespace(kind=k, radar=radar, cfar=cfar, c=c)
    if k in ("calls", "frame", "trace", "recon", "grad"):
        vn, fn, s.grid = _mesh(c, seed)
        s.verts, s.faces = torch.from_numpy(vn).to(DEV), torch.from_numpy(fn).to(DEV)
        s.K = c["K"]
    if k in ("calls", "trace"):
        s.scene = sbr.Scene(s.verts, s.faces)
        s.paths = sbr.PathBuffers(s.grid.n_rays, s.K, radar.n_virt)
        s.paths.mem.zero_()  # slots that no path fills read as zero
        if c.get("materials"):
            s.scene.set_materials(EPS, torch.from_numpy(_materials(c, seed, len(fn))).to(DEV))
    if k == "calls":
        s.ws = torch.empty(sbr.synth_ws_bytes(radar, s.paths.cap), dtype=torch.uint8, device=DEV)
        s.cube = torch.empty((radar.n_virt, radar.n_chirps, radar.n_samples, 2), device=DEV)
        s.state = sbr.PcState(radar, cfar)
        s.points = torch.empty((cfar.k_max, 4), device=DEV)
    if k == "frame":
        s.fwd = sbr.Forward(s.verts, s.faces, radar, s.grid, s.K, cfar)
    if k in ("synth", "synth_bwd"):
        L, A, R = _records(c, seed)
        s.P = L.shape[1]
        s.paths = sbr.PathBuffers(c["G"] ** 2, c["K"], radar.n_virt)
        s.paths.mem.zero_()
        s.paths.prep()[:, :s.P] = _pack(L, A)(radar.n_samples)
        hi = L.float()
        raw = torch.stack([hi, (L - hi.to(F64)).float()], -1)
        cap = s.paths.cap
        at = s.paths.s.path_len - s.paths.mem.data_ptr()
        s.paths.mem[at:at + 8 * radar.n_virt * cap].view(torch.float32).view(radar.n_virt, cap, 2)[:, :s.P] = raw
        if c.get("moving"):
            s.paths.path_rate()[:, :s.P] = R.float()
        s.paths.count_tensor().fill_(s.P)
        s.ws = torch.empty(sbr.synth_ws_bytes(radar, cap), dtype=torch.uint8, device=DEV)
        shape = (radar.n_virt, radar.n_chirps, radar.n_samples, 2)
        if k == "synth":
            s.cube = torch.empty(shape, device=DEV)
            s.mode = (sbr.PHASE_FP64 if c["mode"] == "fp64" else sbr.PHASE_SPLIT) | (sbr.SYNTH_MOVING if c["moving"] else 0)
        else:
            s.gcube = _upstream(c, seed)
    if k == "points":
        s.cube = torch.view_as_real(_cube(c, seed)).float().contiguous()
        s.state = sbr.PcState(radar, cfar)
        s.points = torch.empty((cfar.k_max, 4), device=DEV)
    if k == "recon":
        s.rec = Reconstruction(vn, fn, _target(c, seed), radar, s.grid, s.K, cfar, loss="image")
        s.rec.step()
        s.rec.capture()
    if k == "grad":
        s.sim = Simulator(fn, len(vn), radar, s.grid, s.K, cfar)
        s.target = _target(c, seed)
        s.grad = torch.zeros_like(s.verts)
    return s


def _upstream(c, seed):
    """dL/dcube [V, C, N_s, 2]: smooth in range (a few tones) plus noise, as an image loss gives it."""
    radar = _radar(c)
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = torch.arange(radar.n_samples, device=DEV, dtype=F64)
    f, a = (torch.rand(radar.n_virt, radar.n_chirps, 8, generator=g, dtype=F64, device=DEV) for _ in range(2))
    x = torch.einsum("vct,vctn->vcn", a.to(C128), _polar(f[..., None] * n))
    x = x + 0.1 * torch.view_as_complex(torch.randn(*x.shape, 2, generator=g, dtype=F64, device=DEV))
    return torch.view_as_real(x).float().contiguous()


def run(s):
    k = s.kind
    if k == "calls":
        s.scene.update(s.verts)
        sbr.trace(s.scene, s.radar, s.grid, s.K, out=s.paths)
        sbr.synthesize(s.paths, s.radar, out=s.cube, ws=s.ws)
        sbr.pointcloud(s.cube, s.radar, s.cfar, state=s.state, out=s.points)
        return {"cube": s.cube, "power": s.state.power(), "points": s.points, "n": s.state.n_points_tensor()}
    if k == "frame":
        s.fwd.set_vertices(s.verts)
        s.fwd.run()
        return {"cube": s.fwd.cube, "power": s.fwd.state.power(), "points": s.fwd.points,
                "n": s.fwd.state.n_points_tensor()}
    if k == "trace":
        s.scene.update(s.verts)
        p = sbr.trace(s.scene, s.radar, s.grid, s.K, out=s.paths)
        tri, tuv = p.hits()
        return {"tri": tri, "tuv": tuv, "pos": p.hit_pos(), "weight": p.ray_weight(), "first": p.ray_first(),
                "prep": p.prep()}
    if k == "synth":
        return {"cube": sbr.synthesize(s.paths, s.radar, s.mode, out=s.cube, ws=s.ws)}
    if k == "synth_bwd":
        glen, gamp = sbr.synthesize_bwd(s.paths, s.radar, s.gcube, ws=s.ws)
        return {"glen": glen[:, :s.P], "gamp": gamp[:, :s.P]}  # the paths there are: the rest is not written
    if k == "points":
        pts, st = sbr.pointcloud(s.cube, s.radar, s.cfar, state=s.state, out=s.points)
        return {"power": st.power(), "points": pts, "n": st.n_points_tensor()}
    if k == "recon":
        s.rec.verts.copy_(s.verts)
        s.rec.replay()
        return {"loss": s.rec.loss, "grad": s.rec.grad}
    s.grad.zero_()
    s.sim.forward_image(s.verts)
    loss, gcube = sbr.image_loss(s.sim.state, s.target, gcube=s.sim.gcube)
    s.sim.backward_cube(s.verts, gcube, s.grad)
    return {"loss": loss, "grad": s.grad}


def work(case):
    c, k = case, case["kind"]
    V, C, N = 4 * c["tx"], c.get("nc", 1), c.get("ns", 256)
    R, K = c.get("G", 0) ** 2, c.get("K", 1)
    cube = 8 * V * C * N
    cells = c.get("theta", 64) * c.get("elev", 1) * N
    if k in ("synth", "synth_bwd"):
        P = _paths(c)
        rec = 16 * V * P + (4 * V * P if c.get("moving") else 0)
        # at least one phasor and one sum per record (and chirp of a moving scene)
        return {"bytes": rec + cube + (8 * V * P if k == "synth_bwd" else 0),
                "flops": 16.0 * V * P * (C if c.get("moving") else 1)}
    if k == "points":
        return {"bytes": cube + 4 * cells, "flops": 5.0 * V * C * N * math.log2(N * C) + 8.0 * V * C * cells}
    P = 0.6 * R  # about this many paths
    mesh = 18 * c["tris"]
    if k == "trace":
        return {"bytes": mesh + 48 * R * K + 8 * R + 24 * V * P + 8 * P, "flops": 300.0 * R + 100.0 * V * P}
    back = k in ("recon", "grad")
    return {"bytes": mesh * (2 if back else 1) + cube + 4 * cells,
            "flops": (2.0 if back else 1.0) * (300.0 * R + 116.0 * V * P + 5.0 * V * C * N * math.log2(N * C)
                                               + 8.0 * V * C * cells)}


def exact(case, seed):
    c, k = case, case["kind"]
    radar = _radar(c)
    if k in ("recon", "grad"):
        return _image_grad(c, seed, 0.1 if k == "recon" else 0.0)
    if k in ("calls", "frame", "trace"):
        vn, fn, grid = _mesh(c, seed)
        if len(fn) * grid.n_rays * c["K"] > 1e11:
            return None  # a minute and more of brute force
        v, f = torch.from_numpy(vn).to(DEV).to(F64), torch.from_numpy(fn).to(DEV).long()
        tri, ts = _bounces(v, f, grid, c["K"])
        if k == "trace":
            return {"tri": None, "tuv": None, "pos": None, "weight": _dirs(grid)[1], "first": None, "prep": None}
        cube = _model_cube(v, f, tri, grid, radar)
        return {"cube": torch.view_as_real(cube.resolve_conj()).contiguous(), "power": _power(cube, radar, c),
                "points": None, "n": None}
    if k == "points":
        return {"power": _power(torch.view_as_complex(torch.view_as_real(_cube(c, seed)).float().to(F64)), radar, c),
                "points": None, "n": None}
    L, A, R = _records(c, seed)
    rec = _pack(L, A)(radar.n_samples).to(F64)
    phi, delta, A = rec[..., 0], rec[..., 1] + rec[..., 2], rec[..., 3]
    if k == "synth_bwd":
        g = torch.view_as_complex(_upstream(c, seed).to(F64)).sum(1)
        ns = radar.n_samples
        glen, gamp = torch.empty_like(phi), torch.empty_like(phi)
        n = torch.arange(ns, device=DEV, dtype=F64)
        b = 1 << ((ns.bit_length() - 1) // 2)
        na, nb = torch.arange(ns // b, device=DEV, dtype=F64) * b, torch.arange(b, device=DEV, dtype=F64)
        step = (1 << 24) // max(b, ns // b)
        for i in range(len(g)):
            G = torch.stack([g[i].conj(), g[i].conj() * n]).reshape(2, ns // b, b)
            for s in range(0, phi.shape[1], step):
                p, q, a = (x[i, s:s + step] for x in (phi, delta, A))
                U = _polar(p[:, None] + q[:, None] * na)
                W = _polar(q[:, None] * nb)
                s0, s1 = ((U * (W @ x.T)).sum(1) for x in G)
                gamp[i, s:s + step] = s0.real
                # d/dL of the phase 2 pi (f0 / c + n B / (c N_s)) L
                glen[i, s:s + step] = -2 * math.pi * a * (F0 / C0 * s0.imag + BW / (C0 * ns) * s1.imag)
        return {"glen": glen, "gamp": gamp}
    if c["mode"] == "fp64":
        hi = L.float().to(F64)
        L = hi + (L - hi).float().to(F64)
        phi, delta = F0 / C0 * L, BW / (C0 * radar.n_samples) * L
        phi, delta = phi - phi.round(), delta - delta.round()
    if not c["moving"]:
        cube = _sum(phi, delta, A, radar.n_samples)[:, None].expand(-1, radar.n_chirps, -1)
    else:
        R, per = R.float().to(F64), TREP / C0
        cube = torch.stack([_sum(phi + R * (j * per * F0), delta + R * (j * per * BW / radar.n_samples), A,
                                 radar.n_samples) for j in range(radar.n_chirps)], 1)
    return {"cube": torch.view_as_real(cube.resolve_conj()).contiguous()}
