"""Performance cases of the tracker: what a user has it do, through its public entry points.

The work is reconstruction of continuous-readout time frames (Tracker.track,
Tracker.track_batch), the online cluster removal that follows it
(Tracker.cluster_removal), the refit of given tracks and its gradient by the
correction map (Tracker.refit, autograd.refit_chi2) and the allocation-free
neighbour links (tpc_links_noalloc).  Inputs are the synthetic frames of
paper_2601_20569_gb300.synth at sizes from one sector with a few dozen tracks
to a batch of full 2.8 ms frames, strict (deterministic) and fast arithmetic.

A case is a dict of plain values:
  kind      "track", "removal", "refit", "grad" or "links"
  workload  preset of the generator
  clusters  clusters of the call, all frames together
  frames    frames of one batch call (1: Tracker.track)
  fast      arithmetic mode (False: strict)
  graph     the chain is replayed from a captured CUDA graph
  shuffle   clusters in random order instead of by particle
  extras    the chain's optional parts are on (extrapolation, a second seeding
            iteration, edge following, merging across the central electrode)
  map       correction map set (with a distorted workload)
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2601_20569_gb300 import synth, tpc
from paper_2601_20569_gb300.autograd import refit_chi2
from paper_2601_20569_gb300.options import TrackerOptions

# clusters per primary (one_sector, central_event) or collision (the others)
CLUSTERS = {"one_sector": 53.0, "central_event": 155.0, "timeframe": 124e3,
            "timeframe_distorted": 124e3, "stress": 124e3}


def case(kind, workload, clusters, *, frames=1, fast=False, graph=False, shuffle=False,
         extras=False, map=False, name=None):
    c = dict(kind=kind, workload=workload, clusters=int(clusters), frames=frames, fast=fast,
             graph=graph, shuffle=shuffle, extras=extras, map=map)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a real-time loop or an allocator callback asks for the links of one
        # sector (200 tracks): launches and latency only
        case("links", "one_sector", 10575, name="links_one_sector"),
        # the smallest whole call: quality control on one sector, one frame at a
        # time, deterministic mode, as the constructor's defaults have it
        case("track", "one_sector", 3493, name="track_sector_strict"),
        # one central collision of 12,000 primaries, triggered readout: the
        # ordinary single call of an online farm (fast mode, replayed graph)
        case("track", "central_event", 1850000, fast=True, graph=True, name="track_event_fast"),
        # the same kind of event checked bit for bit against the CPU, clusters
        # in arrival order rather than by particle, with the correction map
        case("track", "central_event", 775001, shuffle=True, map=True,
             name="track_event_map_strict"),
        # every optional part of the chain on: the development settings
        case("track", "central_event", 1083333, fast=True, graph=True, extras=True,
             name="track_event_extras_fast"),
        # calibrated running: continuous readout at twice the rate with
        # distortions, a fifth of the tracks loopers
        case("track", "stress", 1300000, fast=True, graph=True, map=True,
             name="track_stress_fast"),
        # reprocessing in the deterministic mode, frame by frame
        case("track", "timeframe", 6000000, name="track_frame_strict"),
        # the production form and the benchmark's: full 2.8 ms frames at 50 kHz
        # (140 collisions each) tracked as one batch
        case("track", "timeframe", 34600000, frames=2, fast=True, graph=True,
             name="track_batch_fast"),
        # cluster reduction after tracking: one event with loopers, one frame
        case("removal", "central_event", 460000, name="removal_event"),
        case("removal", "timeframe", 4000000, fast=True, graph=True, name="removal_frame"),
        # refit of an event's tracks with the present map (deterministic mode)
        case("refit", "central_event", 620000, map=True, name="refit_event_strict"),
        # one step of a map calibration: chi2 of every track forward, its
        # gradient by the map's control points backward
        case("grad", "timeframe_distorted", 1200000, fast=True, map=True,
             name="refit_grad_frame"),
    ]


# per kind and workload: the smallest and the largest number of clusters
RANGES = [
    ("links", "one_sector", 1000, 60000),
    ("track", "one_sector", 1000, 80000),
    ("track", "central_event", 40000, 2100000),
    ("track", "timeframe", 200000, 9000000),
    ("track", "stress", 200000, 1500000),
    ("removal", "central_event", 70000, 1400000),
    ("removal", "timeframe", 200000, 5000000),
    ("refit", "central_event", 40000, 900000),
    ("grad", "central_event", 40000, 900000),
    ("grad", "timeframe_distorted", 200000, 1400000),
]


def draw(rng):
    kind, workload, lo, hi = rng.choice(RANGES)
    c = case(kind, workload, math.exp(rng.uniform(math.log(lo), math.log(hi))))
    c["shuffle"] = rng.random() < 0.25
    c["map"] = kind in ("refit", "grad") or workload == "stress"
    if kind != "links":
        c["fast"] = rng.random() < 0.5
    if kind == "track":
        c["graph"] = rng.random() < 0.5
        c["extras"] = workload != "stress" and rng.random() < 0.2
        if workload == "central_event":
            c["map"] = rng.random() < 0.3
        if workload in ("central_event", "timeframe") and rng.random() < 0.4:
            c["frames"] = rng.randint(2, 4)
    return c


def options(c):
    if c["kind"] == "removal":
        return TrackerOptions(cr_mode=2)
    if c["extras"]:
        return TrackerOptions(ext_rows=20, seed_iters=2, edge_rows=20, ac_merge=1)
    if c["workload"] == "one_sector":
        return TrackerOptions(ms_theta=0.0)  # the preset has no scattering
    return TrackerOptions()


def make_frame(c, seed, n):
    """A frame of n clusters: the generator's, cut after the n-th (5 % of them noise)."""
    w = c["workload"]
    kw = {}
    if c["map"] and w == "central_event":
        kw["distort"] = True
    if c["kind"] == "removal" and w == "central_event":
        kw["looper_frac"] = 0.2
    if c["extras"]:
        kw["vz_sigma"] = 10.0  # vertices along z, so that tracks cross the electrode
    noise = n // 20
    parts, rest, got, have_noise = [], [], 0, 0
    for k in range(100):
        if got >= n - noise and have_noise >= noise:
            break
        size = 1.05 * max(n - noise - got, n // 20) / CLUSTERS[w] / 0.95
        if w in ("one_sector", "central_event"):
            f = synth.generate(w, seed=seed + k, n_primaries=int(size) + 3, **kw)
        else:
            f = synth.generate(w, seed=seed + k, mean_collisions=size + 0.5, **kw)
        m = int(np.count_nonzero(f.label >= 0))  # by particle, then the noise
        use, more = min(m, n - noise - got), min(f.n - m, noise - have_noise)
        for a, b in ((0, use), (m, m + more)):
            (parts if a == 0 else rest).append([v[a:b] for v in (f.y, f.z, f.q, f.row, f.sector)])
        got, have_noise = got + use, have_noise + more
    cols = [np.concatenate([p[i] for p in parts + rest]) for i in range(5)]
    if c["shuffle"]:
        order = np.random.default_rng(seed).permutation(n)
        cols = [a[order] for a in cols]
    return cols, f.map


class State:
    pass


class Result(dict):
    """Views of a tracker's own buffers, with the tracker that they live in."""

    def __init__(self, views, tracker):
        super().__init__(views)
        self.tracker = tracker


def prepare(c, seed):
    s = State()
    s.kind = c["kind"]
    n = c["clusters"]
    share = [n // c["frames"]] * (c["frames"] - 1)
    share.append(n - sum(share))
    frames = [make_frame(c, 1000 * seed + 100 * k, m) for k, m in enumerate(share)]
    s.dev = [tpc.Tracker.to_device(*cols) for cols, _ in frames]
    s.opts = options(c)
    if s.kind == "links":
        return prepare_links(s, n)
    s.tracker = tpc.Tracker(synth.row_x(), s.opts, mode=int(c["fast"]), cap_clusters=max(n, 1024),
                            max_frames=c["frames"], use_graphs=c["graph"])
    if c["map"]:
        s.coeff = torch.as_tensor(frames[0][1]).cuda()
        s.tracker.set_map(s.coeff)
    if s.kind in ("track", "removal"):
        # the tracker's results live until its next call: the user's own copy
        # has room for the tracks of any frame of this size
        nt, f, i = n // 25 + 256, torch.float32, torch.int32
        shapes = {"params": (nt, 5), "cov": (nt, 15), "chi2": (nt,), "x": (nt,), "z_shift": (nt,),
                  "ndf": (nt,), "sector": (nt,), "n_clusters": (nt,), "key": (nt,),
                  "cl_offset": (nt + 1,), "cl_ids": (n + n // 4,)}
        if s.kind == "removal":
            shapes = {"track_class": (nt,), "leg_parent": (nt,)}
        s.own = {k: torch.zeros(v, device="cuda",
                                dtype=f if k in ("params", "cov", "chi2", "x", "z_shift") else i)
                 for k, v in shapes.items()}
    if s.kind != "track":
        s.tracker.track(*s.dev[0])
    if s.kind in ("refit", "grad"):
        # the tracks to refit are those of the tracking, kept by the user
        r = s.tracker.result()
        nt = n // 160
        if nt > r["params"].shape[0]:
            raise RuntimeError(f"{r['params'].shape[0]} tracks found, {nt} wanted")
        s.tracks = {k: r[k][:nt].clone() for k in ("params", "x", "sector")}
        s.tracks["cl_offset"] = r["cl_offset"][:nt + 1].clone()
        s.tracks["cl_ids"] = r["cl_ids"][:int(s.tracks["cl_offset"][-1])].clone()
        g = torch.Generator(device="cuda").manual_seed(seed)
        s.weight = torch.rand(nt, device="cuda", generator=g) + 0.5  # of each track in the loss
        s.coeff.requires_grad_(s.kind == "grad")
    return s


def keep(s, views):
    """The results in the user's buffers (per-cluster arrays are used where they are)."""
    for k, own in s.own.items():
        own[:len(views[k])].copy_(views[k])
    return Result({**views, **s.own}, s.tracker)


def prepare_links(s, n):
    s.lib = tpc.load()
    s.lib.tpc_links_noalloc.argtypes = [
        ctypes.POINTER(tpc.Geometry), ctypes.POINTER(tpc.Options), ctypes.POINTER(tpc.Clusters),
        ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    s.lib.tpc_links_noalloc.restype = ctypes.c_int
    s.row_x = np.ascontiguousarray(synth.row_x())
    s.geo = tpc.Geometry(36, len(s.row_x), s.row_x.ctypes.data)
    s.copt = tpc.make_options(s.opts, mode=0, cap_clusters=max(n, 1))
    y, z, q, row, sector = s.dev[0]
    s.cl = tpc.Clusters(n, y.data_ptr(), z.data_ptr(), q.data_ptr(), row.data_ptr(),
                        sector.data_ptr())
    s.up = torch.empty(n, dtype=torch.int32, device="cuda")
    s.dn = torch.empty(n, dtype=torch.int32, device="cuda")
    return s


def run(s):
    if s.kind == "links":
        rc = s.lib.tpc_links_noalloc(ctypes.byref(s.geo), ctypes.byref(s.copt), ctypes.byref(s.cl),
                                     s.up.data_ptr(), s.dn.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
        if rc:
            raise RuntimeError(f"tpc_links_noalloc: status {rc}")
        return {"up": s.up, "dn": s.dn}
    if s.kind == "track":
        if len(s.dev) > 1:
            s.tracker.track_batch(s.dev)
        else:
            s.tracker.track(*s.dev[0])
        return keep(s, s.tracker.result())
    if s.kind == "removal":
        return keep(s, s.tracker.cluster_removal(s.opts))
    if s.kind == "refit":
        out = s.tracker.refit(s.dev[0], s.tracks, s.coeff)
        # a track that cannot be refitted has no clusters and no parameters
        ok = out["n_clusters"] > 0
        return Result({"chi2": out["chi2"], "n_clusters": out["n_clusters"],
                       "params": torch.where(ok[:, None], out["params"], 0.0),
                       "cov": torch.where(ok[:, None], out["cov"], 0.0),
                       "x": torch.where(ok, out["x"], 0.0)}, s.tracker)
    s.coeff.grad = None
    chi2 = refit_chi2(s.tracker, s.dev[0], s.tracks, s.coeff)
    (s.weight * chi2).sum().backward()
    return {"chi2": chi2.detach(), "grad": s.coeff.grad}


# Kalman steps per cluster: the chain's filter and refit of the tracklet, the
# sector refit's two passes and the fit's three iterations; about 400 floating
# operations each (helix step, covariance transport, update).
STEP_FLOPS = 400.0


def work(c):
    n = float(c["clusters"])
    if c["kind"] == "links":
        # y, z, row, sector read; sorted position, z and id written and read;
        # links written; a few dozen operations per cluster and window
        return {"bytes": n * (10 + 24 + 8), "flops": n * 60.0}
    if c["kind"] == "track":
        # input 12, sorted copy written and read 24, links 16, cleaning 8,
        # attachment 4, cluster reads of the fits 28
        return {"bytes": n * 92.0, "flops": n * 7 * STEP_FLOPS}
    if c["kind"] == "removal":
        # sorted position and id read, flags accumulated, written in input order
        return {"bytes": n * (12 + 4 + 1), "flops": n * 30.0}
    # refit: per cluster of a track its id, y, z, row and sector, and the flags;
    # four filter passes and the map's 3 x 64 spline terms; the gradient replays
    # the three iterations and scatters the 3 x 64 terms
    refs = 0.6 * n
    flops = refs * (4 * STEP_FLOPS + 400.0)
    if c["kind"] == "grad":
        return {"bytes": refs * 2 * 16.0, "flops": 2 * flops}
    return {"bytes": refs * 16.0, "flops": flops}


# --------------------------------------------------------------- 64-bit values
# The refit (and its gradient) in plain torch, 64 bits, all tracks at once: an
# extended Kalman filter outward over the raw clusters, then three linearised
# passes (inward, outward with the two-filter interpolation, inward with the
# cuts) over the corrected clusters.  The tracking itself has no such value: its
# results hang on discrete decisions (links, ownership, mutual best pairs).


def _helix(r, dx, kb):
    """Step of (y, z, sin phi, tan lambda, q/pT) by dx: new state, Jacobian, |sin phi|."""
    y, z, s0, tl, q = r.unbind(1)
    kap = q * kb
    s1 = s0 + kap * dx
    c0, c1 = (1 - s0 * s0).clamp_min(1e-9).sqrt(), (1 - s1 * s1).clamp_min(1e-9).sqrt()
    num, den = s0 + s1, c0 + c1
    t = num / den
    chord = dx * (1 + t * t).sqrt()
    u = 0.5 * kap * chord
    small = u.abs() < 1e-3
    us = torch.where(small, torch.ones_like(u), u.clamp(-0.9999999, 0.9999999))
    au = torch.where(small, 1 + u * u / 6 + 3 * u ** 4 / 40, torch.asin(us) / us)
    b = 1 / (1 - (u * u).clamp_max(0.9999999)).sqrt()
    # derivative of asin(u)/u
    da = torch.where(small, u / 3 + 0.3 * u ** 3, (b - torch.asin(us) / us) / us)
    new = torch.stack([y + dx * t, z + tl * chord * au, s1, tl, q], 1)
    dt_ds = (2 * den + num * (s0 / c0 + s1 / c1)) / den ** 2
    dt_dk = dx * (den + num * s1 / c1) / den ** 2
    g = dx * t / (1 + t * t).sqrt()
    f = torch.eye(5, dtype=r.dtype, device=r.device).repeat(r.shape[0], 1, 1)
    f[:, 0, 2] = dx * dt_ds
    f[:, 0, 4] = dx * dt_dk * kb
    f[:, 1, 2] = tl * g * dt_ds * b
    f[:, 1, 3] = chord * au
    f[:, 1, 4] = tl * (g * dt_dk * b + 0.5 * chord ** 2 * da) * kb
    f[:, 2, 4] = dx * kb
    return new, f, s1.abs()


class _Fit:
    """One block of tracks: padded station lists and the filter's pieces."""

    def __init__(self, cl, tracks, lo, hi, coeff, o, row_x):
        y, z, row, sector = cl
        off = tracks["cl_offset"].long()
        d = dict(dtype=torch.float64, device=y.device)
        self.n = off[lo + 1:hi + 1] - off[lo:hi]
        S = int(self.n.max())
        k = torch.arange(S, device=y.device)
        self.have = k[None] < self.n[:, None]
        at = (off[lo:hi, None] + k).clamp_max(len(tracks["cl_ids"]) - 1)
        ids = tracks["cl_ids"][at].long()
        self.y, self.z = y[ids].double(), z[ids].double()
        self.sec = sector[ids].long()
        self.x = torch.as_tensor(row_x, **d)[row[ids].long()]
        self.p0 = tracks["params"][lo:hi].double()
        self.x0 = tracks["x"][lo:hi].double()
        self.s0 = tracks["sector"][lo:hi].long()
        self.z0 = self.p0[:, 1] - self.p0[:, 3] * (self.x0 ** 2 + self.p0[:, 0] ** 2).sqrt()
        self.o, self.kb = o, -o.bz * 0.00299792458
        self.pitch = (row_x[-1] - row_x[0]) / (len(row_x) - 1)
        self.seed = torch.diag(torch.tensor(o.seed_c, **d))
        self.noise = torch.diag(torch.tensor([o.sigma_y ** 2, o.sigma_z ** 2], **d))
        self.D = self.correction(coeff.double())

    def correction(self, c):
        """The cubic B-spline map at every cluster."""
        ncomp, nz, nr, nphi = c.shape

        def span(t, n):
            t = t.clamp(0, n - 3)
            i = t.floor().clamp_max(n - 4)
            return i.long(), t - i

        def weights(f):
            return torch.stack([(1 - f) ** 3 / 6, (3 * f ** 3 - 6 * f ** 2 + 4) / 6,
                                (-3 * f ** 3 + 3 * f ** 2 + 3 * f + 1) / 6, f ** 3 / 6], -1)

        m = self.have
        x, y, z = self.x[m], self.y[m], (self.z - self.z0[:, None])[m]
        half = math.tan(math.radians(10.0))
        tp = (self.sec[m] % 18 + 0.5 + 0.5 * (y / x) / half) * (nphi / 18) - 0.5
        ip = tp.floor()
        r0, r1 = synth.MAP_R
        ir, fr = span(((x * x + y * y).sqrt() - r0) * ((nr - 3) / (r1 - r0)), nr)
        z0, z1 = synth.MAP_Z
        iz, fz = span((z.clamp(z0, z1) - z0) * ((nz - 3) / (z1 - z0)), nz)
        wp, wr, wz = weights(tp - ip), weights(fr), weights(fz)
        e = torch.arange(4, device=c.device)
        jp = (ip.long()[:, None] - 1 + e) % nphi
        cell = ((iz[:, None] + e)[:, :, None, None] * nr + (ir[:, None] + e)[:, None, :, None]) \
            * nphi + jp[:, None, None, :]
        w = wz[:, :, None, None] * wr[:, None, :, None] * wp[:, None, None, :]
        flat = c.reshape(ncomp, -1)
        D = torch.stack([(flat[i][cell] * w).sum((1, 2, 3)) for i in range(ncomp)], 1)
        full = torch.zeros(*m.shape, 3, dtype=c.dtype, device=c.device)
        return full.index_put((m.nonzero()[:, 0], m.nonzero()[:, 1]), D)

    def scatter_noise(self, C, s, tl, dx):
        th2 = self.o.ms_theta ** 2 * dx.abs() / self.pitch
        a = 1 + tl * tl
        C[:, 2, 2] += th2 * (1 - s * s) * a
        C[:, 3, 3] += th2 * a * a

    def turn(self, r, x, sec, to):
        """Rotation of state r at x into the sector `to` (where it differs)."""
        ds = (to % 18 - sec % 18 + 18) % 18
        ok = (ds == 0) | (ds == 1) | (ds == 17)
        ang = torch.where(ds == 1, 20.0, torch.where(ds == 17, -20.0, 0.0)).double()
        ca, sa = torch.cos(torch.deg2rad(ang)), torch.sin(torch.deg2rad(ang))
        y, z, s, tl, q = r.unbind(1)
        c = (1 - s * s).clamp_min(1e-9).sqrt()
        xn, yn = x * ca + y * sa, y * ca - x * sa
        sn, cn = s * ca - c * sa, c * ca + s * sa
        ok = ok & (cn > 0) & (sn.abs() < self.o.fit_max_snp)
        cn = cn.clamp_min(1e-9)
        J = torch.eye(5, dtype=r.dtype, device=r.device).repeat(r.shape[0], 1, 1)
        J[:, 0, 0] = c / cn
        J[:, 1, 0] = -sa * tl / cn
        J[:, 2, 0] = -sa * q * self.kb
        J[:, 2, 2] = cn / c
        return torch.stack([yn, z, sn, tl, q], 1), xn, J, ok

    def gain(self, C):
        return C[:, :, :2] @ torch.linalg.inv(C[:, :2, :2] + self.noise)

    def start(self):
        """The outward extended Kalman pass over the raw clusters."""
        p, x, sec = self.p0.clone(), self.x0.clone(), self.s0.clone()
        C = self.seed.repeat(len(p), 1, 1)
        alive = self.n > 0
        for k in range(self.y.shape[1]):
            do = alive & self.have[:, k]
            q, xq, J, ok1 = self.turn(p, x, sec, self.sec[:, k])
            dx = self.x[:, k] - xq
            q, F, s = _helix(q, dx, self.kb)
            F = F @ J
            Cq = F @ C @ F.mT
            self.scatter_noise(Cq, q[:, 2], q[:, 3], dx)
            K = self.gain(Cq)
            m = torch.stack([self.y[:, k], self.z[:, k]], 1) - q[:, :2]
            alive = alive & ~(do & ~(ok1 & (s < self.o.fit_max_snp)))
            do = do & alive
            p = torch.where(do[:, None], q + (K @ m[:, :, None])[:, :, 0], p)
            C = torch.where(do[:, None, None], Cq - K @ Cq[:, :2, :], C)
            x = torch.where(do, self.x[:, k], x)
            sec = torch.where(do, self.sec[:, k], sec)
        return p, x, alive

    def sweep(self, it, p, ref, x, alive, stored, flag):
        """Iteration it (0 inward, 1 outward, 2 inward with cuts) about ref."""
        S, o = self.y.shape[1], self.o
        T = len(p)
        rows = torch.arange(T, device=p.device)
        C = self.seed.repeat(T, 1, 1)
        chi2 = torch.zeros(T, dtype=p.dtype, device=p.device)
        nused = torch.zeros(T, dtype=torch.long, device=p.device)
        outp, outx, outC = p.detach().clone(), x.clone(), C.clone()
        go = alive.clone()  # iteration 3 stops a track without failing it
        sec = None
        for j in range(S):
            k = torch.full((T,), j, device=p.device) if it == 1 else (self.n - 1 - j)
            here = (k >= 0) & (j < self.n)
            k = k.clamp_min(0)
            to = self.sec[rows, k]
            X = self.x[rows, k]
            do = go & here
            with torch.no_grad():
                if j == 0:
                    q, F = ref.clone(), torch.eye(5, dtype=p.dtype, device=p.device).repeat(T, 1, 1)
                    Cq, okm = C, torch.ones_like(go)
                else:
                    q, xq, J, ok1 = self.turn(ref, x, sec, to)
                    dx = X - xq
                    q, F, s = _helix(q, dx, self.kb)
                    F = F @ J
                    Cq = F @ C @ F.mT
                    self.scatter_noise(Cq, q[:, 2], q[:, 3], dx)
                    okm = ok1 & (s < o.fit_max_snp)
                bad = do & ~okm
                go = go & ~bad
                if it < 2:
                    alive = alive & ~bad
                do = do & go
                at_x = x if j == 0 else X
            pq = q + (F @ (p - ref)[:, :, None])[:, :, 0]
            # corrected cluster, moved back to the pad row along the reference
            D = self.D[rows, k]
            h, _, hs = _helix(q, D[:, 0], self.kb)
            m = torch.stack([self.y[rows, k] + D[:, 1] - (h[:, 0] - q[:, 0]),
                             self.z[rows, k] + D[:, 2] - (h[:, 1] - q[:, 1])], 1)
            with torch.no_grad():
                okh = hs < o.fit_max_snp
                if it < 2:
                    bad = do & ~okh
                    go, alive = go & ~bad, alive & ~bad
                    do = do & go
                if it == 0:
                    stored[0][rows[do], k[do]] = pq.detach()[do, :2]
                    stored[1][rows[do], k[do]] = Cq[do][:, :2, :2]
                use = do
                if it == 1:
                    W = torch.linalg.inv(Cq[:, :2, :2])
                    sc = stored[1][rows, k]
                    sc = torch.where(do[:, None, None], sc, self.noise)
                    V = torch.linalg.inv(sc)
                    I = torch.linalg.inv(W + V)
                    pos = I @ (W @ pq.detach()[:, :2, None] +
                               V @ stored[0][rows, k][:, :, None])
                    res = m.detach() - pos[:, :, 0]
                    c2 = (res[:, None] @ torch.linalg.inv(I + self.noise) @ res[:, :, None])[:, 0, 0]
                    flag[rows[do], k[do]] = (c2 > o.int_chi2)[do]
                if it == 2:
                    use = do & ~flag[rows, k] & okh
                Winv = torch.linalg.inv(Cq[:, :2, :2] + self.noise)
                K = Cq[:, :, :2] @ Winv
            res = m - pq[:, :2]
            if it == 2:
                c2 = (res[:, None] @ Winv @ res[:, :, None])[:, 0, 0]
                use = use & (c2.detach() <= o.final_chi2)
                chi2 = chi2 + torch.where(use, c2, torch.zeros_like(c2))
                nused += use
            pu = torch.where(use[:, None], pq + (K @ res[:, :, None])[:, :, 0], pq)
            p = torch.where(do[:, None], pu, p)
            with torch.no_grad():
                Cu = torch.where(use[:, None, None], Cq - K @ Cq[:, :2, :], Cq)
                C = torch.where(do[:, None, None], Cu, C)
                ref = torch.where(do[:, None], q, ref)
                x = torch.where(do, at_x, x)
                sec = to.clone() if sec is None else torch.where(do, to, sec)
                if it == 2:
                    outp = torch.where(use[:, None], p.detach(), outp)
                    outx = torch.where(use, x, outx)
                    outC = torch.where(use[:, None, None], C, outC)
        return p, x, alive, chi2, nused, outp, outx, outC

    def fit(self):
        p, x, alive = self.start()
        T, S = self.y.shape
        stored = (torch.zeros(T, S, 2, dtype=p.dtype, device=p.device),
                  self.noise.repeat(T, S, 1, 1))
        flag = torch.zeros(T, S, dtype=torch.bool, device=p.device)
        for it in range(3):
            p, x, alive, chi2, n, op, ox, oc = self.sweep(it, p, p.detach(), x, alive, stored, flag)
        i, j = np.tril_indices(5)
        ok = alive & (n > 0)
        zero = torch.zeros((), dtype=p.dtype, device=p.device)
        return {"chi2": torch.where(alive, chi2, zero), "params": torch.where(ok[:, None], op, zero),
                "cov": torch.where(ok[:, None], oc[:, i, j], zero), "x": torch.where(ok, ox, zero)}


def exact(c, seed):
    if c["kind"] not in ("refit", "grad"):
        return None
    s = prepare(c, seed)  # the clusters, tracks, weights and map of the case
    y, z, _, row, sector = s.dev[0]
    coeff = s.coeff.detach().double().requires_grad_(c["kind"] == "grad")
    nt = int(s.tracks["params"].shape[0])
    step = 8192
    outs, grad = [], torch.zeros_like(coeff)
    for lo in range(0, nt, step):
        hi = min(nt, lo + step)
        with torch.set_grad_enabled(c["kind"] == "grad"):
            fit = _Fit((y, z, row, sector), s.tracks, lo, hi, coeff, s.opts,
                       synth.row_x().astype(np.float64))
            out = fit.fit()
        if c["kind"] == "grad":
            loss = (s.weight[lo:hi].double() * out["chi2"]).sum()
            grad = grad + torch.autograd.grad(loss, coeff)[0]
        outs.append({k: v.detach() for k, v in out.items()})
    whole = {k: torch.cat([o[k] for o in outs]) for k in outs[0]}
    if c["kind"] == "grad":
        return {"chi2": whole["chi2"], "grad": grad.detach()}
    return dict(whole, n_clusters=None)
