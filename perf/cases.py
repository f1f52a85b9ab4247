"""Performance cases of the track fit, the hit binning, the combinatorial
build, the re-fit and the serving loop, each through the binding
(paper_1605_05508_gb300.kf) as a program that reconstructs events calls it.

The inputs are simplified barrel events (uniform field, concentric
cylinders, smeared hits, uniform noise), drawn on the GPU in double precision
from the seed alone and rounded to float32 once.  `exact` is a plain
double-precision torch rendering of the same filter.
"""
import math

import numpy as np
import torch

from paper_1605_05508_gb300 import kf

C_LIGHT = 0.00299792458  # GeV / (T cm)
BZ, SIGMA_XY, SIGMA_Z = 3.8, 0.01, 0.1
MASS = kf.PION_MASS
CHI2_CUT = 30.0
DEV = "cuda"
TRIL_I, TRIL_J = np.tril_indices(6)  # packed lower triangle, row-major


def f32(v):
    return float(np.float32(v))


# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # One small event (1 000 tracks, 10 layers): a trigger-like caller that fits event by event, where
        # latency and launches count.
        dict(name="fit_event_small", kind="fit", n=1000, layers=10, lo=False, ineff=0.0, x_x0=0.0, pt="std"),
        # The same event fitted in double precision, the form that validation runs use.
        dict(name="fit_event_f64", kind="fit64", n=1000, events=1, layers=10),
        # One full event of about 20 000 tracks with detector material (3 % of a radiation length a layer) and
        # 2 % missing hits: the ordinary single-event fit, an odd size.
        dict(name="fit_event_material", kind="fit", n=19997, layers=10, lo=True, ineff=0.02, x_x0=0.03, pt="std"),
        # 200 events of 20 000 tracks in one call: the batch fit of an offline pass, the largest call.
        dict(name="fit_batch", kind="fit", n=4000000, layers=10, lo=True, ineff=0.0, x_x0=0.0, pt="std"),
        # A million tracks over 20 layers, half of them below 1 GeV (curling up before the outer layers) and
        # half 10 - 100 GeV: long tracks of very different curvature.
        dict(name="fit_long_mix", kind="fit", n=1000003, layers=20, lo=True, ineff=0.0, x_x0=0.0, pt="mix"),
        # 25 events of 20 000 tracks held in pinned host memory: a caller whose data lives on the host.
        dict(name="fit_host", kind="host", n=500000, layers=10),
        # The hits of one 20 000-hits-a-layer event sorted into bins (default, ordered form).
        dict(name="bin_event", kind="bin", events=1, layers=7, hits=20000, ragged=False),
        # The hits of 50 events sorted into bins (default, ordered form).
        dict(name="bin_batch", kind="bin", events=50, layers=7, hits=20000, ragged=False),
        # One event of 5 000 seeds reconstructed with the default settings: seed fit, binning, clone-engine
        # build with 6 candidates a seed; event-by-event reconstruction.
        dict(name="reco_event", kind="reco", events=1, seeds=5000, ragged=False, cands=6, noise=3.0, fine=False,
             refit=False, x_x0=0.0),
        # 50 events of 5 000 seeds at once, seed fit and binning on two streams, unordered binning with the
        # sub-bin look-up: the throughput form of the same reconstruction.
        dict(name="reco_batch", kind="reco", events=50, seeds=5000, ragged=False, cands=6, noise=3.0, fine=True,
             refit=False, x_x0=0.0),
        # 12 events of very uneven size (500 - 50 000 tracks), best-hit building (1 candidate), then the
        # re-fit of the built tracks over all layers.
        dict(name="reco_ragged_refit", kind="reco", events=12, seeds=5000, ragged=True, cands=1, noise=3.0,
             fine=False, refit=True, x_x0=0.0),
        # Serving: 10 requests of uneven size submitted back to back from one thread and collected.
        dict(name="serve_burst", kind="serve", events=10, seeds=5000, cands=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "host", "fit64", "bin", "reco", "reco", "reco", "serve"])
    if kind == "fit":
        layers = rng.choice([7, 10, 10, 13, 20])
        return dict(kind=kind, n=_log_int(rng, 200, 40000000 // layers), layers=layers, lo=rng.random() < 0.7,
                    ineff=rng.choice([0.0, 0.02, 0.1]), x_x0=rng.choice([0.0, 0.0, 0.03]),
                    pt=rng.choice(["std", "mix"]))
    if kind == "host":
        return dict(kind=kind, n=_log_int(rng, 5000, 1500000), layers=rng.choice([7, 10, 12]))
    if kind == "fit64":
        events = rng.randint(1, 4)
        return dict(kind=kind, n=_log_int(rng, 200, 10000), events=events, layers=10)
    if kind == "bin":
        return dict(kind=kind, events=_log_int(rng, 1, 50), layers=rng.choice([5, 7]), hits=_log_int(rng, 300, 30000),
                    ragged=rng.random() < 0.5)
    if kind == "reco":
        fine = rng.random() < 0.5
        return dict(kind=kind, events=_log_int(rng, 1, 30), seeds=_log_int(rng, 300, 8000), ragged=rng.random() < 0.5,
                    cands=rng.choice([1, 2, 3, 4, 6, 8]), noise=rng.choice([1.0, 3.0, 5.0]), fine=fine,
                    refit=rng.random() < 0.4, x_x0=rng.choice([0.0, 0.0, 0.02]))
    return dict(kind=kind, events=rng.randint(3, 10), seeds=_log_int(rng, 1000, 5000), cands=rng.choice([1, 3, 6]))


# --------------------------------------------------------------------------- generating the inputs


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rand(g, n, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _particles(g, n, pt="std"):
    q = torch.where(_rand(g, n) < 0.5, 1.0, -1.0).double()
    if pt == "std":
        p_t = _rand(g, n, 0.5, 10.0)
    else:
        p_t = torch.where(_rand(g, n) < 0.5, _rand(g, n, 0.2, 1.0), _rand(g, n, 10.0, 100.0))
    phi, eta = _rand(g, n, 0.0, 2.0 * math.pi), _rand(g, n, -1.0, 1.0)
    vtx = _randn(g, 3, n) * torch.tensor([[0.01], [0.01], [1.0]], device=DEV, dtype=torch.float64)
    return q, torch.cat([vtx, torch.stack([p_t * torch.cos(phi), p_t * torch.sin(phi), p_t * torch.sinh(eta)])])


def _cross(st, a, R):
    """State [6, n] on the first outward crossing of the cylinder r = R (a = q c Bz signed), the path length
    and whether it is reached: the circle-circle intersection, polished by Newton steps on the path length."""
    x, y, z, px, py, pz = st
    pt = torch.hypot(px, py)
    p = torch.hypot(pt, pz)
    rho = pt / a.abs()
    cx, cy = x + py / a, y - px / a
    d = torch.hypot(cx, cy)
    cosang = (R * R - d * d - rho * rho) / (2.0 * rho * d)
    ok = cosang.abs() <= 1.0
    alpha, psi_c, psi_0 = torch.acos(cosang.clamp(-1.0, 1.0)), torch.atan2(cy, cx), torch.atan2(y - cy, x - cx)
    turn = torch.full_like(x, math.inf)
    for sgn in (1.0, -1.0):
        t = torch.where(a > 0, psi_0 - (psi_c + sgn * alpha), (psi_c + sgn * alpha) - psi_0)
        turn = torch.minimum(turn, torch.remainder(t, 2.0 * math.pi))
    s = turn * p / a.abs()

    def at(s):
        th = a * s / p
        sa, ca = torch.sin(th) / a, 2.0 * torch.sin(0.5 * th) ** 2 / a
        dx, dy = px * sa + py * ca, py * sa - px * ca
        c, sn = torch.cos(th), torch.sin(th)
        return th, sa, ca, dx, dy, px * c + py * sn, py * c - px * sn, c, sn
    for _ in range(3):
        _, _, _, dx, dy, PX, PY, _, _ = at(s)
        g = (x * x + y * y - R * R) + 2.0 * (x * dx + y * dy) + dx * dx + dy * dy
        dg = 2.0 * ((x + dx) * PX + (y + dy) * PY) / p
        s = torch.where(dg.abs() > 1e-3, s - g / dg, s)
    th, sa, ca, dx, dy, PX, PY, c, sn = at(s)
    X, Y = x + dx, y + dy
    rp = X * PX + Y * PY
    ok = ok & (rp > 0) & (s > 0)
    return torch.stack([X, Y, z + pz * s / p, PX, PY, pz]), ok, (s, p, pt, th, sa, ca, c, sn, rp)


def _theta2(p2, xe):
    """Highland angle squared for a unit-charge pion of squared momentum p2 over xe radiation lengths."""
    m = f32(MASS)
    e2 = p2 + m * m
    return 0.0136 ** 2 * e2 / (p2 * p2) * xe * (1.0 + 0.038 * torch.log(xe * e2 / p2)) ** 2


def _kink(g, st, x_x0):
    pos, mom = st[:3], st[3:]
    p = mom.norm(dim=0)
    d = mom / p
    cos_inc = ((pos[0] * d[0] + pos[1] * d[1]).abs() / torch.hypot(pos[0], pos[1])).clamp_min(1e-6)
    th0 = _theta2(p * p, x_x0 / cos_inc).sqrt()
    u1 = torch.stack([-d[1], d[0], torch.zeros_like(p)])
    u1 = u1 / u1.norm(dim=0)
    u2 = torch.linalg.cross(d, u1, dim=0)
    k = _randn(g, 2, p.numel()) * th0
    d = d + torch.tan(k[0]) * u1 + torch.tan(k[1]) * u2
    return torch.cat([pos, d / d.norm(dim=0) * p])


def _hits(g, q, truth, radii, x_x0, ineff):
    """Smeared hits [L, 3, n] float32 and their valid flags: on every layer up to the last one reached."""
    n = q.numel()
    a = q * (C_LIGHT * BZ)
    sig = torch.tensor([[SIGMA_XY], [SIGMA_XY], [SIGMA_Z]], device=DEV, dtype=torch.float64)
    alive = torch.ones(n, dtype=torch.bool, device=DEV)
    xyz = torch.zeros((len(radii), 3, n), device=DEV)
    valid = torch.zeros((len(radii), n), dtype=torch.uint8, device=DEV)
    st = truth
    for l, R in enumerate(radii):
        nx, ok, _ = _cross(st, a, R)
        alive = alive & ok
        xyz[l] = torch.where(alive, nx[:3] + sig * _randn(g, 3, n), torch.zeros_like(nx[:3])).float()
        valid[l] = alive & (_rand(g, n) >= ineff) if ineff else alive
        if x_x0:
            st = torch.where(alive, _kink(g, nx, x_x0), st)
    return xyz, valid


def _vertex_seeds(g, q, truth):
    """Seeds: the vertex state smeared by the stated diagonal covariance."""
    n = q.numel()
    p = truth[3:].norm(dim=0)
    sd = torch.cat([torch.tensor([[0.01], [0.01], [1.0]], device=DEV, dtype=torch.float64).expand(3, n),
                    (0.01 * p).expand(3, n)])
    cov = torch.zeros((21, n), device=DEV)
    for i in range(6):
        cov[i * (i + 1) // 2 + i] = (sd[i] ** 2).float()
    return (truth + sd * _randn(g, 6, n)).float(), cov, q.to(torch.int8)


def _radii(layers):
    return [4.0 * (i + 1) for i in range(layers)]


def _fit_inputs(case, seed):
    g = _gen(seed)
    n, L = case["n"], case["layers"]
    parts = []
    for b in range(0, n, 1 << 20):  # bounded scratch
        q, truth = _particles(g, min(1 << 20, n - b), case.get("pt", "std"))
        parts.append((*_vertex_seeds(g, q, truth),
                      *_hits(g, q, truth, _radii(L), case.get("x_x0", 0.0), case.get("ineff", 0.0))))
    return tuple(torch.cat(t, dim=-1).contiguous() if len(parts) > 1 else t[0].contiguous() for t in zip(*parts))


def _event_sizes(case):
    """Tracks of each event: the stated number, or spread evenly over the logarithm of 500 .. 50 000 (scaled
    with the stated number) in a shuffled order."""
    E, n = case["events"], case["seeds"]
    if not case.get("ragged", True):
        return [n] * E
    f = (np.arange(E) + 0.5) / E
    sizes = np.exp(np.log(n / 10.0) + f * math.log(100.0)).round().astype(int)
    return [int(s) for s in np.random.default_rng(E).permutation(sizes)]


N_SEED_LAYERS, N_BUILD_LAYERS = 3, 7


def _reco_inputs(case, seed):
    """Vertex seeds and seeding-layer hits of every event, and the raw hits (track hits and uniform noise, in
    random order) of every (event, building layer) segment."""
    g = _gen(seed)
    sizes = _event_sizes(case)
    radii = _radii(N_SEED_LAYERS + N_BUILD_LAYERS)
    x_x0 = case.get("x_x0", 0.0)
    n = sum(sizes)
    q, truth = _particles(g, n)
    par, cov, charge = _vertex_seeds(g, q, truth)
    xyz, valid = _hits(g, q, truth, radii, x_x0, 0.0)
    segs, offs, b = [], [0], 0
    for s in sizes:
        n_noise = int(round(case.get("noise", 3.0) * s))
        for l in range(N_SEED_LAYERS, len(radii)):
            R = radii[l]
            trk = xyz[l, :, b:b + s][:, valid[l, b:b + s] != 0]
            phi, zmax = _rand(g, n_noise, 0.0, 2.0 * math.pi), R * math.sinh(1.0) + 3.0
            sm = _randn(g, 3, n_noise)
            nz = torch.stack([R * torch.cos(phi) + SIGMA_XY * sm[0], R * torch.sin(phi) + SIGMA_XY * sm[1],
                              _rand(g, n_noise, -zmax, zmax) + SIGMA_Z * sm[2]]).float()
            h = torch.cat([trk, nz], dim=1)
            h = h[:, torch.randperm(h.shape[1], generator=g, device=DEV)]
            segs.append(h)
            offs.append(offs[-1] + h.shape[1])
        b += s
    return dict(sizes=sizes, par=par, cov=cov, charge=charge, xyz=xyz[:N_SEED_LAYERS].contiguous(),
                valid=valid[:N_SEED_LAYERS].contiguous(), hits=torch.cat(segs, dim=1).contiguous(), offs=offs)


def _bin_inputs(case, seed):
    g = _gen(seed)
    E, L, n = case["events"], case["layers"], case["hits"]
    radii = _radii(N_SEED_LAYERS + L)[N_SEED_LAYERS:]
    per = [n] * E
    if case["ragged"]:
        f = (np.arange(E) + 0.5) / E
        per = [max(1, int(v)) for v in np.exp(np.log(n) + (f - 1.0) * math.log(30.0))]
        per = [int(v) for v in np.random.default_rng(E).permutation(per)]
    offs = [0]
    for m in per:
        for _ in range(L):
            offs.append(offs[-1] + m)
    R = torch.tensor(radii, device=DEV, dtype=torch.float64).repeat(E).repeat_interleave(
        torch.tensor([m for m in per for _ in range(L)], device=DEV))
    n_hits = offs[-1]
    phi = _rand(g, n_hits, 0.0, 2.0 * math.pi)
    track = _rand(g, n_hits) < 0.25  # track hits are uniform in eta, the noise in z
    z = torch.where(track, R * torch.sinh(_rand(g, n_hits, -1.0, 1.0)) + _randn(g, n_hits),
                    _rand(g, n_hits, -1.0, 1.0) * (R * math.sinh(1.0) + 3.0))
    sm = _randn(g, 3, n_hits)
    return torch.stack([R * torch.cos(phi) + SIGMA_XY * sm[0], R * torch.sin(phi) + SIGMA_XY * sm[1],
                        z + SIGMA_Z * sm[2]]).float().contiguous(), offs


# --------------------------------------------------------------------------- prepare and run


def _context(layers, x_x0=0.0, **kw):
    return kf.Context(_radii(layers), BZ, SIGMA_XY, SIGMA_Z, CHI2_CUT, x_x0=[x_x0] * layers if x_x0 else None, **kw)


def _empty(*shape, dtype=torch.float32):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _out_tracks(n, charge, lo=True, dtype=torch.float32):
    return kf.Tracks(_empty(6, n, dtype=dtype), _empty(21, n, dtype=dtype), charge, _empty(3, n) if lo else None)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "fit":
        par, cov, q, xyz, valid = _fit_inputs(case, seed)
        L, n = xyz.shape[0], xyz.shape[2]
        st.update(ctx=_context(L, case["x_x0"]), seeds=kf.Tracks(par, cov, q), hits=kf.TrackHits(xyz, valid),
                  out=_out_tracks(n, q, case["lo"]), chi2=_empty(L, n), status=_empty(n, dtype=torch.int32))
    elif kind == "fit64":
        par, cov, q, xyz, valid = _fit_inputs(case, seed)
        L, n = xyz.shape[0], xyz.shape[2]
        off = [n * e // case["events"] for e in range(case["events"] + 1)]
        st.update(ctx=_context(L), seeds=kf.Tracks(par.double(), cov.double(), q), hits=kf.TrackHits(xyz, valid),
                  out=_out_tracks(n, q, False, torch.float64), off=off, chi2=_empty(L, n, dtype=torch.float64),
                  status=_empty(n, dtype=torch.int32))
    elif kind == "host":
        par, cov, q, xyz, valid = _fit_inputs(case, seed)
        L, n = xyz.shape[0], xyz.shape[2]

        def pin(t):
            return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)

        def host(*shape, dtype=torch.float32):
            return torch.empty(shape, dtype=dtype, pin_memory=True)
        hq = pin(q)
        st.update(ctx=_context(L), seeds=kf.Tracks(pin(par), pin(cov), hq), hits=kf.TrackHits(pin(xyz), pin(valid)),
                  out=kf.Tracks(host(6, n), host(21, n), hq, host(3, n)), chi2=host(L, n),
                  status=host(n, dtype=torch.int32))
    elif kind == "bin":
        xyz, offs = _bin_inputs(case, seed)
        E, L = case["events"], case["layers"]
        st.update(ctx=_context(N_SEED_LAYERS + L),
                  lh=kf.LayerHits(xyz, torch.tensor(offs, device=DEV), E, L, N_SEED_LAYERS),
                  bins=kf.HitBins(_empty(xyz.shape[1], 4), _empty(E * L, kf.NBINS + 1, dtype=torch.int32)))
    elif kind == "reco":
        d = _reco_inputs(case, seed)
        E, Lb, n, nh = case["events"], N_BUILD_LAYERS, d["par"].shape[1], d["hits"].shape[1]
        i32 = torch.int32
        ctx = _context(N_SEED_LAYERS + Lb, case["x_x0"], max_cands=case["cands"])
        if case["fine"]:
            kf.kf_set_tuning(ctx, **{**kf.kf_get_tuning(ctx), "bin_unordered": 1})
        st.update(ctx=ctx, seeds=kf.Tracks(d["par"], d["cov"], d["charge"]), hits=kf.TrackHits(d["xyz"], d["valid"]),
                  fit=_out_tracks(n, d["charge"]), fit_status=_empty(n, dtype=i32),
                  lh=kf.LayerHits(d["hits"], torch.tensor(d["offs"], device=DEV), E, Lb, N_SEED_LAYERS),
                  bins=kf.HitBins(_empty(nh, 4), _empty(E * Lb, kf.NBINS + 1, dtype=i32),
                                  fine_off=_empty(E * Lb, kf.NBINS_FINE + 1, dtype=i32) if case["fine"] else None),
                  seed_off=torch.tensor(np.cumsum([0] + d["sizes"]), device=DEV),
                  res=kf.BuildResult(_out_tracks(n, d["charge"]), _empty(n), _empty(n, dtype=i32),
                                     _empty(n, dtype=i32), _empty(Lb, n, dtype=i32), _empty(n, dtype=i32)))
        if case["fine"]:
            st.update(s_fit=torch.cuda.Stream(), s_bin=torch.cuda.Stream(), fork=torch.cuda.Event())
        if case["refit"]:
            st.update(re=_out_tracks(n, d["charge"]), re_chi2=_empty(N_SEED_LAYERS + Lb, n),
                      re_status=_empty(n, dtype=i32))
    else:
        d = _reco_inputs(case, seed)
        Lb, events, b, lb = N_BUILD_LAYERS, [], 0, 0
        t = {k: d[k].cpu().numpy() for k in ("par", "cov", "charge", "xyz", "valid", "hits")}
        for s in d["sizes"]:
            o = np.asarray(d["offs"][lb:lb + Lb + 1], dtype=np.int64)
            events.append({k: np.ascontiguousarray(v) for k, v in dict(
                seed_par=t["par"][:, b:b + s], seed_cov=t["cov"][:, b:b + s], seed_charge=t["charge"][b:b + s],
                seed_hits=t["xyz"][:, :, b:b + s], seed_valid=t["valid"][:, b:b + s],
                layer_xyz=t["hits"][:, o[0]:o[-1]], layer_off=o - o[0]).items()})
            b += s
            lb += Lb
        ctx = _context(N_SEED_LAYERS + Lb, max_cands=case["cands"])
        kf.kf_serve_start(ctx, N_SEED_LAYERS, Lb, case["cands"])
        st.update(ctx=ctx, events=events)
    torch.cuda.synchronize()
    return st


def _tracks_out(t):
    return [t.par, t.par_lo, t.cov] if t.par_lo is not None else [t.par, t.cov]


def run(st):
    kind, ctx = st["case"]["kind"], st["ctx"]
    if kind in ("fit", "host"):
        fn = kf.kf_fit if kind == "fit" else kf.kf_fit_host
        fn(ctx, st["seeds"], st["hits"], st["out"], st["chi2"], st["status"])
        return _tracks_out(st["out"]) + [st["chi2"], st["status"]]
    if kind == "fit64":
        kf.kf_fit_f64(ctx, st["seeds"], st["hits"], st["out"], st["off"], st["chi2"], st["status"])
        return _tracks_out(st["out"]) + [st["chi2"], st["status"]]
    if kind == "bin":
        kf.kf_bin_hits(ctx, st["lh"], st["bins"])
        return [st["bins"].hits.view(torch.int32), st["bins"].bin_off]
    if kind == "reco":
        if "fork" in st:  # the seed fit and the binning side by side, joined before the build
            main = torch.cuda.current_stream()
            st["fork"].record(main)
            st["s_bin"].wait_event(st["fork"])
            st["s_fit"].wait_event(st["fork"])
            kf.kf_bin_hits(ctx, st["lh"], st["bins"], st["s_bin"])
            kf.kf_fit(ctx, st["seeds"], st["hits"], st["fit"], None, st["fit_status"], st["s_fit"])
            main.wait_stream(st["s_bin"])
            main.wait_stream(st["s_fit"])
        else:
            kf.kf_fit(ctx, st["seeds"], st["hits"], st["fit"], None, st["fit_status"])
            kf.kf_bin_hits(ctx, st["lh"], st["bins"])
        r = st["res"]
        kf.kf_build(ctx, st["fit"], st["seed_off"], st["bins"], st["case"]["cands"], r)
        out = _tracks_out(r.best) + [r.chi2_tot, r.n_hits, r.status, r.hit_idx, r.n_cands]
        if "re" in st:
            kf.kf_refit(ctx, st["seeds"], st["hits"], st["seed_off"], st["lh"], r.hit_idx, st["re"], st["re_chi2"],
                        st["re_status"])
            out += _tracks_out(st["re"]) + [st["re_chi2"], st["re_status"]]
        return out
    tickets = [kf.kf_submit(ctx, ev) for ev in st["events"]]
    out = []
    for t, ev in zip(tickets, st["events"]):
        r = kf.kf_poll(ctx, t, ev["seed_par"].shape[1], N_BUILD_LAYERS, want_cov=True)
        out.append([r[k] for k in ("best_par", "best_cov", "chi2_tot", "n_hits", "status", "hit_idx")])
    return out


# --------------------------------------------------------------------------- what a pass cannot do without


def work(case):
    """Bytes: each input read once, each output written once.  Flops: 1 442 per track and layer of the filter;
    of the build, per live candidate and layer (about 1 + 0.45 (cands - 1) of them a seed) 1 650 for the
    propagation, the window, its chi2 values and the update."""
    kind = case["kind"]
    if kind in ("fit", "host", "fit64"):
        n, L = case["n"], case["layers"]
        if kind == "fit64":
            per = 2 * (6 + 21) * 8 + 1 + L * 13 + L * 8 + 4
        else:
            per = 2 * (6 + 21) * 4 + (12 if case.get("lo", True) else 0) + 1 + L * 13 + L * 4 + 4
        return {"bytes": n * per, "flops": n * L * 1442}
    if kind == "bin":
        E, L, n = case["events"], case["layers"], case["hits"]
        f = (np.arange(E) + 0.5) / E
        hits = L * (E * n if not case["ragged"] else int(np.sum(np.exp(np.log(n) + (f - 1.0) * math.log(30.0)))))
        return {"bytes": hits * 28 + E * L * (kf.NBINS + 1) * 4, "flops": hits * 40}
    n = sum(_event_sizes(case))
    hits = N_BUILD_LAYERS * n * (1.0 + case.get("noise", 3.0))
    Lb, Ls = N_BUILD_LAYERS, N_SEED_LAYERS
    seeds = (6 + 21) * 4 + 1 + Ls * 13
    result = (6 + 3 + 21) * 4 + 4 * 4 + Lb * 4
    flops = n * (Ls * 1442 + Lb * 1650 * (1.0 + 0.45 * (case["cands"] - 1)))
    byts = n * (seeds + result) + hits * 12
    if case.get("refit"):
        byts += n * ((6 + 3 + 21) * 4 + (Ls + Lb) * 4 + 4)
        flops += n * (Ls + Lb) * 1442
    return {"bytes": int(byts), "flops": int(flops)}


# --------------------------------------------------------------------------- the same in 64 bits


def _full(cov):
    C = torch.zeros((cov.shape[1], 6, 6), device=DEV, dtype=torch.float64)
    for e, (i, j) in enumerate(zip(TRIL_I, TRIL_J)):
        C[:, i, j] = C[:, j, i] = cov[e].double()
    return C


def _packed(C):
    return torch.stack([C[:, i, j] for i, j in zip(TRIL_I, TRIL_J)])


V = (f32(SIGMA_XY) ** 2, f32(SIGMA_XY) ** 2, f32(SIGMA_Z) ** 2)


def _propagate(x, C, a, R, x_x0):
    """State [6, n] and covariance [n, 6, 6] on the cylinder r = R by the surface Jacobian, and whether each
    track got there (those that did not are left as they were)."""
    nx, ok, (s, p, pt, th, sa, ca, c, sn, rp) = _cross(x, a, R)
    ok = ok & (rp >= 0.01 * R * pt)
    X, Y, PX, PY, pz = nx[0], nx[1], nx[3], nx[4], nx[5]
    n = x.shape[1]
    D = torch.zeros((n, 6, 6), device=DEV, dtype=torch.float64)
    for i in (0, 1, 2, 5):
        D[:, i, i] = 1.0
    own = {(0, 0): sa, (0, 1): ca, (1, 0): -ca, (1, 1): sa, (2, 2): s / p, (3, 0): c, (3, 1): sn, (4, 0): -sn,
           (4, 1): c}
    slope = (-PX * s / p ** 3, -PY * s / p ** 3, -pz * s / p ** 3, -PY * th / p ** 2, PX * th / p ** 2)
    for i in range(5):
        for k in range(3):
            D[:, i, 3 + k] = slope[i] * x[3 + k] + own.get((i, k), 0.0)
    w = (X[:, None] * D[:, 0] + Y[:, None] * D[:, 1]) * (p / rp)[:, None]
    dF = torch.stack([PX / p, PY / p, pz / p, a * PY / p, -a * PX / p, torch.zeros_like(p)], dim=1)
    J = D - dF[:, :, None] * w[:, None, :]
    Cn = J @ C @ J.transpose(1, 2)
    if x_x0:
        P = nx[3:]
        p2 = p * p
        xe = x_x0 / (rp.abs() / (torch.hypot(X, Y) * p)).clamp_min(1e-6)
        th2 = _theta2(p2, xe)
        Cn[:, 3:, 3:] += th2[:, None, None] * (p2[:, None, None] * torch.eye(3, device=DEV, dtype=torch.float64) -
                                               P.T[:, :, None] * P.T[:, None, :])
    return torch.where(ok, nx, x), torch.where(ok[:, None, None], Cn, C), ok


def _s_inverse(C):
    S = C[:, :3, :3] + torch.diag(torch.tensor(V, device=DEV, dtype=torch.float64))
    r0, r1, r2 = S[:, 0], S[:, 1], S[:, 2]
    c0, c1, c2 = (torch.linalg.cross(u, v) for u, v in ((r1, r2), (r2, r0), (r0, r1)))
    return torch.stack([c0, c1, c2], dim=2) / (r0 * c0).sum(1)[:, None, None]


def _update(x, C, Si, m):
    K = C[:, :, :3] @ Si
    A = torch.eye(6, device=DEV, dtype=torch.float64).repeat(len(C), 1, 1)
    A[:, :, :3] -= K
    x = x + (K @ (m - x[:3]).T[:, :, None])[:, :, 0].T
    Vd = torch.diag(torch.tensor(V, device=DEV, dtype=torch.float64))
    return x, A @ C @ A.transpose(1, 2) + K @ Vd @ K.transpose(1, 2)


def _exact_fit(par, cov, charge, xyz, valid, radii, x_x0):
    """The filter over the layers: state [6, n], covariance [n, 6, 6], chi2 [L, n] (-1 without an update)."""
    xs, Cs, chis = [], [], []
    x_x0 = f32(x_x0)
    for b in range(0, par.shape[1], 400000):
        sl = slice(b, b + 400000)
        x, C, a = par[:, sl].double(), _full(cov[:, sl]), charge[sl].double() * (C_LIGHT * f32(BZ))
        live = torch.ones(x.shape[1], dtype=torch.bool, device=DEV)
        chi2 = torch.full((len(radii), x.shape[1]), -1.0, device=DEV, dtype=torch.float64)
        for l, R in enumerate(radii):
            nx, nC, ok = _propagate(x, C, a, R, x_x0)
            live = live & ok
            m = xyz[l, :, sl].double()
            Si = _s_inverse(nC)
            r = (m - nx[:3]).T
            upd = live & (valid[l, sl] != 0)
            chi2[l] = torch.where(upd, (r[:, None, :] @ Si @ r[:, :, None])[:, 0, 0], chi2[l])
            ux, uC = _update(nx, nC, Si, m)
            x = torch.where(upd, ux, torch.where(live, nx, x))
            C = torch.where(upd[:, None, None], uC, torch.where(live[:, None, None], nC, C))
        xs.append(x)
        Cs.append(C)
        chis.append(chi2)
    return torch.cat(xs, 1), torch.cat(Cs), torch.cat(chis, 1)


def _window_pairs(x, C, R, seg, hits, key, order):
    """(candidate, hit) pairs that can have chi2 < cut: hits of the candidate's segment within its phi window."""
    X, Y = x[0], x[1]
    r = torch.hypot(X, Y)
    cp, sp = X / r, Y / r
    s00, s10, s11 = C[:, 0, 0] + V[0], C[:, 1, 0], C[:, 1, 1] + V[1]
    wt = (CHI2_CUT * (sp * sp * s00 - 2 * sp * cp * s10 + cp * cp * s11)).sqrt()
    wn = (CHI2_CUT * (cp * cp * s00 + 2 * sp * cp * s10 + sp * sp * s11)).sqrt()
    half = (1.01 * torch.atan2(wt, (R - wn).clamp_min(1e-3)) + 1e-9).clamp_max(math.pi)
    mid = torch.atan2(Y, X) + 16.0 * seg
    lo, hi = torch.searchsorted(key, mid - half), torch.searchsorted(key, mid + half)
    cand = torch.repeat_interleave(torch.arange(len(mid), device=DEV), hi - lo)
    first = torch.cumsum(hi - lo, 0) - (hi - lo)
    hit = order[torch.arange(len(cand), device=DEV) - first[cand] + lo[cand]]
    wz = 1.01 * (CHI2_CUT * (C[:, 2, 2] + V[2])).sqrt() + 1e-6
    near = (hits[2, hit] - x[2, cand]).abs() < wz[cand]
    return cand[near], hit[near]


def _rank(owner, nh, chi2, parent, hit):
    """Order of the children by (owner, more hits, lower chi2, parent rank, hit id), and each one's rank among
    its owner's."""
    o = torch.arange(len(owner), device=DEV)
    for k in (hit, parent, chi2, -nh, owner):
        o = o[torch.sort(k[o], stable=True)[1]]
    own = owner[o]
    start = torch.searchsorted(own, own)
    return o, torch.arange(len(o), device=DEV) - start


def _exact_build(x, C, charge, event, hits, offs, radii, x_x0, n_max):
    """The clone engine in full: the best candidate's state, covariance, summed chi2 and hit ids of every seed."""
    n, Lb = x.shape[1], len(radii)
    a_seed = charge.double() * (C_LIGHT * f32(BZ))
    hits = hits.double()
    off = torch.tensor(offs, device=DEV)
    seg_of = torch.repeat_interleave(torch.arange(len(offs) - 1, device=DEV), off[1:] - off[:-1])
    phi = torch.atan2(hits[1], hits[0])
    key = torch.cat([phi - 2 * math.pi, phi, phi + 2 * math.pi]) + 16.0 * seg_of.repeat(3)
    ids = torch.arange(hits.shape[1], device=DEV).repeat(3)
    keep = (key - 16.0 * seg_of.repeat(3)).abs() <= 2 * math.pi  # the copies a window can reach
    key, o = torch.sort(key[keep])
    order = ids[keep][o]
    owner, rank = torch.arange(n, device=DEV), torch.zeros(n, dtype=torch.long, device=DEV)
    nh, chi2 = torch.zeros(n, dtype=torch.long, device=DEV), torch.zeros(n, device=DEV, dtype=torch.float64)
    path = torch.full((Lb, n), -1, dtype=torch.long, device=DEV)
    dead = torch.zeros(n, dtype=torch.bool, device=DEV)
    for l, R in enumerate(radii):
        nx, nC, ok = _propagate(x, C, a_seed[owner], R, f32(x_x0))
        dead = dead | ~ok
        x, C = torch.where(dead, x, nx), torch.where(dead[:, None, None], C, nC)
        Si = _s_inverse(C)
        live = torch.nonzero(~dead)[:, 0]
        pc, ph = [], []
        for b in range(0, len(live), 200000):
            i = live[b:b + 200000]
            c, h = _window_pairs(x[:, i], C[i], R, event[owner[i]] * Lb + l, hits, key, order)
            r = (hits[:, h] - x[:3, i[c]]).T
            v = (r[:, None, :] @ Si[i[c]] @ r[:, :, None])[:, 0, 0]
            pc.append(torch.stack([i[c], h])[:, v < CHI2_CUT])
            ph.append(v[v < CHI2_CUT])
        pair, v = torch.cat(pc, 1), torch.cat(ph)
        none = torch.ones(len(owner), dtype=torch.bool, device=DEV)
        none[pair[0]] = False
        lone = torch.nonzero(none)[:, 0]
        par = torch.cat([pair[0], lone])
        hit = torch.cat([pair[1], torch.full_like(lone, -1)])
        has = hit >= 0
        c2 = chi2[par] + torch.cat([v, torch.zeros(len(lone), device=DEV, dtype=torch.float64)])
        o, rk = _rank(owner[par], nh[par] + has, c2, rank[par], hit)
        o = o[rk < n_max]
        rank = rk[rk < n_max]
        par, hit, chi2 = par[o], hit[o], c2[o]
        has = hit >= 0
        nh, owner, dead = nh[par] + has, owner[par], dead[par]
        x, C, Si, path = x[:, par], C[par], Si[par], path[:, par]
        ux, uC = _update(x, C, Si, hits[:, hit.clamp_min(0)])
        x, C = torch.where(has, ux, x), torch.where(has[:, None, None], uC, C)
        path[l] = hit  # global hit index
    best = torch.nonzero(rank == 0)[:, 0]  # one a seed, in seed order
    return x[:, best], C[best], chi2[best], path[:, best]


def _exact_reco(case, seed, d):
    radii = _radii(N_SEED_LAYERS + N_BUILD_LAYERS)
    x, C, _ = _exact_fit(d["par"], d["cov"], d["charge"], d["xyz"], d["valid"], radii[:N_SEED_LAYERS],
                         case.get("x_x0", 0.0))
    out, ev0, b = [], 0, 0
    for s in d["sizes"]:  # event by event: bounded scratch
        sl = slice(b, b + s)
        o = d["offs"][ev0 * N_BUILD_LAYERS:(ev0 + 1) * N_BUILD_LAYERS + 1]
        ev = torch.zeros(s, dtype=torch.long, device=DEV)
        bx, bC, c2, path = _exact_build(x[:, sl], C[sl], d["charge"][sl], ev, d["hits"][:, o[0]:o[-1]],
                                        [v - o[0] for v in o], radii[N_SEED_LAYERS:], case.get("x_x0", 0.0),
                                        case["cands"])
        out.append((bx, bC, c2, torch.where(path >= 0, path + o[0], path)))
        ev0, b = ev0 + 1, b + s
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "host", "fit64"):
        par, cov, q, xyz, valid = _fit_inputs(case, seed)
        x, C, chi2 = _exact_fit(par, cov, q, xyz, valid, _radii(case["layers"]), case.get("x_x0", 0.0))
        lo = [None] if kind == "host" or (kind == "fit" and case["lo"]) else []
        return [x] + lo + [_packed(C), chi2, None]
    if kind == "bin":
        return None  # whole numbers and moved bytes
    d = _reco_inputs(case, seed)
    ev = _exact_reco(case, seed, d)
    if kind == "serve":
        return [[x.cpu().numpy(), _packed(C).cpu().numpy(), c2.cpu().numpy(), None, None, None]
                for x, C, c2, _ in ev]
    x, C, c2, path = (torch.cat([e[i] for e in ev], dim=0 if i in (1, 2) else 1) for i in range(4))
    out = [x, None, _packed(C), c2, None, None, None, None]
    if case["refit"]:
        h = d["hits"][:, path.clamp_min(0)].permute(1, 0, 2) * (path >= 0)[:, None, :]
        rx, rC, rchi = _exact_fit(d["par"], d["cov"], d["charge"], torch.cat([d["xyz"], h]),
                                  torch.cat([d["valid"], (path >= 0).to(torch.uint8)]),
                                  _radii(N_SEED_LAYERS + N_BUILD_LAYERS), case.get("x_x0", 0.0))
        out += [rx, None, _packed(rC), rchi, None]
    return out
