"""Workloads for timing the Kalman step library through its Python entry points.

Each case is one call (or one burst of calls) that a tracking program makes:
a single propagate+update step on a device batch, the step on a compressed
covariance store, the step on arrays in host memory, a multi-layer chain over
resident tracks, or a burst of events through the serving loop.  Inputs are
made on the GPU from a seed, with the distributions of the synthetic workloads
in ``paper_2401_14221_gb300/workload.py`` (vertex, pT, eta, covariance, hit
smearing); ``exact`` is the same filter in 64-bit PyTorch, written from the
helix and the textbook update.
"""
import math

import numpy as np
import torch

from paper_2401_14221_gb300 import kf

DEV = "cuda"
BZ = 3.8                      # T
ALPHA = 0.299792458e-2        # GeV / (cm T), unit charge
SIGMA = (0.01, 0.01, 0.05, 0.01, 1e-3, 1e-3)  # cm, cm, cm, relative, rad, rad
PRECISION = {"fp32": kf.KF_FP32, "fp64_update": kf.KF_FP64_UPDATE, "joseph": kf.KF_JOSEPH,
             "fp64": kf.KF_FP64, "adaptive": kf.KF_ADAPTIVE, "df_update": kf.KF_DF_UPDATE}
LAYER_FLOPS = 500             # 32-bit operations of one propagate+update of one track
PLANE_Z, CYLINDER_R = 50.0, 30.0


def listed():
    return [
        # One event's tracks to the next disk: the smallest configuration, a
        # call that a per-event loop makes, where latency and launch count.
        {"name": "p2z_fp32_8k", "op": "step", "kind": "p2z", "tracks": 8192, "precision": "fp32",
         "width": 32, "pt": "narrow", "surfaces": "one"},
        # The paper's batch: 100 events of 9,600 tracks to a barrel layer.
        {"name": "p2r_fp32_960k", "op": "step", "kind": "p2r", "tracks": 960000,
         "precision": "fp32", "width": 32, "pt": "narrow", "surfaces": "one"},
        # Structure-of-arrays data of another program, tightly measured hits:
        # the precision study's million tracks with the double-float update.
        {"name": "p2z_df_1m_soa", "op": "step", "kind": "p2z", "tracks": 1000000,
         "precision": "df_update", "width": 0, "pt": "wide", "surfaces": "one"},
        # The precision study with gain and covariance update in FP64.
        {"name": "p2r_fp64_update_960k", "op": "step", "kind": "p2r", "tracks": 960000,
         "precision": "fp64_update", "width": 32, "pt": "wide", "surfaces": "one"},
        # The precision study's reference arithmetic: every operation in FP64.
        {"name": "p2r_fp64_1m", "op": "step", "kind": "p2r", "tracks": 1000000,
         "precision": "fp64", "width": 64, "pt": "wide", "surfaces": "one"},
        # Tracks kept with FP32 sigmas and FP16 correlations.
        {"name": "p2r_compressed_960k", "op": "compressed", "kind": "p2r", "tracks": 960000,
         "precision": "fp32", "width": 32, "pt": "narrow", "surfaces": "one"},
        # A ragged batch in which every track has its own cylinder, some never
        # reached and some at grazing incidence: FP32 with FP64 where needed.
        {"name": "p2r_adaptive_ragged_soa", "op": "step", "kind": "p2r", "tracks": 300007,
         "precision": "adaptive", "width": 0, "pt": "wide", "surfaces": "per_track"},
        # 64 events through 15 layers at FP32, seeds kept (the chain works in
        # place, so a program that keeps its seeds copies them first).
        {"name": "chain_fp32_64ev", "op": "chain", "tracks": 440000, "precision": "fp32",
         "width": 32},
        # One event of median size, fitted as it arrives: latency counts.
        {"name": "chain_adaptive_event", "op": "chain", "tracks": 5000, "precision": "adaptive",
         "width": 0},
        # The whole 256-event batch at the accuracy that holds for every track.
        {"name": "chain_adaptive_256ev", "op": "chain", "tracks": 1750003,
         "precision": "adaptive", "width": 32},
        # A burst of events through the serving loop, results in host memory.
        {"name": "serve_16ev", "op": "serve", "events": 16, "sizes": 7, "precision": "adaptive"},
        # The paper's batch in pinned host memory, transfers in the call.
        {"name": "host_p2r_960k", "op": "host", "kind": "p2r", "tracks": 960000,
         "precision": "fp32", "width": 32, "pt": "narrow", "surfaces": "one"},
    ]


def draw(rng):
    """One more case of the listed ranges: any entry point, 1,000 tracks to the
    largest listed size (spread over the logarithm, mostly odd), any layout,
    precision and kind that is used with it."""
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["step", "step", "step", "compressed", "chain", "chain", "serve", "host"])
    if op == "serve":
        return {"op": op, "events": rng.randint(1, 20), "sizes": rng.randint(100, 9999),
                "precision": rng.choice(["adaptive", "fp32"])}
    width = rng.choice([0, 16, 32, 64, 128])
    if op == "chain":
        precision = rng.choice(["fp32", "adaptive", "adaptive", "joseph", "df_update", "fp64"])
        most = {"fp64": 50000, "df_update": 800000}.get(precision, 1750003)
        return {"op": op, "tracks": log_uniform(500, most), "precision": precision,
                "width": width}
    kind = rng.choice(["p2z", "p2r"])
    if op == "step":
        precision = rng.choice(["fp32", "joseph", "df_update", "fp64_update", "fp64", "adaptive"])
    else:
        precision = rng.choice(["fp32", "joseph"] if op == "compressed" else ["fp32", "adaptive"])
    # a surface of each track's own is reached at grazing incidence at times:
    # only these precisions resolve that
    own = op == "step" and precision in ("adaptive", "fp64") and rng.random() < 0.5
    return {"op": op, "kind": kind, "tracks": log_uniform(1000, 1000000), "precision": precision,
            "width": width, "pt": rng.choice(["narrow", "wide"]),
            "surfaces": "per_track" if own else "one"}


def _event_sizes(case):
    rng = np.random.default_rng(case["sizes"])
    s = np.exp(rng.normal(math.log(5000.0), 1.0, case["events"]))
    return [int(v) for v in np.clip(np.rint(s), 500, 40000)]


def _layers():
    """Eight cylinders and seven planes, alternating outwards."""
    rs, zs = np.linspace(4.0, 110.0, 8), np.linspace(30.0, 280.0, 7)
    out = []
    for i in range(8):
        out.append(("p2r", float(np.float32(rs[i]))))
        if i < 7:
            out.append(("p2z", float(np.float32(zs[i]))))
    return out


def work(case):
    """Bytes: every input read once, every output written once (a plane needs
    x, y and their 2x2 covariance of a hit).  FP64 work is counted in the same
    number of operations."""
    hit = {"p2z": 4 * (2 + 3), "p2r": 4 * (3 + 6)}
    if case["op"] in ("chain", "serve"):
        n = case["tracks"] if case["op"] == "chain" else sum(_event_sizes(case))
        lay = _layers()
        return {"bytes": n * (2 * 4 * 27 + 2 + sum(hit[k] for k, _ in lay)),
                "flops": n * LAYER_FLOPS * len(lay)}
    n = case["tracks"]
    track = 4 * (6 + 6) + 2 * 15 if case["op"] == "compressed" else 4 * 27
    own = 4 if case["surfaces"] == "per_track" else 0
    return {"bytes": n * (2 * track + 2 + hit[case["kind"]] + own), "flops": n * LAYER_FLOPS}


# ------------------------------------------------------------ 64-bit filter

def _sinc(h):
    """sin(h)/h and its derivative."""
    small = h.abs() < 0.05
    hs = torch.where(small, torch.ones_like(h), h)
    S = torch.where(small, 1 - h * h / 6 * (1 - h * h / 20 * (1 - h * h / 42)), torch.sin(hs) / hs)
    dS = torch.where(small, -h / 3 * (1 - h * h / 10 * (1 - h * h / 28 * (1 - h * h / 54))),
                     (torch.cos(hs) - S) / hs)
    return S, dS


def _wrap(a):
    w = a - 2 * math.pi * torch.round(a / (2 * math.pi))
    return torch.where(w <= -math.pi, w + 2 * math.pi, w)


def _path(kind, p, omega, surf):
    """Transverse path to the surface and the mask of tracks that reach it."""
    x, y, z, _, phi, th = p
    if kind == "p2z":
        return (surf - z) * torch.tan(th), torch.cos(th).abs() > 1e-4
    cp, sp = torch.cos(phi), torch.sin(phi)
    d = surf * surf - (x * x + y * y)
    a, b = x * cp + y * sp, y * cp - x * sp
    disc = a * a + (1 + omega * b - 0.25 * d * omega * omega) * d
    ok = (d > 0) & (disc >= 0)
    den = a + torch.sqrt(disc.clamp_min(0))
    h = torch.atan2(omega * d, 2 * den)   # half turning angle to the crossing
    w = torch.where(omega.abs() > 1e-12, omega, torch.ones_like(omega))
    return torch.where(omega.abs() > 1e-12, 2 * h / w, d / den), ok


def _helix(p, omega, s):
    """State after the transverse path s (phi not wrapped)."""
    x, y, z, k, phi, th = p
    h = 0.5 * omega * s
    L = s * _sinc(h)[0]
    return torch.stack([x + L * torch.cos(phi + h), y + L * torch.sin(phi + h),
                        z + s / torch.tan(th), k, phi + 2 * h, th])


def _step64(kind, p, C, q, surf, hit, hc):
    """One propagate + update of tracks p [6, n], C [n, 6, 6]; tracks that do
    not reach the surface are left as they are."""
    w = -ALPHA * float(np.float32(BZ)) * q
    omega = w * p[3]
    s, ok = _path(kind, p, omega, surf)
    s = torch.where(ok, s, torch.ones_like(s))
    out = _helix(p, omega, s)
    if kind == "p2z":
        out[2] = surf
    phi, th = p[4], p[5]
    h = 0.5 * omega * s
    S, dS = _sinc(h)
    cm, sm, c1, s1 = torch.cos(phi + h), torch.sin(phi + h), torch.cos(out[4]), torch.sin(out[4])
    cot = 1 / torch.tan(th)
    n = s.shape[0]
    J = torch.zeros(n, 6, 6, dtype=torch.float64, device=s.device)
    for i in range(6):
        J[:, i, i] = 1
    g = 0.5 * s * s * w
    J[:, 0, 3], J[:, 1, 3] = g * (dS * cm - S * sm), g * (dS * sm + S * cm)
    J[:, 0, 4], J[:, 1, 4] = -s * S * sm, s * S * cm
    J[:, 4, 3] = w * s
    J[:, 2, 5] = -s / torch.sin(th) ** 2
    dp = torch.stack([c1, s1, cot, torch.zeros_like(s), omega, torch.zeros_like(s)], 1)
    if kind == "p2z":   # s = (surf - z) tan(theta): z' does not move
        ds = torch.zeros(n, 6, dtype=torch.float64, device=s.device)
        ds[:, 2], ds[:, 5] = -torch.tan(th), (surf - p[2]) / torch.cos(th) ** 2
        J = J + dp[:, :, None] * ds[:, None, :]
        J[:, 2, :] = 0
    else:               # x'^2 + y'^2 = R^2
        ds = -(out[0][:, None] * J[:, 0] + out[1][:, None] * J[:, 1])
        ds = ds / (out[0] * c1 + out[1] * s1)[:, None]
        J = J + dp[:, :, None] * ds[:, None, :]
    Cp = J @ C @ J.transpose(1, 2)
    H = torch.zeros(n, 2, 6, dtype=torch.float64, device=s.device)
    V = torch.zeros(n, 2, 2, dtype=torch.float64, device=s.device)
    if kind == "p2z":
        H[:, 0, 0] = H[:, 1, 1] = 1
        V[:, 0, 0], V[:, 1, 1] = hc[0], hc[2]
        V[:, 0, 1] = V[:, 1, 0] = hc[1]
        r = torch.stack([hit[0] - out[0], hit[1] - out[1]], 1)
    else:
        ir = 1 / torch.hypot(hit[0], hit[1])
        ux, uy = -hit[1] * ir, hit[0] * ir
        H[:, 0, 0], H[:, 0, 1], H[:, 1, 2] = ux, uy, 1
        V[:, 0, 0] = ux * ux * hc[0] + 2 * ux * uy * hc[1] + uy * uy * hc[2]
        V[:, 0, 1] = V[:, 1, 0] = ux * hc[3] + uy * hc[4]
        V[:, 1, 1] = hc[5]
        r = torch.stack([ux * (hit[0] - out[0]) + uy * (hit[1] - out[1]), hit[2] - out[2]], 1)
    U = Cp @ H.transpose(1, 2)
    M = H @ U + V
    det = M[:, 0, 0] * M[:, 1, 1] - M[:, 0, 1] * M[:, 1, 0]
    pd = (M[:, 0, 0] > 0) & (det > 0)
    Mi = torch.stack([M[:, 1, 1], -M[:, 0, 1], -M[:, 1, 0], M[:, 0, 0]], 1) / det[:, None]
    K = U @ Mi.reshape(n, 2, 2)
    IKH = torch.eye(6, dtype=torch.float64, device=s.device) - K @ H
    Cu = IKH @ Cp @ IKH.transpose(1, 2) + K @ V @ K.transpose(1, 2)
    pu = out + (K @ r[:, :, None])[:, :, 0].T
    pn = torch.where(pd, pu, out)
    Cn = torch.where(pd[:, None, None], Cu, Cp)
    pn[4] = _wrap(pn[4])
    return torch.where(ok, pn, p), torch.where(ok[:, None, None], Cn, C)


_LOW = [(i, j) for i in range(6) for j in range(i + 1)]
_OFF = [(i, j) for i in range(6) for j in range(i)]


def _full(c):
    """Packed [21, n] -> [n, 6, 6]."""
    C = torch.empty(c.shape[1], 6, 6, dtype=torch.float64, device=c.device)
    for e, (i, j) in enumerate(_LOW):
        C[:, i, j] = C[:, j, i] = c[e].double()
    return C


def _packed(C):
    return torch.stack([C[:, i, j] for i, j in _LOW])


# ------------------------------------------------------------------- inputs

def _rng(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(*shape, dtype=torch.float64, device=DEV, generator=g)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, dtype=torch.float64, device=DEV, generator=g)

    return normal, uniform


def _truth(normal, uniform, n, pt, eta):
    q = torch.where(uniform(0, 1, n) < 0.5, 1.0, -1.0).double()
    p = torch.stack([0.01 * normal(n), 0.01 * normal(n), 5.0 * normal(n),
                     1 / uniform(pt[0], pt[1], n), uniform(-math.pi, math.pi, n),
                     2 * torch.atan(torch.exp(-uniform(eta[0], eta[1], n)))])
    return p, q


def _smeared(normal, truth):
    """Covariance C = A A^T + diag(sigma^2) and a start state truth + N(0, C)."""
    n = truth.shape[1]
    sig = torch.tensor(SIGMA, dtype=torch.float64, device=DEV)[:, None].repeat(1, n)
    sig[3] *= truth[3]
    A = normal(n, 6, 6) * (0.1 * sig).T[:, :, None]
    C = A @ A.transpose(1, 2) + torch.diag_embed((sig * sig).T)
    start = truth + (A @ normal(n, 6, 1))[:, :, 0].T + sig * normal(6, n)
    start[4] = _wrap(start[4])
    return start.float(), _packed(C).float()


def _hit(normal, kind, at, ok, surf, n):
    """Smeared hit [3, n] and its covariance [6, n] (a placeholder off `ok`)."""
    hit, hc = (torch.zeros(c, n, dtype=torch.float64, device=DEV) for c in (3, 6))
    if kind == "p2z":
        hit[0] = torch.where(ok, at[0] + 0.01 * normal(n), 0.0)
        hit[1] = torch.where(ok, at[1] + 0.01 * normal(n), 0.0)
        hit[2] = surf
        hc[0] = hc[2] = hc[5] = 1e-4
    else:
        a = torch.where(ok, torch.atan2(at[1], at[0]) + 0.01 * normal(n) / surf, 0.0)
        c, s = torch.cos(a), torch.sin(a)
        hit[0], hit[1] = surf * c, surf * s
        hit[2] = torch.where(ok, at[2] + 0.05 * normal(n), 0.0)
        hc[0], hc[1], hc[2], hc[5] = 1e-4 * s * s, -1e-4 * s * c, 1e-4 * c * c, 2.5e-3
    return hit.float(), hc.float()


def _go(kind, p, q, surf):
    """True state on the surface, and whether the track reaches it."""
    omega = -ALPHA * BZ * q * p[3]
    s, ok = _path(kind, p, omega, surf)
    return _helix(p, omega, s), ok


def _step_inputs(case, seed):
    """Canonical inputs ([components, n] on the GPU) of a single-step case."""
    n, kind = case["tracks"], case["kind"]
    normal, uniform = _rng(seed)
    pt = (0.5, 10.0) if case["pt"] == "narrow" else (0.2, 100.0)
    truth, q = _truth(normal, uniform, n, pt, (1.5, 2.5) if kind == "p2z" else (-1.5, 1.5))
    if case["surfaces"] == "one":
        surf = torch.full((1,), PLANE_Z if kind == "p2z" else CYLINDER_R, device=DEV)
    else:
        surf = uniform(*((20.0, 120.0) if kind == "p2z" else (5.0, 150.0)), n).float()
    at, ok = _go(kind, truth, q, surf.double())
    state, cov = _smeared(normal, truth)
    hit, hc = _hit(normal, kind, at, ok, surf.double(), n)
    return {"state": state, "cov": cov, "q": q.to(torch.int8), "surf": surf, "hit": hit, "hc": hc}


def _chain_inputs(n, seed):
    """Tracks from a pool of true ones, smeared on their own, a hit per layer."""
    normal, uniform = _rng(seed)
    m = min(65536, n)
    truth, q = _truth(normal, uniform, m, (0.5, 10.0), (1.5, 2.5))
    pick = (torch.arange(n, device=DEV) if n == m
            else uniform(0, m, n).long().clamp_(max=m - 1))
    state, cov = _smeared(normal, truth[:, pick])
    hits, hcs, cur = [], [], truth
    alive = torch.ones(m, dtype=torch.bool, device=DEV)
    for kind, pos in _layers():
        at, ok = _go(kind, cur, q, pos)
        alive_here = alive & ok
        h, c = _hit(normal, kind, at[:, pick], alive_here[pick], pos, n)
        hits.append(h)
        hcs.append(c)
        cur = torch.where(alive_here, at, cur)
    return {"state": state, "cov": cov, "q": q[pick].to(torch.int8), "hits": hits, "hcs": hcs}


def _to_layout(a, width):
    """[C, n] -> the flat array of the layout (blocks padded with zeros)."""
    if not width:
        return a.contiguous().reshape(-1)
    C, n = a.shape
    nb = -(-n // width)
    pad = torch.zeros(C, nb * width, dtype=a.dtype, device=a.device)
    pad[:, :n] = a
    return pad.reshape(C, nb, width).transpose(0, 1).contiguous().reshape(-1)


def _rho_to_layout(r, width):
    """[15, n] correlations -> seven rows of pairs and one row per block."""
    w = width or r.shape[1]
    b = _to_layout(r, width).reshape(-1, 15, w)
    pairs = b[:, :14].reshape(-1, 7, 2, w).transpose(2, 3).reshape(-1, 14 * w)
    return torch.cat([pairs, b[:, 14]], 1).contiguous().reshape(-1)


def _compress(C):
    """[21, n] -> sigma [6, n] and correlations [15, n] in [-1, 1]."""
    C = C.double()
    tri = {ij: e for e, ij in enumerate(_LOW)}
    sig = torch.stack([C[tri[i, i]] for i in range(6)]).clamp_min(0).sqrt()
    rho = []
    for i, j in _OFF:
        den = sig[i] * sig[j]
        one = torch.ones_like(den)
        rho.append(torch.where(den > 0, C[tri[i, j]] / torch.where(den > 0, den, one), 0.0))
    return sig, torch.stack(rho).clamp(-1, 1)


def _layout(case):
    w = case["width"]
    return kf.make_layout(kf.KF_AOSOA if w else kf.KF_SOA, w or 32, case["tracks"])


_SERVERS = {}   # a program keeps its serving loop; one per precision


def _server(precision):
    if precision not in _SERVERS:
        lay = _layers()
        arena = torch.empty(1 << 30, dtype=torch.uint8, device=DEV)
        _SERVERS[precision] = kf.Server(BZ, [int(k == "p2r") for k, _ in lay],
                                        [z for _, z in lay], arena, max_events_in_flight=64,
                                        precision=PRECISION[precision])
    return _SERVERS[precision]


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def prepare(case, seed):
    prec = PRECISION[case["precision"]]
    if case["op"] == "serve":
        sizes = _event_sizes(case)
        n = sum(sizes)
        x = _chain_inputs(n, seed)
        hits, hcs = torch.stack(x["hits"]), torch.stack(x["hcs"])
        out = {"state": torch.zeros(6 * n, pin_memory=True),
               "cov": torch.zeros(21 * n, pin_memory=True),
               "status": torch.zeros(n, dtype=torch.uint8, pin_memory=True)}
        events, lo = [], 0
        for s in sizes:
            hi = lo + s
            events.append((_pinned(x["state"][:, lo:hi].contiguous()),
                           _pinned(x["cov"][:, lo:hi].contiguous()), _pinned(x["q"][lo:hi]),
                           _pinned(hits[:, :, lo:hi].contiguous()),
                           _pinned(hcs[:, :, lo:hi].contiguous()),
                           out["state"][6 * lo:6 * hi].view(6, s),
                           out["cov"][21 * lo:21 * hi].view(21, s), out["status"][lo:hi]))
            lo = hi
        return {"op": "serve", "server": _server(case["precision"]), "events": events, "out": out}
    w = case["width"]
    if case["op"] == "chain":
        x = _chain_inputs(case["tracks"], seed)
        state, cov = _to_layout(x["state"], w), _to_layout(x["cov"], w)
        hits = torch.cat([_to_layout(h, w) for h in x["hits"]])
        hcs = torch.cat([_to_layout(h, w) for h in x["hcs"]])
        lay = _layers()
        dc = kf.DeviceChain(n=case["tracks"], layout=_layout(case),
                            layers=kf.make_layers([int(k == "p2r") for k, _ in lay],
                                                  [z for _, z in lay]),
                            state0=state, cov0=cov, state=state.clone(), cov=cov.clone(),
                            charge=x["q"], hits=hits, hit_covs=hcs,
                            status=torch.zeros(case["tracks"], dtype=torch.uint8, device=DEV),
                            bz=BZ, f3=hits.numel() // len(lay), f6=hcs.numel() // len(lay))
        return {"op": "chain", "chain": dc, "precision": prec}
    x = _step_inputs(case, seed)
    if case["op"] == "compressed":
        sig, rho = _compress(x["cov"])
        sig = _to_layout(sig.float(), w)
        rho = _rho_to_layout(rho.half(), w)
        state = _to_layout(x["state"], w)
        outs = [torch.zeros_like(state), torch.zeros_like(sig), torch.zeros_like(rho)]
        status = torch.zeros(case["tracks"], dtype=torch.uint8, device=DEV)
        return {"op": "compressed", "kind": kf.KF_P2Z if case["kind"] == "p2z" else kf.KF_P2R,
                "params": kf.make_params(BZ, prec), "layout": _layout(case),
                "in": [state, sig, rho], "out": outs, "charge": x["q"],
                "hit": _to_layout(x["hit"], w), "hc": _to_layout(x["hc"], w), "surf": x["surf"],
                "own": int(x["surf"].numel() > 1), "status": status}
    place = _pinned if case["op"] == "host" else (lambda t: t)
    state, cov = place(_to_layout(x["state"], w)), place(_to_layout(x["cov"], w))
    fields = dict(kind=int(case["kind"] == "p2r"), n=case["tracks"], layout=_layout(case),
                  state_in=state, cov_in=cov,
                  state_out=place(torch.zeros_like(state)), cov_out=place(torch.zeros_like(cov)),
                  charge=place(x["q"]), hit=place(_to_layout(x["hit"], w)),
                  hit_cov=place(_to_layout(x["hc"], w)), surf=place(x["surf"]),
                  status=place(torch.zeros(case["tracks"], dtype=torch.uint8, device=DEV)), bz=BZ)
    if case["op"] == "host":
        fields["workspace"] = torch.empty(kf.kf_host_workspace_bytes(fields["layout"], 0),
                                          dtype=torch.uint8, device=DEV)
        return {"op": "host", "batch": kf.HostBatch(**fields), "precision": prec}
    return {"op": "step", "batch": kf.DeviceBatch(**fields), "precision": prec}


def run(state):
    op = state["op"]
    if op in ("step", "host"):
        b = state["batch"]
        b.run(state["precision"])
        return [b.state_out, b.cov_out, b.status]
    if op == "chain":
        dc = state["chain"]
        dc.reset()
        dc.run(state["precision"])
        return [dc.state, dc.cov, dc.status]
    if op == "compressed":
        s = state
        kf.kf_propagate_update_compressed(s["kind"], s["params"], s["layout"], *s["in"], *s["out"],
                                          s["charge"], s["hit"], s["hc"], s["surf"], s["own"],
                                          s["status"])
        return [*s["out"], s["status"]]
    srv = state["server"]
    for t in [srv.submit(*e) for e in state["events"]]:
        srv.wait(t)
    return [state["out"]["state"], state["out"]["cov"], state["out"]["status"]]


# -------------------------------------------------------------------- exact

def _chain64(x, n):
    """The chain in 64 bits, in pieces that fit the card beside the inputs."""
    ps, cs = [], []
    for lo in range(0, n, 200000):
        c = slice(lo, min(n, lo + 200000))
        p, C, q = x["state"][:, c].double(), _full(x["cov"][:, c]), x["q"][c].double()
        for (kind, pos), h, v in zip(_layers(), x["hits"], x["hcs"]):
            p, C = _step64(kind, p, C, q, pos, h[:, c].double(), v[:, c].double())
        ps.append(p)
        cs.append(_packed(C))
    return torch.cat(ps, 1), torch.cat(cs, 1)


def exact(case, seed):
    out = _exact(case, seed)
    if case["op"] in ("chain", "serve") and case["precision"] not in ("adaptive", "fp64"):
        # a few tracks barely reach an outer cylinder (incidence cosine down to
        # 0.004); with 32-bit state between layers their covariance, the
        # largest in the batch, is not resolved: it has no value to compare
        out[1] = None
    return out


def _exact(case, seed):
    if case["op"] == "serve":
        sizes = _event_sizes(case)
        p, c = _chain64(_chain_inputs(sum(sizes), seed), sum(sizes))
        flat, lo = [[], []], 0
        for s in sizes:
            flat[0].append(p[:, lo:lo + s].reshape(-1))
            flat[1].append(c[:, lo:lo + s].reshape(-1))
            lo += s
        return [torch.cat(flat[0]), torch.cat(flat[1]), None]
    w = case["width"]
    if case["op"] == "chain":
        p, c = _chain64(_chain_inputs(case["tracks"], seed), case["tracks"])
        return [_to_layout(p, w), _to_layout(c, w), None]
    x = _step_inputs(case, seed)
    if case["op"] == "compressed":   # the store's own rounding of the input is not an error
        sig, rho = _compress(x["cov"])
        sig, rho = sig.float().double(), rho.half().double()
        cov = torch.zeros(21, case["tracks"], dtype=torch.float64, device=DEV)
        for e, (i, j) in enumerate(_LOW):
            cov[e] = sig[i] * sig[j] * (1.0 if i == j else rho[_OFF.index((i, j))])
        x["cov"] = cov
    p, C = _step64(case["kind"], x["state"].double(), _full(x["cov"]), x["q"].double(),
                   x["surf"].double(), x["hit"].double(), x["hc"].double())
    c = _packed(C)
    if case["op"] == "compressed":
        sig, rho = _compress(c)
        return [_to_layout(p, w), _to_layout(sig, w), _rho_to_layout(rho, w), None]
    return [_to_layout(p, w), _to_layout(c, w), None]
