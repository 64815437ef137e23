"""What is measured: the work that a user of this package has it do, through its public entry points.

A filter frame (`LETKF.step`, `LETKFPair.step`, a served frame) is the unit of use: slopes in, prediction
out, the ensemble updated.  Every pass runs one frame (the server: two per system) from an ensemble in the
steady state of a running loop, and reads the updated ensemble back, as a checkpoint does.
"""

import functools
import math

import numpy as np
import torch

from paper_1310_5954_gb300 import LETKF, LETKFPair, Server, _lib

PITCH = 0.5             # metres between actuators
R0, L0 = 1.0, 25.0      # Fried parameter and outer scale of the turbulence, metres
FRAME = 1e-3            # seconds per frame
N_SLOPES = 4            # frames of slopes that a state holds; passes take them in turn
RESTART = 16            # passes after which a loop goes back to its checkpoint: filters of few members drift off
                        # over hundreds of frames, and what is timed is a loop that follows the truth


def _case(name, kind, n_sub, m, precision, path, sigma=0.2, a=0.995, a2=0.0, obstruction=0.0, dom_sub=4, halo=2,
          piston="off", noise="dense", wind=15.0, mix=""):
    return dict(name=name, kind=kind, n_sub=n_sub, m=m, precision=precision, path=path, sigma=sigma, a=a, a2=a2,
                obstruction=obstruction, dom_sub=dom_sub, halo=halo, piston=piston, noise=noise, wind=wind, mix=mix)


def listed():
    return [
        # a small system on the tuned path: a laboratory or 4 m class loop, where latency and launches count
        _case("step 8x8 m20 mixed", "step", 8, 20, "mixed", "fused", sigma=0.1, a=0.99, halo=1, wind=10.0),
        # the same system in 64 bits: the reference arithmetic that a user checks a set-up with
        _case("step 8x8 m20 fp64 plain", "step", 8, 20, "fp64", "plain", sigma=0.1, a=0.99, halo=1, wind=10.0),
        # an 8 m class system, fewer domains than SMs
        _case("step 40x40 m50 mixed", "step", 40, 50, "mixed", "fused", sigma=0.15, obstruction=0.14, wind=10.0),
        # the same system with the package's default precision and path
        _case("step 40x40 m50 fp32 plain", "step", 40, 50, "fp32", "plain", sigma=0.15, obstruction=0.14, wind=10.0),
        # odd sizes, AR(2) turbulence and piston removal inside the loop
        _case("step 49x49 m77 mixed ar2 pist", "step", 49, 77, "mixed", "fused", sigma=0.13, a=1.58, a2=-0.585,
              obstruction=0.11, piston="in_loop"),
        # the ELT-scale system that the project's benchmark quotes
        _case("step 80x80 m100 mixed", "step", 80, 100, "mixed", "fused", obstruction=0.28),
        # the same system held in 32 bits throughout (noise factor included)
        _case("step 80x80 m100 fp32", "step", 80, 100, "fp32", "fused", obstruction=0.28),
        # the ELT-scale system with a wide ensemble (observation-space analysis)
        _case("step 80x80 m200 mixed", "step", 80, 200, "mixed", "fused", obstruction=0.28),
        # two filters with shifted domain partitions, run together
        _case("pair 80x80 m100 mixed", "pair", 80, 100, "mixed", "fused", obstruction=0.28),
        # global ETKF, 16 m class and ELT scale
        _case("global 32x32 m197", "step", 32, 197, "fp32", "global", sigma=0.1, a=0.99, wind=10.0),
        _case("global 80x80 m1024", "step", 80, 1024, "fp32", "global", obstruction=0.28),
        # one GPU serving loops of several sizes at once, slopes and predictions on the host
        _case("serve six systems", "serve", 64, 200, "mixed", "fused",
              mix="16:20:0.1:0.05 32:50:0.2:0.2 40:100:0.15:0.14 64:200:0.25:0.1 64:20:0.3:0.0 40:50:0.2:0.25"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["fused", "fused", "fused", "dual", "plain32", "plain64", "pair", "global", "serve"])
    sigma, obs, wind = rng.uniform(0.1, 0.3), rng.uniform(0.0, 0.28), rng.uniform(5.0, 25.0)
    c = dict(sigma=sigma, obstruction=obs, wind=wind, noise=rng.choice(["dense", "dense", "dense", "white"]))
    if what == "fused":
        ar2 = rng.random() < 0.2
        if ar2:
            c.update(a=1.58, a2=-0.585)
        return _case("", "step", _log(rng, 8, 80), _log(rng, 20, 126), rng.choice(["mixed", "mixed", "fp32"]), "fused",
                     halo=rng.choice([1, 2, 2]), piston=rng.choice(["off", "off", "output", "in_loop"]), **c)
    if what == "dual":
        return _case("", "step", _log(rng, 8, 64), rng.randint(128, 256), rng.choice(["mixed", "mixed", "fp32"]), "fused",
                     piston=rng.choice(["off", "off", "in_loop"]), **c)
    if what == "plain32":
        dom, halo = rng.choice([(4, 1), (4, 2), (5, 2), (6, 3)])   # the last is wider than the fused path holds
        return _case("", "step", _log(rng, 8, 40), _log(rng, 20, 100), "fp32", "plain", dom_sub=dom, halo=halo, **c)
    if what == "plain64":
        return _case("", "step", _log(rng, 8, 20), _log(rng, 20, 64), "fp64", "plain", halo=rng.choice([1, 2]), **c)
    if what == "pair":
        return _case("", "pair", _log(rng, 16, 64), _log(rng, 20, 110), "mixed", "fused", **c)
    if what == "global":
        return _case("", "step", _log(rng, 16, 64), _log(rng, 64, 800), "fp32", "global", **c)
    mix = " ".join("%d:%d:%.3f:%.3f" % (rng.choice([16, 24, 32, 40, 57]), rng.choice([20, 50, 64, 100, 150, 200]),
                                        rng.uniform(0.1, 0.3), rng.uniform(0.0, 0.28)) for _ in range(rng.randint(2, 6)))
    return _case("", "serve", 57, 200, "mixed", "fused", mix=mix, wind=wind)


# ---- geometry, turbulence and ensembles -----------------------------------------------------------

class _Geo:
    """Circular pupil with a central obstruction, Fried actuators, estimation domains (numpy)."""

    def __init__(self, n, obstruction):
        q = 20
        t = 2 * np.arange(q * n) + 1 - q * n
        d2 = t[:, None].astype(np.int64) ** 2 + t[None, :].astype(np.int64) ** 2
        lit = (d2 <= (q * n) ** 2) & (d2 >= (obstruction * q * n) ** 2)
        sub = 2 * lit.reshape(n, q, n, q).sum(axis=(1, 3)) >= q * q
        act = np.zeros((n + 1, n + 1), dtype=bool)
        for i in (0, 1):
            for j in (0, 1):
                act[i:n + i, j:n + j] |= sub
        self.n, self.sub, self.act = n, sub, act
        self.sub_rc, self.act_rc = np.argwhere(sub), np.argwhere(act)
        index = -np.ones(act.shape, dtype=np.int64)
        index[act] = np.arange(len(self.act_rc))
        r, c = self.sub_rc.T
        # the four corner actuators of each valid subaperture: (r, c) (r, c+1) (r+1, c) (r+1, c+1)
        self.corners = np.stack([index[r, c], index[r, c + 1], index[r + 1, c], index[r + 1, c + 1]], axis=1)
        self.n_act, self.n_subv = len(self.act_rc), len(self.sub_rc)

    def slopes(self, x):
        """Fried slopes of x (n_act, ...): all x-slopes, then all y-slopes."""
        a = [x[self.corners[:, k]] for k in range(4)]
        cat = torch.cat if isinstance(x, torch.Tensor) else np.concatenate
        return cat([0.5 * ((a[1] + a[3]) - (a[0] + a[2])), 0.5 * ((a[2] + a[3]) - (a[0] + a[1]))])

    def owner(self, b, offset=0):
        last = (self.n - 1 + offset) // b
        rc = np.minimum((self.act_rc + offset) // b, last)
        return rc[:, 0], rc[:, 1]

    def domains(self, b, halo, offset=0):
        """[(owned actuators, observed subapertures)] of the blocks that own an actuator."""
        I, J = self.owner(b, offset)
        out = []
        for i, j in sorted(set(zip(I.tolist(), J.tolist()))):
            lo_r, lo_c = b * i - offset - halo, b * j - offset - halo
            s = self.sub_rc
            seen = (s[:, 0] >= lo_r) & (s[:, 0] < lo_r + b + 2 * halo) & (s[:, 1] >= lo_c) & (s[:, 1] < lo_c + b + 2 * halo)
            out.append((np.flatnonzero((I == i) & (J == j)), np.flatnonzero(seen)))
        return out


@functools.lru_cache(maxsize=16)
def _geo(n, obstruction):
    return _Geo(n, obstruction)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _covariance(d):
    """Phase covariance at a distance d (pitches): Kolmogorov's r^(5/3) structure function up to the outer scale."""
    s0 = 3.44 * (L0 / R0) ** (5.0 / 3.0)
    return s0 * torch.exp(-(d * PITCH / L0) ** (5.0 / 3.0))


@functools.lru_cache(maxsize=8)
def _noise_factor(n, obstruction, a, a2, wind):
    """Lower-triangular L, L L^T the covariance of the AR innovation of this turbulence under frozen flow."""
    rc = torch.as_tensor(_geo(n, obstruction).act_rc, dtype=torch.float64, device=_device())
    dr, dc = (rc[:, k][:, None] - rc[:, k][None, :] for k in (0, 1))
    step = wind * FRAME / PITCH

    def lagged(k):
        return _covariance(torch.hypot(dr, dc + k * step)) + _covariance(torch.hypot(dr, dc - k * step))

    Q = (1 + a * a + a2 * a2) * _covariance(torch.hypot(dr, dc)) - (a - a * a2) * lagged(1)
    if a2:
        Q = Q - a2 * lagged(2)
    Q.diagonal().add_(1e-5 * Q.diagonal().mean().item() + 1e-6)
    return np.ascontiguousarray(torch.linalg.cholesky(Q).cpu().numpy())


def _fields(gen, count, n, rms, scale, shifts=(0.0,)):
    """[len(shifts)][count, n+1, n+1]: random smooth fields (power law up to `scale` pitches) moved along a row."""
    g = 1 << max(5, math.ceil(math.log2(1.5 * (n + 1))))
    dev = _device()
    k = torch.fft.fftfreq(g, device=dev, dtype=torch.float64)
    ky, kx = k[:, None], torch.fft.rfftfreq(g, device=dev, dtype=torch.float64)[None, :]
    amp = (kx * kx + ky * ky + 1.0 / scale ** 2) ** (-11.0 / 12.0)
    out = [torch.empty(count, n + 1, n + 1, device=dev, dtype=torch.float64) for _ in shifts]
    for i in range(0, count, 64):
        w = torch.randn(min(64, count - i), g, g, generator=gen, device=dev, dtype=torch.float64)
        f = torch.fft.rfft2(w) * amp
        norm = None
        for s, o in zip(shifts, out):
            x = torch.fft.irfft2(f * torch.exp(-2j * math.pi * kx * s), s=(g, g))
            norm = x.square().mean(dim=(1, 2), keepdim=True).sqrt() if norm is None else norm
            o[i:i + 64] = (rms * x / norm)[:, :n + 1, :n + 1]
    return out


def _system(n, obstruction, m, sigma, a, a2, wind, seed):
    """A running loop's ensemble (n x m) and slopes of N_SLOPES frames, float64: the estimate follows the truth to
    within the ensemble's spread; the observed (second) instant's spread is that of a loop in its steady state."""
    geo = _geo(n, obstruction)
    gen = torch.Generator(device=_device()).manual_seed(seed)
    act = torch.as_tensor(geo.act, device=_device())
    step = wind * FRAME / PITCH
    turb = math.sqrt(3.44 * (L0 / R0) ** (5.0 / 3.0))
    truth = [f[0][act] for f in _fields(gen, 1, n, turb, L0 / PITCH, [k * step for k in range(-1, N_SLOPES)])]
    spread = 0.7 * sigma
    err = _fields(gen, m + 1, n, spread, 8.0)[0][:, act]
    inc = _fields(gen, m, n, 0.15, 20.0)[0][:, act]
    anom = err[:m] - err[:m].mean(dim=0)
    second = (truth[0] + err[m])[:, None] + anom.T
    first = (truth[1] + err[m])[:, None] + ((a + a2) * anom + inc - inc.mean(dim=0)).T
    noise = torch.randn(N_SLOPES, 2 * geo.n_subv, generator=gen, device=_device(), dtype=torch.float64)
    ys = [geo.slopes(truth[k]) + sigma * noise[k] for k in range(N_SLOPES)]
    return torch.cat([first, second]), torch.stack(ys)


def _inputs(case, seed):
    """What a state is made from: per system its keyword arguments, ensembles and slopes (float64)."""
    systems = []
    rows = ([tuple(float(v) for v in s.split(":")) for s in case["mix"].split()] if case["kind"] == "serve"
            else [(case["n_sub"], case["m"], case["sigma"], case["obstruction"])])
    for k, (n, m, sigma, obs) in enumerate(rows):
        n, m, s = int(n), int(m), (int(seed) * 1000 + 17 * k) % (1 << 31)
        q = {"q_white": 0.1} if case["noise"] == "white" else {
            "q_sqrt": _noise_factor(n, obs, case["a"], case["a2"], case["wind"])}
        kw = dict(n_sub=n, m=m, ar1_a=case["a"], ar2_a=case["a2"], sigma=sigma, dom_sub=case["dom_sub"],
                  halo=case["halo"], obstruction=obs, precision=case["precision"], path=case["path"], seed=s,
                  piston=case["piston"], **q)
        X, ys = _system(n, obs, m, sigma, case["a"], case["a2"], case["wind"], s)
        dt = torch.float64 if case["precision"] == "fp64" else torch.float32
        X, ys = X.to(dt), ys.to(dt)
        if case["kind"] == "pair":      # the second filter's ensemble
            X = [X, _system(n, obs, m, sigma, case["a"], case["a2"], case["wind"], s)[0].to(dt).flip(1).contiguous()]
        systems.append((kw, X, ys))
    return systems


def prepare(case, seed):
    systems = _inputs(case, seed)
    if case["kind"] == "serve":
        srv = Server(max_pending=8)
        ids, outs, hosts, start = [], [], [], []
        for kw, X, ys in systems:
            sid = srv.admit(**{k: v for k, v in kw.items() if k != "path"})
            outs.append(srv.set_output(sid, 2))
            hosts.append(ys.cpu().numpy())
            ids.append(sid)
            start.append(X)
        s = {"kind": "serve", "srv": srv, "ids": ids, "outs": outs, "ys": hosts, "start": start, "k": 0}
        _restore(s)
        return s
    kw, X, ys = systems[0]
    if case["kind"] == "pair":
        f = LETKFPair(**{k: v for k, v in kw.items() if k not in ("path", "piston")})
        filters = [f.a, f.b]
    else:
        f = LETKF(**kw)
        filters, X = [f], [X]
    s = {"kind": case["kind"], "f": f, "filters": filters, "ys": [y.contiguous() for y in ys], "start": X, "k": 0,
         "out": torch.empty(f.info.n_act, dtype=f.dtype, device=f.device), "state": [torch.empty_like(x) for x in X]}
    _restore(s)
    torch.cuda.synchronize()
    return s


def _restore(s):
    """The checkpoint's ensembles, the frame counters going on."""
    if s["kind"] == "serve":
        for sid, x in zip(s["ids"], s["start"]):
            _lib.letkf_set_state(_lib.letkf_server_context(s["srv"].srv, sid), x.data_ptr(), 2 * s["k"])
        torch.cuda.synchronize()    # a server's streams are its own
    else:
        for g, x in zip(s["filters"], s["start"]):
            g.set_state(x, s["k"])


def run(s):
    k = s["k"]
    if k and k % RESTART == 0:
        _restore(s)
    s["k"] = k + 1
    if s["kind"] == "serve":
        srv = s["srv"]
        for j in (2 * k, 2 * k + 1):
            for sid, y in zip(s["ids"], s["ys"]):
                srv.submit(sid, y[j % N_SLOPES])
            srv.pump()
        srv.drain()
        srv.records()
        return {"predictions": s["outs"], "ensembles": [srv.state(sid)[0] for sid in s["ids"]]}
    s["f"].step(s["ys"][k % N_SLOPES], out=s["out"])
    for g, x in zip(s["filters"], s["state"]):
        g.get_state(out=x)
    return {"prediction": s["out"], "ensembles": s["state"]}


# ---- the work of a pass ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _tables(n, obstruction, dom_sub, halo):
    return tuple((len(o), 2 * len(s)) for o, s in _geo(n, obstruction).domains(dom_sub, halo))


def _frame_work(n, obs, m, case):
    geo = _geo(n, obs)
    eb = 8 if case["precision"] == "fp64" else 4
    doms = ((geo.n_act, 2 * geo.n_subv),) if case["path"] == "global" else _tables(n, obs, case["dom_sub"], case["halo"])
    flops, na = 0.0, geo.n_act
    for own, p in doms:
        if p:
            q = min(p, m)           # Gram, symmetric matrix function, rows times transform
            flops += 2.0 * m * p * q + 4.0 * q ** 3 + 2.0 * 2 * own * m * q
    nbytes = 2 * 2 * na * m * eb + 2 * geo.n_subv * eb + na * eb    # ensemble in and out, slopes, prediction
    if case["noise"] == "dense":
        flops += 1.0 * na * na * m
        nbytes += na * (na + 1) / 2 * (2 if case["precision"] == "mixed" else eb)
    return nbytes, flops, 2 * na * m * eb


def work(case):
    if case["kind"] == "serve":
        nbytes = flops = 0.0
        for s in case["mix"].split():
            n, m, _, obs = (float(v) for v in s.split(":"))
            b, f, _ = _frame_work(int(n), obs, int(m), case)
            nbytes, flops = nbytes + 2 * b, flops + 2 * f
        return {"bytes": nbytes, "flops": flops}
    b, f, _ = _frame_work(case["n_sub"], case["obstruction"], case["m"], case)
    k = 2 if case["kind"] == "pair" else 1
    return {"bytes": k * b, "flops": k * f}


# ---- the same frames in 64 bits -------------------------------------------------------------------

def _normals(seed, frame, m, count):
    """Philox4x32-10 and Box-Muller normals (count, m): counter (j // 4, member, frame, 1), key = seed."""
    nq = (count + 3) // 4
    mask = np.uint64(0xFFFFFFFF)
    shape = (nq, m)
    c = [np.broadcast_to(np.arange(nq, dtype=np.uint64)[:, None], shape), np.broadcast_to(np.arange(m, dtype=np.uint64), shape),
         np.full(shape, frame, dtype=np.uint64), np.full(shape, 1, dtype=np.uint64)]
    k = [np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)]
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k[0], p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ k[1], p0 & mask]
        k = [(k[0] + np.uint64(0x9E3779B9)) & mask, (k[1] + np.uint64(0xBB67AE85)) & mask]
    u = [(v.astype(np.float64) + 0.5) / 4294967296.0 for v in c]
    z = []
    for i in (0, 2):
        r, t = np.sqrt(-2.0 * np.log(u[i])), 2.0 * np.pi * u[i + 1]
        z += [r * np.cos(t), r * np.sin(t)]
    return np.stack(z, axis=1).reshape(4 * nq, m)[:count]


def _transform(Yp, d, sigma):
    c = Yp.shape[1] - 1.0
    lam, U = np.linalg.eigh(c * np.eye(Yp.shape[1]) + Yp.T @ Yp / sigma ** 2)
    w = U @ ((U.T @ (Yp.T @ d)) / lam) / sigma ** 2
    return w[:, None] + (U * np.sqrt(c / lam)) @ U.T


def _pistons(geo, doms, x, y):
    """Least-squares piston per domain from the slope residual of x, no piston added per group of domains."""
    owner = np.empty(geo.n_act, dtype=np.int64)
    for l, (own, _) in enumerate(doms):
        owner[own] = l
    P = np.zeros((geo.n_act, len(doms)))
    P[np.arange(geo.n_act), owner] = 1.0
    DP = geo.slopes(P)
    delta = np.linalg.lstsq(DP.T @ DP, DP.T @ (y - geo.slopes(x)), rcond=1e-10)[0]
    group = np.arange(len(doms))
    links = np.argwhere(np.abs(DP).T @ np.abs(DP) > 0)
    while True:
        low = group.copy()
        np.minimum.at(low, links[:, 0], group[links[:, 1]])
        if np.array_equal(low, group):
            break
        group = low
    size = P.sum(axis=0)
    for g in np.unique(group):
        at = group == g
        delta[at] -= size[at] @ delta[at] / size[at].sum()
    return delta[owner]


def _exact_frames(kw, X, ys, frames, offset=0):
    geo = _geo(kw["n_sub"], kw["obstruction"])
    na, m = geo.n_act, kw["m"]
    doms = ([(np.arange(na), np.arange(geo.n_subv))] if kw["path"] == "global"
            else geo.domains(kw["dom_sub"], kw["halo"], offset))
    preds = []
    for k in range(frames):
        y = ys[k % N_SLOPES]
        mean = X.mean(axis=1, keepdims=True)
        Xp, Y = X - mean, geo.slopes(X[na:])
        d = y - Y.mean(axis=1)
        Yp = Y - Y.mean(axis=1, keepdims=True)
        Xa = X.copy()
        for own, sub in doms:
            if len(sub):
                obs = np.concatenate([sub, geo.n_subv + sub])
                rows = np.concatenate([own, na + own])
                Xa[rows] = mean[rows] + Xp[rows] @ _transform(Yp[obs], d[obs], kw["sigma"])
        z = _normals(kw["seed"], k, m, na)
        v = kw["q_sqrt"] @ z if "q_sqrt" in kw else kw["q_white"] * z
        X = np.concatenate([kw["ar1_a"] * Xa[:na] + kw["ar2_a"] * Xa[na:] + v, Xa[:na]])
        x = X[:na].mean(axis=1)
        if kw["piston"] != "off":
            s = _pistons(geo, doms, x, y)
            x = x + s
            if kw["piston"] == "in_loop":
                X = X + np.concatenate([s, s])[:, None]
        preds.append(x)
    return preds, X


def exact(case, seed):
    systems = _inputs(case, seed)
    preds, states = [], []
    frames = 2 if case["kind"] == "serve" else 1
    for kw, X, ys in systems:
        ys = ys.double().cpu().numpy()
        if case["kind"] == "pair":
            each = [_exact_frames(dict(kw, seed=kw["seed"] + j), x.double().cpu().numpy(), ys, 1, o)
                    for j, (x, o) in enumerate(zip(X, (0, kw["dom_sub"] // 2)))]
            return {"prediction": 0.5 * (each[0][0][0] + each[1][0][0]), "ensembles": [e[1] for e in each]}
        p, x = _exact_frames(kw, X.double().cpu().numpy(), ys, frames)
        preds.append(np.stack(p))
        states.append(x)
    if case["kind"] == "serve":
        return {"predictions": preds, "ensembles": states}
    return {"prediction": preds[0][0], "ensembles": states}
