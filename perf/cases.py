"""The work that a user of the hydro library has it do, as cases that can be timed.

A case is one pass through the public entry points (``Hydro.step``,
``Hydro.step_rungs``, the staged calls, the starting-pressure network) on one
of the problems of this repository: the jittered lattice wave, the Sod tube,
the Sedov blast, the clustered log-normal box and many independent boxes in
one launch.  The generators below lay the particles down on the GPU from the
seed alone; every lattice carries a jitter of 1e-3 spacings.

A pass of ``step`` starts from the prepared state (one device copy, as a
restarted or repeated step does), so that every pass does the same work; the
smoothing lengths of that state are the converged ones that a running
simulation carries from its last step, kept in single precision as a snapshot
stores them.

``exact`` restates the step in plain torch in 64 bits: pair sums over an
explicit pair list, none of the library's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_12243_gb300 import hydro

FIELDS = ("x", "y", "z", "m", "px", "py", "pz", "E", "U", "h", "omega")
DEV = "cuda"
F64 = torch.float64
NTRAIN = 12 * 64 + 64 + 64 * 64 + 64 + 64 + 1   # trainable parameters of the network

# launch parameters a program saved from hydro_autotune on a large clustered
# box (list radius 1.05 h, 128 slots)
SAVED_TUNING = dict(search_margin=1.05, nbr_slots=128, grad_min_ctas=5, flux_min_ctas=4,
                    flux_queue=1, grad_rank=1)


def _case(name, kind, ic, n, **kw):
    c = dict(name=name, kind=kind, ic=ic, n=n, precision="fp64", scheme="mfv", riemann="exact",
             kernel="wendland", n_ngb=32.0, gamma=5.0 / 3.0, tuned=False, gravity=False,
             sorted=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest step: a test-sized box, all launches and latency
        _case("wave_16_mixed", "step", "wave", 16, precision="mixed"),
        # the plain step of the method's first configuration, 32^3 with HLLC
        _case("wave_32_fp64_hllc", "step", "wave", 32, riemann="hllc"),
        # the shock tube at its full 1,067,742 particles, with a saved tuning
        _case("sod_78_mixed", "step", "sod", 78, precision="mixed", tuned=True),
        # the same tube in the plain FP64 step that the mixed one is judged by, MFM
        _case("sod_78_fp64_mfm", "step", "sod", 78, scheme="mfm"),
        # the clustered box of 2^24 particles kept in the library's own order
        _case("lognormal_16m_mixed", "step", "lognormal", 1 << 24, precision="mixed", tuned=True,
              sorted=True),
        # a clustered box in the default (FP64) precision, an odd number of
        # particles in the caller's arbitrary order
        _case("lognormal_300k_fp64", "step", "lognormal", 300_007),
        # the blast at its full 128^3, MFM, default launch parameters
        _case("sedov_128_mixed_mfm", "step", "sedov", 128, precision="mixed", scheme="mfm"),
        # 512 boxes of 4k to 64k particles of all generators in one launch
        _case("batch_512_mixed", "step", "batch", 512, precision="mixed", tuned=True),
        # a clustered box with the external acceleration a galaxy run adds
        _case("lognormal_500k_gravity", "step", "lognormal", 500_009, precision="mixed",
              gravity=True),
        # one base step with individual timesteps (the blast's deep rungs)
        _case("rungs_sedov_48_mixed", "rungs", "sedov", 48, precision="mixed"),
        # the stages one by one with their lists and gradients handed out:
        # the paper's setup (cubic spline, 64 neighbours, gamma 1.4), FP64
        _case("stages_43_fp64_cubic", "stages", "wave", 43, kernel="cubic", n_ngb=64.0, gamma=1.4),
        # training the starting-pressure network further on recorded faces
        # (forward, backward, Adam) and using it on them
        _case("train_faces_262k", "train", "faces", 262_144, precision="mixed", steps=64,
              batch=2048),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["step"] * 8 + ["rungs", "stages", "stages", "train"])
    if kind == "train":
        return _anon(_case("", "train", "faces", int(_log(rng, 3000, 262_000)), precision="mixed",
                           steps=rng.randrange(8, 64), batch=int(_log(rng, 500, 2048))))
    precision = rng.choice(["fp64", "mixed", "mixed"])
    kw = dict(precision=precision, scheme=rng.choice(["mfv", "mfm"]),
              riemann=rng.choice(["exact", "exact", "hllc"]))
    if kind == "rungs":
        return _anon(_case("", "rungs", "sedov", 2 * int(_log(rng, 8, 23)), **kw))
    if kind == "stages":
        return _anon(_case("", "stages", "wave", int(_log(rng, 12, 56)), kernel=rng.choice(
            ["cubic", "wendland"]), n_ngb=rng.choice([32.0, 64.0]), gamma=rng.choice(
            [1.4, 5.0 / 3.0]), **kw))
    ic = rng.choice(["wave", "sod", "lognormal", "lognormal", "sedov", "batch"])
    big = precision == "mixed"
    n = {"wave": lambda: int(_log(rng, 9, 120 if big else 60)),
         "sod": lambda: 2 * int(_log(rng, 6, 38 if big else 20)),
         "lognormal": lambda: int(_log(rng, 5000, 4_000_000 if big else 400_000)),
         "sedov": lambda: 2 * int(_log(rng, 6, 60 if big else 28)),
         "batch": lambda: int(_log(rng, 2, 300 if big else 12))}[ic]()
    return _anon(_case("", "step", ic, n, tuned=big and rng.random() < 0.5,
                       sorted=ic != "batch" and rng.random() < 0.3,
                       gravity=ic in ("lognormal", "wave") and rng.random() < 0.2, **kw))


def _anon(c):
    del c["name"]
    return c


# ---------------------------------------------------------------- generators
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _h_guess(nd, n_ngb):
    return (3.0 * n_ngb / (4.0 * math.pi * nd)) ** (1.0 / 3.0)


def _lattice(nx, ny, nz, a, x0, g):
    ax = [(torch.arange(k, device=DEV, dtype=F64) + 0.5) * a for k in (nx, ny, nz)]
    p = torch.stack(torch.meshgrid(*ax, indexing="ij")).reshape(3, -1)
    p[0] += x0
    return p + (torch.rand(p.shape, generator=g, device=DEV, dtype=F64) * 2 - 1) * (1e-3 * a)


def _pack(pos, L, m, v, u, h):
    L = torch.as_tensor(L, dtype=F64, device=DEV)[:, None]
    pos = torch.remainder(pos, L)
    pos = torch.where(pos >= L, pos - L, pos)
    U = m * u
    E = U + 0.5 * m * (v * v).sum(0)
    return torch.cat([pos, m[None], m * v, E[None], U[None], h[None], torch.zeros_like(h)[None]])


def _wave(n, g, gamma, n_ngb):
    a = 1.0 / n
    pos = _lattice(n, n, n, a, 0.0, g)
    rho = 1.0 + 0.1 * torch.sin(2.0 * math.pi * pos[0])
    h = torch.full_like(rho, _h_guess(1.0 / a ** 3, n_ngb))
    return _pack(pos, (1.0, 1.0, 1.0), rho * a ** 3, torch.zeros_like(pos),
                 1.0 / ((gamma - 1.0) * rho), h), (1.0, 1.0, 1.0)


def _sod(n, g, gamma, n_ngb):
    a = 1.0 / n
    left = _lattice(2 * n, n, n, a, 0.0, g)
    right = _lattice(n, n // 2, n // 2, 2 * a, 2.0, g)
    pos = torch.cat([left, right], 1)
    isl = torch.arange(pos.shape[1], device=DEV) < left.shape[1]
    one = torch.ones_like(pos[0])
    rho = torch.where(isl, one, one * 0.125)
    p = torch.where(isl, one, one * 0.1)
    h = _h_guess(rho / a ** 3, n_ngb)
    return _pack(pos, (4.0, 1.0, 1.0), one * a ** 3, torch.zeros_like(pos),
                 p / ((gamma - 1.0) * rho), h), (4.0, 1.0, 1.0)


def _sedov(n, g, gamma, n_ngb):
    a = 1.0 / n
    pos = _lattice(n, n, n, a, 0.0, g)
    r = (pos - 0.5).square().sum(0).sqrt()
    q = (r / (math.sqrt(19.0) / 2.0 * a)).clamp(max=1.0)
    w = (1 - q) ** 4 * (1 + 4 * q)
    m = torch.full_like(r, a ** 3)
    u = 1e-6 / (gamma - 1.0) + w / w.sum() / m
    return _pack(pos, (1.0, 1.0, 1.0), m, torch.zeros_like(pos), u,
                 torch.full_like(r, _h_guess(1.0 / a ** 3, n_ngb))), (1.0, 1.0, 1.0)


def _lognormal(N, g, gamma, n_ngb, grid=None):
    if grid is None:
        grid = int(min(256, max(16, 2 ** round(math.log2(N ** (1.0 / 3.0))))))
    k = torch.fft.fftfreq(grid, device=DEV, dtype=F64) * grid
    kk = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :grid // 2 + 1] ** 2).sqrt()
    amp = torch.where(kk > 0, 1.0 / kk.clamp(min=0.5), torch.zeros_like(kk))
    f = torch.randn((grid, grid, grid), generator=g, device=DEV, dtype=F64)
    f = torch.fft.irfftn(torch.fft.rfftn(f) * amp, s=(grid, grid, grid))
    f = (f - f.mean()) / f.std()
    s = math.log(1e4) / float(f.max() - f.min())
    delta = torch.exp(s * f - 0.5 * s * s).reshape(-1)
    cdf = torch.cumsum(delta, 0)
    cell = torch.searchsorted(cdf, torch.rand(N, generator=g, device=DEV, dtype=F64) * cdf[-1])
    cell.clamp_(max=grid ** 3 - 1)
    ijk = torch.stack([cell // (grid * grid), (cell // grid) % grid, cell % grid])
    pos = (ijk + torch.rand((3, N), generator=g, device=DEV, dtype=F64)) / grid
    rho = delta[cell] / delta.mean()
    cs_shape = rho ** ((gamma - 1.0) / 2.0)
    K = 1.0 / (gamma * cs_shape.mean() ** 2)
    p = K * rho ** gamma
    v = torch.randn((3, N), generator=g, device=DEV, dtype=F64) * 0.1 * (gamma * p / rho).sqrt()
    return _pack(pos, (1.0, 1.0, 1.0), torch.full_like(rho, 1.0 / N), v,
                 p / ((gamma - 1.0) * rho), _h_guess(rho * N, n_ngb)), (1.0, 1.0, 1.0)


def _batch(nbox, g, gamma, n_ngb):
    # (the sizes belong to the problem, the particles to the seed)
    u = np.random.default_rng(nbox).random(nbox)
    sizes = np.exp(math.log(4096) + u * math.log(16)).astype(np.int64)
    parts, lens = [], []
    for k in range(nbox):
        if k % 3 == 0:
            b, L = _wave(max(4, round(sizes[k] ** (1.0 / 3.0))), g, gamma, n_ngb)
        elif k % 3 == 1:
            b, L = _sod(max(12, 2 * round((sizes[k] / 2.25) ** (1.0 / 3.0) / 2.0)), g, gamma, n_ngb)
        else:
            b, L = _lognormal(int(sizes[k]), g, gamma, n_ngb, grid=16)
        parts.append(b)
        lens.append(L)
    off = np.concatenate([[0], np.cumsum([b.shape[1] for b in parts])]).astype(np.int64)
    return torch.cat(parts, 1), lens, off


def _initial(case, seed):
    """(state [11, n], box offsets, box lengths) of the generator."""
    g = _gen(seed)
    make = {"wave": _wave, "sod": _sod, "sedov": _sedov, "lognormal": _lognormal}
    if case["ic"] == "batch":
        st, lens, off = _batch(case["n"], g, case["gamma"], case["n_ngb"])
        return st, off, np.asarray(lens, dtype=np.float64)
    st, L = make[case["ic"]](case["n"], g, case["gamma"], case["n_ngb"])
    if case["kind"] == "stages":   # a moving, disordered state: the lattice long after its start
        n = st.shape[1]
        st[:3] += (torch.rand((3, n), generator=g, device=DEV, dtype=F64) - 0.5) * (0.4 / case["n"])
        v = torch.randn((3, n), generator=g, device=DEV, dtype=F64) * 0.1
        st = _pack(st[:3], L, st[3], v, st[8] / st[3], st[9])
    return st, np.array([0, st.shape[1]], dtype=np.int64), np.asarray([L], dtype=np.float64)


def _gravity(st, seed):
    g = _gen(seed + 77)
    return torch.randn((st.shape[1], 3), generator=g, device=DEV, dtype=F64)


def _views(buf):
    return {k: buf[i] for i, k in enumerate(FIELDS)}


def _faces(n, seed):
    """n recorded face problems [7, n]: states of shock-dominated flows and
    their star pressure (two-shock faces among them)."""
    g = _gen(seed)
    r = torch.rand((5, n), generator=g, device=DEV, dtype=F64)
    rl, pl = torch.exp(6 * r[0] - 3), torch.exp(6 * r[1] - 3)
    rr, pr = rl * torch.exp(2 * r[2] - 1), pl * torch.exp(4 * r[3] - 2)
    cl, cr = (5 / 3 * pl / rl).sqrt(), (5 / 3 * pr / rr).sqrt()
    du = (2.5 * r[4] - 2.0) * torch.minimum(cl, cr)
    ul, ur = -0.5 * du, 0.5 * du
    ps, _ = _star(5.0 / 3.0, rl, ul, pl, cl, rr, ur, pr, cr)
    return torch.stack([rl, ul, pl, rr, ur, pr, ps]).float().contiguous()


# ------------------------------------------------------------- prepare, run
def _config(case, **kw):
    return hydro.default_config(gamma=case["gamma"], precision=case["precision"],
                                scheme=case["scheme"], riemann=case["riemann"],
                                kernel=case["kernel"], n_ngb=case["n_ngb"],
                                sorted_output=int(case["sorted"]), **kw)


def _must(status, what):
    # (HYDRO_ENCOND: particles still ill-conditioned after every growth
    # round, which the step completes and reports; clustered boxes have some)
    if status not in (0, -5):
        raise RuntimeError(f"{what}: status {status}")


def prepare(case, seed):
    if case["kind"] == "train":
        H = hydro.Hydro(_config(case))
        faces = _faces(case["n"], seed)
        rng = np.random.default_rng(seed)
        H.mlp_train(faces, 1, batch=case["batch"], seed=3)   # initial weights, feature ranges
        w = H.mlp_get()
        w[:NTRAIN] = rng.standard_normal(NTRAIN) * 0.1       # a network that is still to be trained
        return dict(case=case, H=H, faces=faces, weights=w)
    init, off, lens = _initial(case, seed)
    H = hydro.Hydro(_config(case))
    H.set_boxes(off, lens)
    if case["tuned"]:
        H.set_tuning(SAVED_TUNING)
    s = dict(case=case, H=H, buf=torch.empty_like(init), init=init)
    s["st"] = _views(s["buf"])
    if case["gravity"]:
        s["acc"] = _gravity(init, seed)
        H.set_gravity(s["acc"])
    if case["kind"] == "stages":
        s["hs"] = init[9] * 1.3
        s["idx"] = torch.zeros(int(init.shape[1] * case["n_ngb"] * 3), dtype=torch.int32, device=DEV)
        s["dt"] = 0.02 / case["n"]
        return s
    # the step before this one: it leaves the converged smoothing lengths (and
    # the library's order, where the program keeps it)
    s["buf"].copy_(init)
    if case["kind"] == "rungs":
        H.set_gravity(None)
    info = H.step(s["st"], -1.0, check=False)
    _must(info["status"], case["ic"])
    if case["sorted"]:
        perm = H.get_order().long()
        init = init[:, perm].contiguous()
        if case["gravity"]:
            s["acc"] = s["acc"][perm].contiguous()
            H.set_gravity(s["acc"])
    init[9] = s["buf"][9].float().double()
    s["init"] = init
    if case["kind"] == "rungs":
        s["dt0"] = float("%.2e" % (20.0 * info["dt"]))
        s["rung"] = torch.zeros(init.shape[1], dtype=torch.int32, device=DEV)
    return s


def run(s):
    case, H = s["case"], s["H"]
    if case["kind"] == "train":
        H.mlp_load(s["weights"])
        loss = H.mlp_train(s["faces"], case["steps"], batch=case["batch"], lr=1e-3, seed=11)
        return dict(loss=loss, weights=H.mlp_get(), guess=H.mlp_predict(s["faces"]))
    st = s["st"]
    s["buf"].copy_(s["init"])
    if case["kind"] == "stages":
        off, idx = H.build_neighbours(st, s["hs"])
        s["idx"][:idx.numel()].copy_(idx)   # (the program's own list storage)
        H.density(st)
        B, G, A, N = H.gradients(st)
        dQ = H.fluxes(st, B, G, A, s["dt"])
        return dict(off=off, idx=s["idx"], h=st["h"], omega=st["omega"], B=B, G=G, A=A, N=N, dQ=dQ)
    if case["kind"] == "rungs":
        H.step_rungs(st, s["dt0"], s["rung"], check=False)
        return dict(st, rung=s["rung"])
    info = H.step(st, -1.0, check=False)
    return dict(st, dt=info["dt"])


def _particles(case):
    n = case["n"]
    return {"wave": n ** 3, "sedov": n ** 3, "sod": 2 * n ** 3 + n ** 3 // 4, "lognormal": n,
            "batch": 22_000 * n, "faces": n}[case["ic"]]


def work(case):
    """Each particle's ten inputs read and eleven outputs written once; per
    particle the sums over its N neighbours: density (about three Newton
    steps of 20 operations each), gradients (110 per neighbour), and half as
    many faces (about 650 operations each)."""
    n, N = _particles(case), case["n_ngb"]
    if case["kind"] == "train":
        per = 2 * (12 * 64 + 64 * 64 + 64)
        return {"bytes": n * 8 * 4 + 3 * 4 * NTRAIN,
                "flops": per * (3.0 * case["steps"] * case["batch"] + n)}
    flops = n * N * (60 + 110 + 0.5 * 650)
    b = n * 21 * 8
    if case["kind"] == "stages":
        b = n * (21 + 6 + 15 + 5 + 1 + 6 + 1) * 8 + 4 * n * N * 1.3 ** 3
    if case["kind"] == "rungs":   # (the deep rungs hold a few particles: one start per particle)
        b, flops = b + 4 * n, flops
    return {"bytes": float(b), "flops": float(flops)}


# --------------------------------------------- the step in plain 64-bit torch
def _pairs(P, L, h):
    """(i, j, d [3, k], r) of every ordered pair j != i with r < h_i."""
    n = h.numel()
    lo = float(h.min()) * 0.999999
    cls = torch.floor(torch.log2(h / lo)).clamp(min=0).long()
    out = []
    for c in cls.unique().tolist():
        mem = torch.nonzero(cls == c)[:, 0]
        hm = float(h[mem].max())
        M = [max(1, min(512, int(float(l) / hm))) for l in L]
        ci = [torch.floor(P[a] / float(L[a]) * M[a]).long().clamp(0, M[a] - 1) for a in range(3)]
        key = (ci[0] * M[1] + ci[1]) * M[2] + ci[2]
        key_s, order = torch.sort(key)
        ncell = M[0] * M[1] * M[2]
        start = torch.searchsorted(key_s, torch.arange(ncell + 1, device=DEV))
        offs = [range(-1, 2) if M[a] >= 3 else range(M[a]) for a in range(3)]
        chunk = max(1, int(6e7 / (27 * max(1.0, n / ncell))))
        for q in mem.split(chunk):
            for dx in offs[0]:
                for dy in offs[1]:
                    for dz in offs[2]:
                        k = [(ci[a][q] + dd) % M[a] if M[a] >= 3 else torch.full_like(q, dd)
                             for a, dd in enumerate((dx, dy, dz))]
                        cell = (k[0] * M[1] + k[1]) * M[2] + k[2]
                        b, e = start[cell], start[cell + 1]
                        cnt = e - b
                        i = torch.repeat_interleave(q, cnt)
                        if not i.numel():
                            continue
                        first = torch.cumsum(cnt, 0) - cnt
                        t = torch.arange(i.numel(), device=DEV)
                        j = order[t - torch.repeat_interleave(first - b, cnt)]
                        d = P[:, j] - P[:, i]
                        d = d - L[:, None] * torch.round(d / L[:, None])
                        r = d.square().sum(0).sqrt()
                        ok = (r < h[i]) & (i != j)
                        out.append((i[ok], j[ok], d[:, ok], r[ok]))
    return (torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out]),
            torch.cat([o[2] for o in out], 1), torch.cat([o[3] for o in out]))


def _shape(kernel, q):
    t = (1 - q).clamp(min=0)
    if kernel == "wendland":
        return t ** 4 * (1 + 4 * q)
    return torch.where(q <= 0.5, 1 - 6 * q * q + 6 * q ** 3, 2 * t ** 3)


def _slope(kernel, q):   # -q f'(q)
    t = (1 - q).clamp(min=0)
    if kernel == "wendland":
        return 20 * q * q * t ** 3
    return torch.where(q <= 0.5, 12 * q * q - 18 * q ** 3, 6 * q * t * t)


def _norm(kernel, h):
    return (21 / (2 * math.pi) if kernel == "wendland" else 8 / math.pi) / h ** 3


def _sum(n, i, v):
    return torch.zeros(n, dtype=F64, device=DEV).index_add_(0, i, v)


def _density(case, P, L, h0, N):
    """h with (4 pi/3) h^3 sum W = N, and omega = 1 / sum W."""
    n, ker = h0.numel(), case["kernel"]
    Kn = 14.0 if ker == "wendland" else 32.0 / 3.0
    R = h0 * 1.1
    half = 0.5 * float(L.min())
    while True:
        R = R.clamp(max=half)
        i, j, d, r = _pairs(P, L, R)
        g = Kn * (1 + _sum(n, i, _shape(ker, r / R[i]))) - N
        bad = (g <= 0) & (R < half)
        if not bool(bad.any()):
            break
        R = torch.where(bad, R * 1.3, R)
    lo, hi, h = torch.zeros_like(R), R.clone(), torch.minimum(h0, R)
    for _ in range(80):
        q = r / h[i]
        f = 1 + _sum(n, i, _shape(ker, q))
        mq = _sum(n, i, torch.where(q < 1, _slope(ker, q), torch.zeros_like(q)))
        g = Kn * f - N
        lo = torch.where(g < 0, torch.maximum(lo, h), lo)
        hi = torch.where(g > 0, torch.minimum(hi, h), hi)
        hn = h - g * h / (Kn * mq).clamp(min=1e-300)
        near = (hn - h).abs() < 1e-10 * h   # (converged: the bracket's ends are rounding)
        hn = torch.where(((hn > lo) & (hn < hi) | near) & (mq > 0), hn, 0.5 * (lo + hi))
        done = float(((hn - h).abs() / h).max()) < 1e-15
        h = hn
        if done:
            break
    sw = _norm(ker, h) * (1 + _sum(n, i, _shape(ker, r / h[i])))
    k = r < h[i]
    return h, 1 / sw, (i[k], j[k], d[:, k], r[k])


def _primitives(case, st, h, om, acc):
    m, p, E, U = st[3], st[4:7], st[7], st[8]
    ekin = p.square().sum(0) / (2 * m)
    egrav = m * acc.square().sum(1).sqrt() * h if acc is not None else 0.0
    hot = (U > 0.01 * (egrav + ekin)) & (E - ekin > 0)
    therm = torch.where(hot, E - ekin, U)
    return torch.cat([(m / om)[None], p / m, (therm * (case["gamma"] - 1) / om)[None]])


def _extreme(n, i, v, base, mode):
    return base.clone().scatter_reduce_(0, i, v, mode, include_self=True)


def _gradients(case, W, h, om, pr):
    i, j, d, r = pr
    n, ker = h.numel(), case["kernel"]
    w = om[j] * _norm(ker, h)[i] * _shape(ker, r / h[i])
    E = [_sum(n, i, w * d[a] * d[b]) for a, b in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]
    M = torch.stack([E[0], E[1], E[2], E[1], E[3], E[4], E[2], E[4], E[5]], 1).reshape(n, 3, 3)
    c = [E[3] * E[5] - E[4] ** 2, E[4] * E[2] - E[1] * E[5], E[1] * E[4] - E[3] * E[2]]
    det = E[0] * c[0] + E[1] * c[1] + E[2] * c[2]
    B = torch.stack([c[0], c[1], c[2], E[0] * E[5] - E[2] ** 2, E[2] * E[1] - E[0] * E[4],
                     E[0] * E[3] - E[1] ** 2], 1) / det[:, None]
    BM = B[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(n, 3, 3)
    ncond = (M.square().sum((1, 2)) * BM.square().sum((1, 2))).sqrt() / 3
    ncond = torch.where(torch.isfinite(ncond), ncond, torch.full_like(ncond, math.inf))
    G, A = [], []
    beta = (2 * (100.0 / ncond).square().clamp(max=1)).clamp(min=1.0)
    for f in range(5):
        df = W[f][j] - W[f][i]
        S = torch.stack([_sum(n, i, w * df * d[a]) for a in range(3)], 1)
        g = torch.einsum("nab,nb->na", BM, S)
        e = 0.5 * (d * g[i].T).sum(0)
        zero = torch.zeros_like(h)
        dp, dm = _extreme(n, i, e, zero, "amax"), _extreme(n, i, e, zero, "amin")
        mx, mn = _extreme(n, i, df, zero, "amax"), _extreme(n, i, df, zero, "amin")
        inf = torch.full_like(h, math.inf)
        ratio = torch.minimum(torch.where(dp > 0, mx / dp, inf), torch.where(dm < 0, mn / dm, inf))
        G.append(g)
        A.append((beta * ratio).clamp(max=1.0))
    cs = (case["gamma"] * W[4] / W[0]).sqrt()
    wdot = sum(d[a] * (W[1 + a][j] - W[1 + a][i]) for a in range(3)) / r
    vs = _extreme(n, i, cs[i] + cs[j] - wdot.clamp(max=0), torch.zeros_like(h), "amax")
    dt = torch.where(vs > 0, 0.2 * h / vs, torch.full_like(h, math.inf))
    return B, BM, torch.stack(G, 1), torch.stack(A, 1), ncond, dt


def _pair_limit(e, a, b, positive):
    d, mean = (a - b).abs(), 0.5 * (a + b)
    d1, d2 = 0.5 * d, 0.25 * d
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    lox, hix = lo - d1, hi + d1
    if positive:
        lox = torch.where(torch.sign(lox) != torch.sign(lo), lo / (1 + d1 / lo.abs()), lox)
        hix = torch.where(torch.sign(hix) != torch.sign(hi), hi / (1 + d1 / hi.abs()), hix)
    up = torch.maximum(torch.minimum(e, mean + d2), lox)
    dn = torch.minimum(torch.maximum(e, mean - d2), hix)
    return torch.where(a == b, a, torch.where(a < b, up, dn))


def _side(g, p, rk, pk, ck):
    A, Bk = 2 / ((g + 1) * rk), (g - 1) / (g + 1) * pk
    q = (A / (p + Bk)).sqrt()
    t = (p / pk) ** ((g - 1) / (2 * g))
    shock = p > pk
    return (torch.where(shock, (p - pk) * q, 2 * ck / (g - 1) * (t - 1)),
            torch.where(shock, q * (1 - 0.5 * (p - pk) / (Bk + p)), t * ck / (g * p)))


def _star(g, rl, ul, pl, cl, rr, ur, pr, cr):
    """Star pressure and velocity of the exact Riemann problem (no vacuum):
    Newton from the two-rarefaction pressure, which lies on the side of the
    root from which the iteration is monotone."""
    z, du = (g - 1) / (2 * g), ur - ul
    num = (cl + cr - 0.5 * (g - 1) * du).clamp(min=1e-12)
    p = (num / (cl / pl ** z + cr / pr ** z)) ** (1 / z)
    for _ in range(60):
        fl, dl = _side(g, p, rl, pl, cl)
        fr, dr = _side(g, p, rr, pr, cr)
        pn = (p - (fl + fr + du) / (dl + dr)).clamp(min=1e-300)
        done = float(((pn - p).abs() / pn).max()) < 1e-15
        p = pn
        if done:
            break
    fl, _ = _side(g, p, rl, pl, cl)
    fr, _ = _side(g, p, rr, pr, cr)
    return p, 0.5 * (ul + ur) + 0.5 * (fr - fl)


def _sample(g, rl, ul, pl, cl, rr, ur, pr, cr, ps, us):
    left = us >= 0
    s = torch.where(left, 1.0, -1.0)
    rK, pK, cK = torch.where(left, rl, rr), torch.where(left, pl, pr), torch.where(left, cl, cr)
    uK, uS = s * torch.where(left, ul, ur), s * us
    t = ps / pK
    g6 = (g - 1) / (g + 1)
    shock = ps > pK
    sK = uK - cK * ((g + 1) / (2 * g) * t + (g - 1) / (2 * g)).sqrt()
    beyond = torch.where(shock, sK >= 0, uK - cK >= 0)
    cm = cK * t ** ((g - 1) / (2 * g))
    star = shock | (uS - cm <= 0)
    rstar = torch.where(shock, rK * (t + g6) / (g6 * t + 1), rK * t ** (1 / g))
    cc = (2 / (g + 1) + g6 / cK * uK).clamp(min=1e-300)
    rs = torch.where(star, rstar, rK * cc ** (2 / (g - 1)))
    vs = torch.where(star, uS, 2 / (g + 1) * (cK + 0.5 * (g - 1) * uK))
    q = torch.where(star, ps, pK * cc ** (2 * g / (g - 1)))
    rs, vs, q = (torch.where(beyond, a, b) for a, b in ((rK, rs), (uK, vs), (pK, q)))
    return rs, s * vs, q, left


def _hllc(g, mfm, rl, ul, pl, cl, wl, rr, ur, pr, cr, wr, nh):
    ppv = (0.5 * (pl + pr) - 0.125 * (ur - ul) * (rl + rr) * (cl + cr)).clamp(min=0)
    g2 = (g + 1) / (2 * g)
    ql = (1 + g2 * (ppv / pl - 1).clamp(min=0)).sqrt()
    qr = (1 + g2 * (ppv / pr - 1).clamp(min=0)).sqrt()
    sl, sr = ul - cl * ql, ur + cr * qr
    ss = (pr - pl + rl * ul * (sl - ul) - rr * ur * (sr - ur)) / (rl * (sl - ul) - rr * (sr - ur))
    ps = pl + rl * (sl - ul) * (ss - ul)
    if mfm:
        return torch.cat([torch.zeros_like(ps)[None], ps * nh, (ps * ss)[None]])
    left = ss >= 0
    r, u, p = torch.where(left, rl, rr), torch.where(left, ul, ur), torch.where(left, pl, pr)
    sK, w = torch.where(left, sl, sr), torch.where(left, wl, wr)
    E = p / (g - 1) + 0.5 * r * (u * u + w.square().sum(0))
    k = r * (sK - u) / (sK - ss)
    e2 = k * (E / r + (ss - u) * (ss + p / (r * (sK - u))))
    out = torch.where(left, sl >= 0, sr <= 0)
    star = ~out
    fm = r * u + torch.where(star, sK * (k - r), 0.0 * r)
    fn = r * u * u + p + torch.where(star, sK * (k * ss - r * u), 0.0 * r)
    fe = u * (E + p) + torch.where(star, sK * (e2 - E), 0.0 * r)
    return torch.cat([fm[None], fn * nh + fm * w, fe[None]])


def _fluxes(case, W, h, om, BM, G, pr, dt):
    """(dQ [5, n], sum dm r [3, n]): what every particle receives in dt.
    G: the limited gradients [n, 5, 3]."""
    n, g, ker = h.numel(), case["gamma"], case["kernel"]
    mfm = case["scheme"] == "mfm"
    dQ = torch.zeros((5, n), dtype=F64, device=DEV)
    dM = torch.zeros((3, n), dtype=F64, device=DEV)
    i, j, d, r = pr
    own = (i < j) | (r >= h[j])
    i, j, d, r = i[own], j[own], d[:, own], r[own]
    for k in torch.arange(i.numel(), device=DEV).split(2_000_000):
        a, b, x, q = i[k], j[k], d[:, k], r[k]
        wi = _norm(ker, h[a]) * _shape(ker, q / h[a])
        wj = torch.where(q < h[b], _norm(ker, h[b]) * _shape(ker, q / h[b]), 0.0 * q)
        A = (om[a] * om[b]) * (torch.einsum("nab,bn->an", BM[a], x) * wi +
                               torch.einsum("nab,bn->an", BM[b], x) * wj)
        Am = A.square().sum(0).sqrt()
        nh = A / Am
        Wa, Wb, Ga, Gb = W[:, a], W[:, b], G[a], G[b]
        l = Wa + 0.5 * torch.einsum("nfa,an->fn", Ga, x)
        m = Wb - 0.5 * torch.einsum("nfa,an->fn", Gb, x)
        l = torch.stack([_pair_limit(l[f], Wa[f], Wb[f], f in (0, 4)) for f in range(5)])
        m = torch.stack([_pair_limit(m[f], Wb[f], Wa[f], f in (0, 4)) for f in range(5)])
        hdt = 0.5 * dt
        acc = torch.zeros_like(x)
        for s, c, gr in ((l, Wa, Ga), (m, Wb, Gb)):
            div = gr[:, 1, 0] + gr[:, 2, 1] + gr[:, 3, 2]
            ac = hdt * gr[:, 4].T / c[0]
            s[0] -= hdt * c[0] * div
            s[1:4] -= ac
            s[4] -= hdt * g * c[4] * div
            acc = acc + ac
        ok = (l[0] > 0) & (l[4] > 0) & (m[0] > 0) & (m[4] > 0)
        l, m = torch.where(ok, l, Wa), torch.where(ok, m, Wb)
        vf = 0.5 * (Wa[1:4] + Wb[1:4] - acc)
        vl, vr = l[1:4] - vf, m[1:4] - vf
        ul, ur = (vl * nh).sum(0), (vr * nh).sum(0)
        wl, wr = vl - ul * nh, vr - ur * nh
        cl, cr = (g * l[4] / l[0]).sqrt(), (g * m[4] / m[0]).sqrt()
        if case["riemann"] == "hllc":
            F = _hllc(g, mfm, l[0], ul, l[4], cl, wl, m[0], ur, m[4], cr, wr, nh)
        else:
            ps, us = _star(g, l[0], ul, l[4], cl, m[0], ur, m[4], cr)
            if mfm:
                F = torch.cat([torch.zeros_like(ps)[None], ps * nh, (ps * us)[None]])
            else:
                rs, u, p, left = _sample(g, l[0], ul, l[4], cl, m[0], ur, m[4], cr, ps, us)
                w = torch.where(left, wl, wr)
                e = 0.5 * rs * (u * u + w.square().sum(0)) + p / (g - 1)
                F = torch.cat([(rs * u)[None], rs * u * (u * nh + w) + p * nh, (u * (e + p))[None]])
            vac = 2 / (g - 1) * (cl + cr) <= ur - ul
            F = torch.where(vac, 0.0 * F, F)
        Fe = F[4] + (F[1:4] * vf).sum(0) + 0.5 * F[0] * vf.square().sum(0)
        c = dt * Am * torch.cat([F[:1], F[1:4] + F[0] * vf, Fe[None]])
        c = torch.where(Am > 0, c, 0.0 * c)
        dQ.index_add_(1, a, -c)
        dQ.index_add_(1, b, c)
        dM.index_add_(1, a, c[0] * x)
        dM.index_add_(1, b, c[0] * x)
    return dQ, dM


def exact(case, seed):
    """The step (or the stages) in 64 bits; None where it would take long
    (over a million or so particles, many boxes, many sub-steps, training)."""
    if case["kind"] in ("train", "rungs") or case["ic"] == "batch" or _particles(case) > 1_200_000:
        return None
    s = prepare(case, seed)
    st, L = s["init"].clone(), torch.as_tensor(_initial_len(case), dtype=F64, device=DEV)
    acc = s.get("acc")
    s["H"].close()
    P, n = st[:3], st.shape[1]
    N = torch.full((n,), float(case["n_ngb"]), dtype=F64, device=DEV)
    if case["kind"] == "stages":
        h, om, pr = _density(case, P, L, st[9], N)
        W = _primitives(case, st, h, om, None)
        B, BM, G, A, nc, _ = _gradients(case, W, h, om, pr)
        dQ, _ = _fluxes(case, W, h, om, BM, G * A[:, :, None], pr, s["dt"])
        v = W[1:4]
        dU = dQ[4] - (v * dQ[1:4]).sum(0) + 0.5 * v.square().sum(0) * dQ[0]
        return dict(off=None, idx=None, h=h, omega=om, B=B, G=G, A=A, N=nc,
                    dQ=torch.cat([dQ, dU[None]]).T)
    for rnd in range(6):
        h, om, pr = _density(case, P, L, st[9], N)
        W = _primitives(case, st, h, om, acc)
        B, BM, G, A, nc, dti = _gradients(case, W, h, om, pr)
        bad = ~(nc <= 100.0)
        if rnd == 5 or not bool(bad.any()):
            break
        N = torch.where(bad, N * 1.2, N)
    dt = float(dti.min())
    dQ, dM = _fluxes(case, W, h, om, BM, G * A[:, :, None], pr, dt)
    m0, p0, E0, U0 = st[3], st[4:7], st[7], st[8]
    v0 = p0 / m0
    m1, p1, E1 = m0 + dQ[0], p0 + dQ[1:4], E0 + dQ[4]
    U1 = U0 + dQ[4] - (v0 * dQ[1:4]).sum(0) + 0.5 * v0.square().sum(0) * dQ[0]
    if acc is not None:
        a = acc.T
        E1 = E1 + 0.5 * dt * ((p0 + p1) * a).sum(0) + 0.5 * (a * dM).sum(0)
        p1 = p1 + 0.5 * dt * (m0 + m1) * a
    x = torch.remainder(P + 0.5 * dt * (v0 + p1 / m1), L[:, None])
    return dict(zip(FIELDS, [*x, m1, *p1, E1, U1, h, om]), dt=dt)


def _initial_len(case):
    return (4.0, 1.0, 1.0) if case["ic"] == "sod" else (1.0, 1.0, 1.0)
