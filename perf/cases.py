"""Performance cases: the calls a fixed-order NLO program makes of this library.

A program samples phase-space points (its own, or the library's generators), has the
Born, n-body or subtracted real-emission weight of every point evaluated, and unweights
them; a served setup sends batches of many integration channels to the request loop.
The sizes, energies and cuts are those of the repository's benchmark and tests and of the
served stream (batches of 256 to 65,536 points), with ragged sizes in between.  Trees with
gluons are evaluated where they are finite, at resolved gluons, as a program with jet cuts
samples them; the subtracted real takes importance-sampled points (soft and collinear
regions populated down to a technical cut, weights bounded), and flat ones in the headline
batch and in float64.

Weights of a mixed-precision handle are single-precision numbers in float64 words: their
ingredients are float32, points are re-evaluated in float64 where the error would pass
the handle's tolerance (1e-5), and the lane layout, which the library picks by timing on
the first call, moves their last float32 bits from process to process.  The program books
them as float32, as event records do, in order on the stream it runs the library on; weights
of a float64 handle stay float64.

``exact`` restates every result in plain torch and 64 bits: explicit Dirac matrices,
linear gluon polarisations, a memoised colour-ordered recursion or plain Feynman diagrams
with colour tensors from the Gell-Mann matrices, and the FKS formulas.
"""
import itertools
import math

import numpy as np
import torch

import paper_2503_07439_gb300 as me

ALPHA, ALPHA_S, MT = 1.0 / 132.507, 0.118, 173.0
GS, EE = math.sqrt(4.0 * math.pi * ALPHA_S), math.sqrt(4.0 * math.pi * ALPHA)
XI_CUT, DELTA = 0.5, 1.0
XI_MIN, Y_MIN = 1e-3, 1e-4
CF, CA = 4.0 / 3.0, 3.0

# process: final-state masses, default partonic energy [GeV], spin and colour average (with
# the identical-particle factor), float operations of one tree |M|^2 and of one subtracted
# real (helicity sums over one member of each flipped pair, shared gluon currents)
PROCESSES = {
    "ee_uu": ((0.0, 0.0), 100.0, 4.0, 691, 0),
    "ee_uug": ((0.0, 0.0, 0.0), 100.0, 4.0, 2931, 4313),
    "gg_tt": ((MT, MT), 1000.0, 256.0, 2819, 0),
    "gg_ttg": ((MT, MT, 0.0), 1000.0, 256.0, 29394, 37850),
    "gg_ttgg": ((MT, MT, 0.0, 0.0), 2000.0, 512.0, 534011 + 76800, 0),
    "uu_tt": ((MT, MT), 1000.0, 36.0, 1445, 0),
    "uu_ttg": ((MT, MT, 0.0), 1000.0, 36.0, 14687, 17657),
}
BORN_OF = {"ee_uug": "ee_uu", "gg_ttg": "gg_tt", "uu_ttg": "uu_tt"}
SERVED = ("ee_uu", "ee_uug", "gg_tt", "gg_ttg", "gg_ttgg", "uu_ttg")
# analysis cuts: both tops central and hard, or the thrust axis away from the beams
HEAVY_CUTS = {"cut_pt_min": 100.0, "cut_abs_y_max": 1.0}
EE_CUTS = {"cut_abs_cos_axis_max": 0.8, "cut_thrust_max": 0.9}


# ---------------------------------------------------------------- the cases
def _case(op, process, n, precision, name=None, points="flat", cuts=False, sqrt_s=0.0):
    c = {"op": op, "process": process, "n": n, "precision": precision, "points": points, "cuts": cuts,
         "sqrt_s": sqrt_s or PROCESSES[process][1]}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small integration channel of the e+e- -> u ubar n-body term, in the default
        # precision: the cost of a call
        _case("nbody", "ee_uu", 999, "fp64", "nbody_ee_uu_999_fp64"),
        # a request of ordinary size of the subtracted real, as adaptive integrators send them
        _case("real", "gg_ttg", 4099, "mixed", "real_gg_ttg_4099", "fks"),
        # the real part of the e+e- K-factor, with the accumulators read back
        _case("real", "ee_uug", 65536, "mixed", "real_ee_uug_65536", "fks"),
        # leading order: a scan of gg -> t tbar over the partonic energy, 400 to 2000 GeV
        _case("born", "gg_tt", 1 << 20, "mixed", "born_gg_tt_scan_1m", "scan"),
        # the headline workload: a full batch of the gg -> t tbar g subtracted real
        _case("real", "gg_ttg", 1 << 20, "mixed", "real_gg_ttg_1m"),
        # the same in the default precision, a ragged batch (a validation run)
        _case("real", "gg_ttg", 30011, "fp64", "real_gg_ttg_30011_fp64"),
        # the quark channel with analysis cuts on every term, large and ragged
        _case("real", "uu_ttg", 600011, "mixed", "real_uu_ttg_cuts_600011", "fks", cuts=True),
        # the multi-leg tree: 24 colour flows
        _case("born", "gg_ttgg", 1 << 18, "mixed", "born_gg_ttgg_262144", "resolved"),
        # the multi-leg tree in the default precision
        _case("born", "gg_ttgg", 8191, "fp64", "born_gg_ttgg_8191_fp64", "resolved"),
        # points of the next Monte-Carlo iteration, sampled on the device in FKS variables
        _case("sample", "gg_ttg", 500009, "fp64", "sample_gg_ttg_500009", "fks"),
        # event generation: a million weighted points unweighted against their maximum
        dict(op="unweight", process="gg_ttg", n=1 << 20, w_max=0.0, name="unweight_1m"),
        # the request loop: batches of six channels from host memory, all in flight
        dict(op="serve", requests=24, lo=256, hi=65536, precision="mixed", name="serve_24"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["born", "born", "born", "nbody", "real", "real", "real", "real", "sample", "unweight", "serve"])
    if op == "unweight":
        return dict(op="unweight", process="gg_ttg", n=_log_uniform(rng, 1000, 1 << 20),
                    w_max=rng.choice([0.0, rng.uniform(5.0, 40.0)]))
    if op == "serve":
        return dict(op="serve", requests=rng.randint(6, 24), lo=256, hi=_log_uniform(rng, 4096, 65536), precision="mixed")
    precision = "fp64" if op == "sample" else rng.choice(["mixed", "mixed", "fp64"])
    if op == "nbody":
        return _case("nbody", "ee_uu", _log_uniform(rng, 500, 1 << 18), precision, cuts=rng.random() < 0.3)
    if op == "born":
        process = rng.choice(sorted(PROCESSES))
        top = {"gg_ttgg": (1 << 18, 8191), "gg_ttg": (1 << 19, 1 << 16)}.get(process, (1 << 20, 1 << 18))
    else:
        process = rng.choice(sorted(BORN_OF))
        top = (1 << 20, 1 << 16)
    n = _log_uniform(rng, 500, top[0] if precision == "mixed" or op == "sample" else top[1])
    e0 = PROCESSES[process][1]
    sqrt_s = rng.choice([e0, round(e0 * rng.uniform(0.8, 2.0), 1)])
    if op == "born":
        points = "scan" if process == "gg_tt" and rng.random() < 0.5 else _tree_points(process)
    else:
        points = "fks" if precision == "mixed" or op == "sample" and rng.random() < 0.7 else "flat"
    return _case(op, process, n, precision, None, points, op != "sample" and rng.random() < 0.4, sqrt_s)


def _tree_points(process):
    return "resolved" if len(PROCESSES[process][0]) > 2 else "flat"


def _sizes(case):
    """Batch sizes of a served burst: evenly spread over the logarithm of the range."""
    r, lo, hi = case["requests"], case["lo"], case["hi"]
    return [int(lo * (hi / lo) ** (((7 * i) % r + 0.5) / r)) for i in range(r)]


def _served(case):
    """(process, kind, n) of each request: the real processes alternate Born and real."""
    out = []
    for i, n in enumerate(_sizes(case)):
        process = SERVED[i % len(SERVED)]
        real = process in BORN_OF and (i // len(SERVED)) % 4 != 3
        out.append((process, "real_subtracted" if real else "born", n))
    return out


# ---------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _uniforms(count, n, seed):
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    return torch.rand((count, n), generator=g, device=_device(), dtype=torch.float64).clamp_(1e-12, 1.0 - 1e-12)


def _rambo(u, masses, rs):
    """Flat phase space (RAMBO with its massive rescaling) from 4 uniforms per particle:
    momenta [4][n_out][n] and weights."""
    nout, n = len(masses), u.shape[1]
    u = u.reshape(nout, 4, n)
    c, phi, e = 2.0 * u[:, 0] - 1.0, 2.0 * math.pi * u[:, 1], -torch.log(u[:, 2] * u[:, 3])
    s = torch.sqrt(1.0 - c * c)
    q = torch.stack([e, e * s * torch.cos(phi), e * s * torch.sin(phi), e * c])
    Q = q.sum(1)
    M = torch.sqrt(Q[0] ** 2 - (Q[1:] ** 2).sum(0))
    b, g = -Q[1:] / M, Q[0] / M
    bq = (b[:, None] * q[1:]).sum(0)
    k = torch.cat([(g * q[0] + bq)[None],
                   q[1:] + b[:, None] * q[0] + (bq / (1.0 + g))[None] * b[:, None]]) * (rs / M)
    w0 = (2.0 * math.pi) ** (4 - 3 * nout) * (0.5 * math.pi) ** (nout - 1) * rs ** (2 * nout - 4) / (
        math.factorial(nout - 1) * math.factorial(nout - 2))
    w = torch.full((n,), w0, dtype=torch.float64, device=u.device)
    if any(masses):
        m = torch.tensor(masses, dtype=torch.float64, device=u.device)[:, None]
        p = k[0].clone()
        x = torch.full((n,), math.sqrt(max(0.0, 1.0 - (sum(masses) / rs) ** 2)), dtype=torch.float64, device=u.device)
        for _ in range(12):
            en = torch.sqrt(m * m + (x * p) ** 2)
            x = x - (en.sum(0) - rs) / (x * p * p / en).sum(0)
        k = torch.cat([torch.sqrt(m * m + (x * p) ** 2)[None], k[1:] * x])
        w = w0 * _rambo_shape(k, rs)
    return k, w


def _rambo_shape(k, rs):
    """The massive RAMBO weight over the massless volume, as a function of the momenta."""
    ka, nout = torch.sqrt((k[1:] ** 2).sum(0)), k.shape[1]
    return (ka.sum(0) / rs) ** (2 * nout - 3) * (ka / k[0]).prod(0) * rs / (ka * ka / k[0]).sum(0)


def _with_beams(k, rs):
    beams = torch.zeros((4, 2, k.shape[2]), dtype=torch.float64, device=k.device)
    beams[0], beams[3, 0], beams[3, 1] = 0.5 * rs, 0.5 * rs, -0.5 * rs
    return torch.cat([beams, k], 1).contiguous()


def _flat(process, n, rs, seed):
    masses = PROCESSES[process][0]
    k, w = _rambo(_uniforms(4 * len(masses), n, seed), masses, rs)
    return _with_beams(k, rs), w


def _resolved(process, n, rs, seed):
    """Flat points with every gluon a resolved jet: in t tbar + gluons a transverse momentum
    and a mass with any other gluon of at least 2.5 % of the energy, in e+e- a mass with
    each quark of at least 10 %."""
    p, w = _flat(process, n + n // 3 + 64, rs, seed)
    legs = range(p.shape[1])
    partons = [l for l in legs[2:] if l >= 4 or process.startswith("ee")]
    least = (0.1 if process.startswith("ee") else 0.025) * rs
    ok = torch.ones_like(w, dtype=torch.bool)
    for a, b in itertools.combinations(partons, 2):
        q = p[:, a] + p[:, b]
        ok &= (q[0] ** 2 - (q[1:] ** 2).sum(0) >= least ** 2) | (b < 4)
    if not process.startswith("ee"):
        for l in partons:
            ok &= p[1, l] ** 2 + p[2, l] ** 2 >= least ** 2
    return _first(n, ok, p, w)


def _importance(process, n, rs, seed):
    """FKS-sampled points outside a technical cut on the emission's energy fraction and angle
    to either reference direction, beyond which float64 momenta no longer fix the weight."""
    p, w = _sampled(process, list(_uniforms(18, n + n // 8 + 64, seed)), rs)
    k = p[:, 4]
    ok = 2.0 * k[0] >= XI_MIN * rs
    for j in ((2, 3) if process == "ee_uug" else (0, 1)):
        y = (k[1:] * p[1:, j]).sum(0) / (k[0] * torch.sqrt((p[1:, j] ** 2).sum(0)))
        ok &= 1.0 - y >= Y_MIN
    return _first(n, ok, p, w)


def _first(n, ok, p, w):
    at = torch.nonzero(ok)[:n, 0]
    return p[:, :, at].contiguous(), w[at].contiguous()


def _scan(n, seed):
    """gg -> t tbar with the partonic energy uniform in 400 to 2000 GeV, no weights."""
    u = _uniforms(3, n, seed)
    rs, c, phi = 400.0 + 1600.0 * u[0], 2.0 * u[1] - 1.0, 2.0 * math.pi * u[2]
    e, s = 0.5 * rs, torch.sqrt(1.0 - c * c)
    k = e * torch.sqrt(1.0 - (MT / e) ** 2)
    t = torch.stack([e, k * s * torch.cos(phi), k * s * torch.sin(phi), k * c])
    return _with_beams(torch.stack([t, torch.cat([t[:1], -t[1:]])], 1), rs), None


def _weights(n, seed):
    """Weights as an NLO integrand leaves them: a long tail, one in eight negative."""
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    w = torch.exp(1.2 * torch.randn(n, generator=g, device=_device(), dtype=torch.float64))
    return torch.where(torch.rand(n, generator=g, device=_device()) < 0.125, -w, w)


def _inputs(points, process, n, rs, seed):
    if points == "scan":
        return _scan(n, seed)
    return {"fks": _importance, "resolved": _resolved, "flat": _flat}[points](process, n, rs, seed)


def _inputs_of(case, seed):
    return _inputs(case["points"], case["process"], case["n"], case["sqrt_s"], seed)


def _served_inputs(case, seed):
    """(process, kind, momenta, weights) of every request of a served burst."""
    return [(process, kind) + _inputs("fks" if kind == "real_subtracted" else _tree_points(process), process, n,
                                      PROCESSES[process][1], seed + i)
            for i, (process, kind, n) in enumerate(_served(case))]


def _precision(case):
    return me.ME_PREC_MIXED if case["precision"] == "mixed" else me.ME_PREC_FP64


def _cuts(case):
    return {} if not case["cuts"] else EE_CUTS if case["process"].startswith("ee") else HEAVY_CUTS


def _booked(f, state):
    """The weights of one call as the program keeps them (see the top of the file)."""
    if state["stream"] is None:
        return f(state["p"], state["w"])
    with torch.cuda.stream(state["stream"]):
        return f(state["p"], state["w"]).float()


def _own_stream(h):
    """The program's stream, with the handle's work on it."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    h.set_stream(s.cuda_stream)
    return s


def prepare(case, seed):
    op = case["op"]
    if op == "unweight":
        h, w = me.Handle(case["process"]), _weights(case["n"], seed)
        return {"case": case, "h": h, "w": w, "seed": seed, "stream": _own_stream(h)}
    if op == "serve":
        batches = [(process, kind, p.cpu().numpy(), w.cpu().numpy()) for process, kind, p, w in _served_inputs(case, seed)]
        return {"case": case, "server": me.Server(precision=_precision(case)), "batches": batches}
    h = me.Handle(case["process"], precision=_precision(case), **_cuts(case))
    if op == "sample":
        return {"case": case, "h": h, "seed": seed}
    p, w = _inputs_of(case, seed)
    return {"case": case, "h": h, "p": p, "w": w, "stream": _own_stream(h) if case["precision"] == "mixed" else None}


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "unweight":
        w = state["w"]
        with torch.cuda.stream(state["stream"]):
            kept, kw, wm, over = state["h"].unweight(w, case["w_max"], seed=state["seed"])
            # the event weight of every point, 0 for the rejected ones
            return [torch.zeros_like(w).index_add_(0, kept, kw), kept.shape[0], wm, over]
    if op == "serve":
        s = state["server"]
        tickets = [s.submit(process, kind, p, w) for process, kind, p, w in state["batches"]]
        return [s.poll(t)["out"].astype(np.float32) for t in tickets]
    h = state["h"]
    if op == "sample":
        return list((h.generate_fks if case["points"] == "fks" else h.generate_flat)(case["n"], state["seed"], case["sqrt_s"]))
    if op == "born":
        return [_booked(h.born, state)]
    if op == "nbody":
        return [_booked(h.nbody_nlo, state)]
    if case["process"] != "ee_uug":
        return [_booked(h.real_subtracted, state)]
    h.set_accumulators((0.0, 0.0, 0.0))
    out = _booked(h.real_subtracted, state)
    return [out, list(h.accumulators())]


def work(case):
    """Every momentum component and weight read once, every result written once; the float
    operations of the amplitudes (most of a point's arithmetic; a mixed-precision handle
    repeats some of them in float64 for a part of the points)."""
    op = case["op"]
    if op == "unweight":
        # weights in, event weights out; ten rounds of a counter-based generator a point
        return {"bytes": 16.0 * case["n"], "flops": 100.0 * case["n"]}
    if op == "serve":
        parts = [work({"op": "real" if kind == "real_subtracted" else "born", "process": process, "n": n})
                 for process, kind, n in _served(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    masses, _, _, tree, real = PROCESSES[case["process"]]
    legs = len(masses) + 2
    if op == "sample":  # momenta and weight out; random numbers, angles, boosts, densities
        return {"bytes": 8.0 * (4 * legs + 1) * case["n"], "flops": 1500.0 * case["n"]}
    words = 4 * legs + (1 if case.get("points") == "scan" else 2)  # momenta, weight, result
    return {"bytes": 8.0 * words * case["n"], "flops": float(real if op == "real" else tree) * case["n"]}


# ---------------------------------------------------------------- exact: Dirac algebra
def _gammas():
    s = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]], complex)]
    z, one = np.zeros((2, 2), complex), np.eye(2, dtype=complex)
    return np.array([np.block([[z, one], [one, z]])] + [np.block([[z, a], [-a, z]]) for a in s])


GAMMA = _gammas()
METRIC = np.array([1.0, -1.0, -1.0, -1.0])


def _on(a, x):
    return torch.as_tensor(a, dtype=torch.complex128, device=x.device)


def _dot(a, b):
    return a[:, 0] * b[:, 0] - (a[:, 1:] * b[:, 1:]).sum(1)


def _slash(V):
    return torch.einsum("nm,mij->nij", V.to(torch.complex128), _on(GAMMA * METRIC[:, None, None], V))


def _u(p, m):
    """Both u spinors of momentum p [n][4], any spin basis: [n][2][4]."""
    chi = np.array([[1, 0, 1, 0], [0, 1, 0, 1]], complex)
    return torch.einsum("nij,sj->nsi", _slash(p) + m * _on(np.eye(4), p), _on(chi, p)) / torch.sqrt(2.0 * (p[:, 0] + m))[:, None, None]


def _v(p, m):
    chi = np.array([[1, 0, -1, 0], [0, 1, 0, -1]], complex)
    return torch.einsum("nij,sj->nsi", m * _on(np.eye(4), p) - _slash(p), _on(chi, p)) / torch.sqrt(2.0 * (p[:, 0] + m))[:, None, None]


def _bar(s):
    return s.conj() @ _on(GAMMA[0], s)


def _current(r, c):
    """r gamma^mu c for every pair of spinors: [n][2][2][4]."""
    return torch.einsum("nsi,mij,ntj->nstm", r, _on(GAMMA, r), c)


def _polarisations(k):
    """Two real transverse polarisation vectors of a gluon k [n][4]."""
    d = k[:, 1:] / torch.sqrt((k[:, 1:] ** 2).sum(1))[:, None]
    a = torch.zeros_like(d)
    a[:, 0] = 1.0
    a[d[:, 0].abs() > 0.7] = torch.tensor([0.0, 1.0, 0.0], dtype=d.dtype, device=d.device)
    e1 = a - (a * d).sum(1)[:, None] * d
    e1 = e1 / torch.sqrt((e1 ** 2).sum(1))[:, None]
    e2 = torch.cross(d, e1, dim=1)
    zero = torch.zeros_like(e1[:, :1])
    return [torch.cat([zero, e], 1).to(torch.complex128) for e in (e1, e2)]


# ---------------------------------------------------------------- exact: colour
def _generators():
    lam = np.zeros((8, 3, 3), complex)
    for i, (a, b) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        lam[i][a, b] = lam[i][b, a] = 1.0
        lam[i + 1][a, b], lam[i + 1][b, a] = -1j, 1j
    lam[[2, 3, 4, 5, 6, 7]] = lam[[7, 3, 4, 5, 6, 2]]  # pairs landed on 0-1, 3-4, 5-6
    lam[2], lam[7] = np.diag([1.0, -1.0, 0.0]), np.diag([1.0, 1.0, -2.0]) / math.sqrt(3.0)
    T = 0.5 * lam
    f = np.einsum("abij,cji->abc", np.einsum("aij,bjk->abik", T, T) - np.einsum("bij,ajk->abik", T, T), T) * -2j
    return T, f.real


T, F = _generators()


def _colour_basis(process):
    """Colour tensors of a process's amplitudes, and the representation of every axis."""
    eye = np.eye(3)
    if process.startswith("gg"):
        ng = len(PROCESSES[process][0])
        out = []
        for perm in itertools.permutations(range(ng)):
            t = eye.astype(complex)
            for _ in perm:  # gluon axes in the order of the string, then sorted
                t = np.tensordot(t, T, axes=([t.ndim - 1], [1]))
                t = np.moveaxis(t, -2, t.ndim - 3) if t.ndim > 3 else np.moveaxis(t, 1, 0)
            axes = [perm.index(g) for g in range(ng)]
            out.append(np.transpose(t, axes + [ng, ng + 1]))
        return out, ["adj"] * ng + ["fund", "anti"]
    if process == "uu_tt":  # axes u, ubar, t, tbar
        return [np.einsum("aij,alk->klij", T, T)], ["anti", "fund", "fund", "anti"]
    if process == "uu_ttg":  # gluon off t, tbar, ubar, u, and the three-gluon vertex
        tt = [np.einsum("aim,bmj,blk->klija", T, T, T), np.einsum("bim,amj,blk->klija", T, T, T),
              np.einsum("bij,alm,bmk->klija", T, T, T), np.einsum("bij,blm,amk->klija", T, T, T),
              np.einsum("bca,cij,blk->klija", F.astype(complex), T, T)]
        return tt, ["anti", "fund", "fund", "anti", "adj"]
    return ([eye] if process == "ee_uu" else [np.einsum("aij->ija", T)]), ["fund", "anti", "adj"]


def _charge(t, axis, rep, a):
    m = T[a] if rep == "fund" else -T[a].T if rep == "anti" else -1j * F[a]
    return np.moveaxis(np.tensordot(m, t, axes=([1], [axis])), 0, axis)


def _gram(process):
    t, _ = _colour_basis(process)
    return np.array([[np.vdot(x, y) for y in t] for x in t])


def _gram_correlated(process, k, l):
    t, rep = _colour_basis(process)
    return np.array([[sum(np.vdot(_charge(x, k, rep[k], a), _charge(y, l, rep[l], a)) for a in range(8)) for y in t] for x in t])


# ---------------------------------------------------------------- exact: amplitudes
def _amp_ttng(p, pol):
    """Colour-ordered t tbar + gluon amplitudes, [n][orderings][spins of t, tbar]."""
    legs = [0, 1] + list(range(4, p.shape[1]))
    q = [p[:, l] * (-1.0 if l < 2 else 1.0) for l in legs]
    pt = p[:, 2]
    J, U = {}, {(): _bar(_u(pt, MT))}
    pairs = {(i, j): _dot(q[i], q[j]) for i in range(len(q)) for j in range(i + 1, len(q))}

    def inv2(s):
        return 2.0 * sum(pairs[tuple(sorted(x))] for x in itertools.combinations(s, 2))

    def mom(s):
        return sum(q[i] for i in s)

    def cur(s):
        if len(s) == 1:
            return pol[s[0]]
        if s not in J:
            tot = 0.0
            for c in range(1, len(s)):
                a, b, qa, qb = cur(s[:c]), cur(s[c:]), mom(s[:c]), mom(s[c:])
                tot = tot + GS * (2.0 * _dot(qb, a)[:, None] * b - 2.0 * _dot(qa, b)[:, None] * a + (qa - qb) * _dot(a, b)[:, None])
            for c in range(1, len(s) - 1):
                for d in range(c + 1, len(s)):
                    a, b, e = cur(s[:c]), cur(s[c:d]), cur(s[d:])
                    tot = tot + GS * GS * (2.0 * _dot(a, e)[:, None] * b - _dot(a, b)[:, None] * e - _dot(b, e)[:, None] * a)
            J[s] = tot / inv2(s)[:, None]
        return J[s]

    def vertex(s):
        return sum(line(s[:c]) @ _slash(cur(s[c:])) for c in range(len(s)))

    def line(s):
        if s not in U:
            Q = mom(s)
            den = 2.0 * _dot(pt, Q) + (inv2(s) if len(s) > 1 else 0.0)
            U[s] = -GS * (vertex(s) @ (_slash(pt + Q) + MT * _on(np.eye(4), p))) / den[:, None, None]
        return U[s]

    v = _v(p[:, 3], MT)
    return torch.stack([GS * torch.einsum("nsi,nti->nst", vertex(s), v) for s in itertools.permutations(range(len(q)))], 1)


def _amp_uu(p, pol):
    """u ubar -> t tbar (g): one amplitude per colour tensor, spins of all quarks."""
    uu, vu, ut, vt = _u(p[:, 0], 0.0), _bar(_v(p[:, 1], 0.0)), _bar(_u(p[:, 2], MT)), _v(p[:, 3], MT)

    def close(light, heavy, s):  # [n][2 ubar][2 u][4] and [n][2 t][2 tbar][4]
        return GS * GS * torch.einsum("nabm,ncdm,m->nabcd", light, heavy, _on(METRIC, p)) / s[:, None, None, None, None]

    s01, t23 = p[:, 0] + p[:, 1], p[:, 2] + p[:, 3]
    if not pol:
        return close(_current(vu, uu), _current(ut, vt), _dot(s01, s01))[:, None]
    g, e, one = p[:, 4], _slash(pol[0]), _on(np.eye(4), p)

    def prop(Q, m, den):
        return (_slash(Q) + m * one) / den[:, None, None]

    light, heavy, s, t = _current(vu, uu), _current(ut, vt), _dot(s01, s01), _dot(t23, t23)
    d = [_dot(p[:, i], g) for i in range(4)]
    r1 = -GS * ut @ e @ prop(p[:, 2] + g, MT, 2.0 * d[2])
    c2 = -GS * torch.einsum("nij,njk,nsk->nsi", prop(-(p[:, 3] + g), MT, 2.0 * d[3]), e, vt)
    r3 = -GS * vu @ e @ prop(-(p[:, 1] - g), 0.0, -2.0 * d[1])
    c4 = -GS * torch.einsum("nij,njk,nsk->nsi", prop(p[:, 0] - g, 0.0, -2.0 * d[0]), e, uu)
    # three-gluon vertex between the light current (momentum s01 in) and the heavy one
    m = METRIC

    def along(k, c):
        return torch.einsum("nm,nabm,m->nab", k.to(torch.complex128), c, _on(m, p))

    le = torch.einsum("nabm,nm,m->nab", light, pol[0], _on(m, p))
    he = torch.einsum("nabm,nm,m->nab", heavy, pol[0], _on(m, p))
    lh = torch.einsum("nabm,ncdm,m->nabcd", light, heavy, _on(m, p))
    ke = [_dot(k, pol[0]) for k in (s01, t23)]
    k1, k2, k3 = s01, -t23, -g  # incoming: light, heavy, gluon
    tri = (torch.einsum("nabcd,n->nabcd", lh, ke[0] + ke[1])  # (k1 - k2).e (l.h)
           + torch.einsum("ncd,nab->nabcd", he, along(k2 - k3, light))
           + torch.einsum("nab,ncd->nabcd", le, along(k3 - k1, heavy)))
    five = -1j * GS ** 3 * tri / (s * t)[:, None, None, None, None]
    return torch.stack([close(light, _current(r1, vt), s), close(light, _current(ut, c2), s),
                        close(_current(r3, uu), heavy, t), close(_current(vu, c4), heavy, t), five], 1)


def _amp_ee(p, pol):
    s01 = p[:, 0] + p[:, 1]
    light = _current(_bar(_v(p[:, 0], 0.0)), _u(p[:, 1], 0.0)) * (-EE / _dot(s01, s01))[:, None, None, None]
    ub, v, eq = _bar(_u(p[:, 2], 0.0)), _v(p[:, 3], 0.0), EE * 2.0 / 3.0
    if not pol:
        cur = _current(ub, v)
    else:
        e, g = _slash(pol[0]), p[:, 4]
        r = -GS * ub @ e @ _slash(p[:, 2] + g) / (2.0 * _dot(p[:, 2], g))[:, None, None]
        c = GS * torch.einsum("nij,njk,nsk->nsi", _slash(p[:, 3] + g), e, v) / (2.0 * _dot(p[:, 3], g))[:, None, None]
        cur = _current(r, v) + _current(ub, c)
    return eq * torch.einsum("nabm,ncdm,m->nabcd", light, cur, _on(METRIC, p))[:, None]


def _me2(process, p, grams=None, fixed=None):
    """Helicity-summed, averaged |M|^2 at p [n][legs][4], contracted with each colour matrix
    (default: the plain one); `fixed`: {gluon number: its polarisation vectors}."""
    grams = [_gram(process)] if grams is None else grams
    amp = _amp_ttng if process.startswith("gg") else _amp_uu if process.startswith("uu") else _amp_ee
    legs = ([0, 1] if process.startswith("gg") else []) + list(range(4, p.shape[1]))
    vectors = [_polarisations(p[:, l]) for l in legs]
    for g, e in (fixed or {}).items():
        vectors[g] = [e.to(torch.complex128)]
    out = [0.0] * len(grams)
    for pol in itertools.product(*vectors):
        A = amp(p, pol).flatten(2)
        for i, G in enumerate(grams):
            out[i] = out[i] + torch.einsum("nxh,xy,nyh->n", A.conj(), _on(G, p), A).real
    return [x / PROCESSES[process][2] for x in out]


# ---------------------------------------------------------------- exact: FKS subtraction
def _unit(v):
    return v / torch.sqrt((v * v).sum(1))[:, None]


def _boost(p, b):
    b2, bp = (b * b).sum(1), (b * p[:, 1:]).sum(1)
    g = 1.0 / torch.sqrt(1.0 - b2)
    g2 = torch.where(b2 > 0, (g - 1.0) / torch.where(b2 > 0, b2, torch.ones_like(b2)), torch.zeros_like(b2))
    return torch.cat([(g * (p[:, 0] + bp))[:, None], p[:, 1:] + (g2 * bp + g * p[:, 0])[:, None] * b], 1)


def _passes(process, p, cuts):
    ok = torch.ones(p.shape[0], dtype=torch.bool, device=p.device)
    if not cuts:
        return ok
    if process.startswith("ee"):
        m = p[:, 2:, 0].argmax(1) + 2
        k = p[torch.arange(p.shape[0], device=p.device), m]
        t, z2 = k[:, 1] * k[:, 1] + k[:, 2] * k[:, 2], k[:, 3] * k[:, 3]
        return (z2 <= cuts["cut_abs_cos_axis_max"] ** 2 * (t + z2)) & (2.0 * k[:, 0] <= cuts["cut_thrust_max"] * (p[:, 0, 0] + p[:, 1, 0]))
    for leg in (2, 3):
        e, x, y, z = (p[:, leg, c] for c in range(4))
        ok &= (x * x + y * y >= cuts["cut_pt_min"] ** 2) & (e + z.abs() <= math.exp(2.0 * cuts["cut_abs_y_max"]) * (e - z.abs()))
    return ok


def _tree(process, p, cuts, factor=1.0):
    return torch.where(_passes(process, p, cuts), factor * _me2(process, p)[0], torch.zeros_like(p[:, 0, 0]))


def _real(process, p, cuts):
    """Real emission minus its FKS counterterms, summed over the sectors, p [n][5][4]."""
    born, fsr = BORN_OF[process], process == "ee_uug"
    rs = p[:, 0, 0] + p[:, 1, 0]
    s, g2 = rs * rs, GS * GS
    ni, xi = _unit(p[:, 4, 1:]), 2.0 * p[:, 4, 0] / rs
    partners = (2, 3) if fsr else (0, 1)
    y = [(ni * _unit(p[:, j, 1:])).sum(1) for j in partners]
    S = [(1.0 - y[1 - i]) / (2.0 - y[0] - y[1]) for i in range(2)]
    R = _tree(process, p, cuts)
    q = torch.cat([torch.ones_like(ni[:, :1]), ni], 1)
    coloured = (2, 3) if fsr else (0, 1, 2, 3)
    axis = {2: 0, 3: 1} if fsr else {0: 0, 1: 1, 2: 2, 3: 3}
    pairs = [(a, b) for a in coloured for b in coloured]
    grams = [_gram(born)] + [_gram_correlated(born, axis[a], axis[b]) for a, b in pairs]
    total = torch.zeros_like(rs)
    soft = None
    for i, j in enumerate(partners):
        if fsr:
            n, e, o = _unit(p[:, j, 1:]), 0.5 * rs, 5 - j
            kb = p[:, :4].clone()
            kb[:, j, 0] = kb[:, o, 0] = e
            kb[:, j, 1:], kb[:, o, 1:] = e[:, None] * n, -e[:, None] * n
            kc, soft = kb, None
            K = s * (1.0 - xi) / (16.0 * math.pi ** 3 * (2.0 - xi * (1.0 - y[i])) ** 2)
            K0, K1 = s / (64.0 * math.pi ** 3), s * (1.0 - xi) / (64.0 * math.pi ** 3)
        else:
            Q = p[:, 0] + p[:, 1] - p[:, 4]
            n = _unit(_boost(p[:, 2], -Q[:, 1:] / Q[:, :1])[:, 1:])
            beta, bq = torch.sqrt(1.0 - 4.0 * MT * MT / s), torch.sqrt((1.0 - 4.0 * MT * MT / (s * (1.0 - xi))).clamp(min=0.0))
            kb = p[:, :4].clone()
            kb[:, 2, 0] = kb[:, 3, 0] = 0.5 * rs
            kb[:, 2, 1:] = (0.5 * rs * beta)[:, None] * n
            kb[:, 3, 1:] = -kb[:, 2, 1:]
            kc = p[:, :4].clone()
            kc[:, j] *= (1.0 - xi)[:, None]
            Qc, M = kc[:, 0] + kc[:, 1], torch.sqrt(s * (1.0 - xi))
            for leg, sign in ((2, 1.0), (3, -1.0)):
                rest = torch.cat([(0.5 * M)[:, None], sign * (0.5 * M * bq)[:, None] * n], 1)
                kc[:, leg] = _boost(rest, Qc[:, 1:] / Qc[:, :1])
            K, K0 = s * bq / (64.0 * math.pi ** 3 * beta), s / (64.0 * math.pi ** 3)
            K1 = K
        if soft is None:  # the initial-state sectors share the soft counter-event
            soft = _me2(born, kb, grams)
        eik = sum(_dot(kb[:, a], kb[:, b]) / (_dot(kb[:, a], q) * _dot(kb[:, b], q)) * v for (a, b), v in zip(pairs, soft[1:]))
        s_soft = S[i] if not fsr else 0.5 * (1.0 + y[i])
        z = 1.0 - xi
        Bc = soft[0] if fsr else _me2(born, kc)[0]
        if fsr:
            coll, sc = CF * (1.0 + z * z) * Bc / z, 2.0 * CF * soft[0]
        elif born == "uu_tt":
            coll, sc = CF * (1.0 + z * z) * Bc / z, 2.0 * CF * soft[0]
        else:
            pt = torch.sqrt(ni[:, 0] ** 2 + ni[:, 1] ** 2)
            ep = torch.stack([torch.zeros_like(pt), ni[:, 0] / pt, ni[:, 1] / pt, torch.zeros_like(pt)], 1)
            Bp = _me2(born, kc, fixed={j: ep})[0]
            coll, sc = 2.0 * CA * ((z + xi * xi * z) * Bc + 2.0 * xi * xi / z * Bp) / z, 2.0 * CA * soft[0]
        G_s = (1.0 - y[i]) * s_soft * K0 * (-4.0 * g2 / s) * eik
        G_c, G_sc = K1 * (2.0 / s) * 2.0 * g2 * coll, K0 * (2.0 / s) * 2.0 * g2 * sc
        th_s, th_c = (xi < XI_CUT) & _passes(born, kb, cuts), y[i] > 1.0 - DELTA
        ct = th_s * G_s + (th_c & _passes(born, kc, cuts)) * G_c - (th_s & th_c) * G_sc
        total = total + R * S[i] - ct / (xi * xi * (1.0 - y[i]) * K)
    return total


# ---------------------------------------------------------------- exact: random numbers, sampler
def _philox(seed, stream, block, n):
    """Philox4x32-10 uniforms 2 block and 2 block + 1 of points 0 .. n - 1."""
    mask = 0xFFFFFFFF
    i = torch.arange(n, device=_device(), dtype=torch.int64)
    c = [i & mask, i >> 32, torch.full_like(i, stream), torch.full_like(i, block)]
    k = [seed & mask, (seed >> 32) & mask]

    def wide(a, b):  # high and low word of a 32 x 32 bit product
        lo = a * (b & 0xFFFF)
        hi = a * (b >> 16) + (lo >> 16)
        return hi >> 16, ((hi << 16) | (lo & 0xFFFF)) & mask

    for _ in range(10):
        (h0, l0), (h1, l1) = wide(0xD2511F53, c[0]), wide(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k[0], l1, h0 ^ c[3] ^ k[1], l0]
        k = [(k[0] + 0x9E3779B9) & mask, (k[1] + 0xBB67AE85) & mask]
    return [((c[a] >> 5).double() * 67108864.0 + (c[a + 1] >> 6).double() + 0.5) / 9007199254740992.0 for a in (0, 2)]


def _sampled(process, u, rs):
    """The FKS sampler on 18 uniforms a point: a flat channel (share 1/4) and one channel per
    sector (3/8 each); xi flat, 1 - y = 2 v^2 with v flat above sqrt(5e-7), angles flat."""
    s, fsr = rs * rs, process == "ee_uug"
    masses, vmin = PROCESSES[process][0], math.sqrt(0.5e-6)
    v = vmin + (1.0 - vmin) * u[4 if fsr else 2]
    yj, second = 1.0 - 2.0 * v * v, u[0] >= 0.625
    if fsr:
        cd, phi_d, xi, phi = 2.0 * u[1] - 1.0, 2.0 * math.pi * u[2], u[3], 2.0 * math.pi * u[5]
        sd = torch.sqrt(1.0 - cd * cd)
        nj = torch.stack([sd * torch.cos(phi_d), sd * torch.sin(phi_d), cd], 1)
        a = torch.zeros_like(nj)
        a[:, 2] = 1.0
        ea = _unit(a - cd[:, None] * nj)
        eb = torch.cross(nj, ea, dim=1)
        sr = torch.sqrt((1.0 - yj) * (1.0 + yj))
        ni = yj[:, None] * nj + sr[:, None] * (torch.cos(phi)[:, None] * ea + torch.sin(phi)[:, None] * eb)
        ei, ej = 0.5 * rs * xi, rs * (1.0 - xi) / (2.0 - xi * (1.0 - yj))
        pj = torch.cat([ej[:, None], ej[:, None] * nj], 1)
        pg = torch.cat([ei[:, None], ei[:, None] * ni], 1)
        po = torch.cat([(rs - ej - ei)[:, None], -(pj + pg)[:, 1:]], 1)
        w = second[:, None]
        p2, p3 = torch.where(w, po, pj), torch.where(w, pj, po)
    else:
        xi_max = 1.0 - 4.0 * MT * MT / s
        xi, phi, c, phi2 = xi_max * u[1], 2.0 * math.pi * u[3], 2.0 * u[4] - 1.0, 2.0 * math.pi * u[5]
        y = torch.where(second, -yj, yj)
        e, st = 0.5 * rs * xi, torch.sqrt((1.0 - y) * (1.0 + y))
        pg = torch.stack([e, e * st * torch.cos(phi), e * st * torch.sin(phi), e * y], 1)
        Q0 = rs - e
        M2 = Q0 * Q0 - e * e
        ps, sp = torch.sqrt(0.25 * M2 - MT * MT), torch.sqrt((1.0 - c) * (1.0 + c))
        d = torch.stack([sp * torch.cos(phi2), sp * torch.sin(phi2), c], 1) * ps[:, None]
        half = 0.5 * torch.sqrt(M2)[:, None]
        b = -pg[:, 1:] / Q0[:, None]
        p2, p3 = _boost(torch.cat([half, d], 1), b), _boost(torch.cat([half, -d], 1), b)
    k = torch.stack([p2, p3, pg], 1).permute(2, 1, 0)
    flat = u[0] < 0.25
    k = torch.where(flat, _rambo(torch.stack(u[6:18]), masses, rs)[0], k)
    p = _with_beams(k, rs)
    # multichannel weight: 1 / (sum of the channels' densities at the point)
    ng, x = k[1:, 2] / torch.sqrt((k[1:, 2] ** 2).sum(0)), 2.0 * k[0, 2] / rs
    w3 = s / (256.0 * math.pi ** 3)
    h = 0.25 / (w3 * _rambo_shape(k, rs) if any(masses) else w3)

    def density(y):
        g = 1.0 / (4.0 * torch.sqrt((0.5 * (1.0 - y)).clamp(min=1e-300)) * (1.0 - vmin))
        return torch.where(1.0 - y >= 1e-6, g, torch.zeros_like(g))

    if fsr:
        for j in (0, 1):
            y = (ng * k[1:, j]).sum(0) / torch.sqrt((k[1:, j] ** 2).sum(0))
            K = s * (1.0 - x) / (16.0 * math.pi ** 3 * (2.0 - x * (1.0 - y)) ** 2)
            h = h + 1.5 * density(y) / (x * K)
    else:
        beta = math.sqrt(1.0 - 4.0 * MT * MT / s)
        K = s * torch.sqrt((1.0 - 4.0 * MT * MT / (s * (1.0 - x))).clamp(min=0.0)) / (64.0 * math.pi ** 3 * beta)
        h = h + 1.5 * (density(ng[2]) + density(-ng[2])) / ((1.0 - 4.0 * MT * MT / s) * beta * x * K)
    return p, 1.0 / h


# ---------------------------------------------------------------- exact
def _in_chunks(f, p, per):
    k = p.permute(2, 1, 0)
    return torch.cat([f(k[a:a + per]) for a in range(0, k.shape[0], per)])


def _evaluated(op, process, p, w, cuts):
    per = 16384 if process == "gg_ttgg" else 65536
    if op == "real":
        x = _in_chunks(lambda k: _real(process, k, cuts), p, per)
    else:
        c = 5.0 - 2.0 * math.pi ** 2 / 3.0 - (3.0 + 4.0 * math.log(XI_CUT)) * math.log(0.5 * DELTA)
        factor = 1.0 + ALPHA_S * CF / (2.0 * math.pi) * c if op == "nbody" else 1.0
        x = _in_chunks(lambda k: _tree(process, k, cuts, factor), p, per)
    return x if w is None else w * x


def exact(case, seed):
    op = case["op"]
    if op == "unweight":
        w = _weights(case["n"], seed)
        wm = case["w_max"] if case["w_max"] > 0.0 else float(w.abs().max())
        keep = _philox(seed, 1, 0, case["n"])[0] * wm < w.abs()
        events = torch.where(w.abs() > wm, w, torch.copysign(torch.full_like(w, wm), w)) * keep
        return [events, int(keep.sum()), wm, int((w.abs() > wm).sum())]
    if op == "serve":
        return [_evaluated("real" if kind == "real_subtracted" else "born", process, p, w, {}).cpu().numpy()
                for process, kind, p, w in _served_inputs(case, seed)]
    if op == "sample":
        u = [x for b in range(9) for x in _philox(seed, 0, b, case["n"])]
        if case["points"] == "fks":
            return list(_sampled(case["process"], u, case["sqrt_s"]))
        k, w = _rambo(torch.stack(u[:12]), PROCESSES[case["process"]][0], case["sqrt_s"])
        return [_with_beams(k, case["sqrt_s"]), w]
    p, w = _inputs_of(case, seed)
    out = _evaluated(op, case["process"], p, w, _cuts(case))
    if op == "real" and case["process"] == "ee_uug":
        return [out, [float(out.sum()), float((out * out).sum()), float(case["n"])]]
    return [out]
