"""The work a program gives this library, as timed cases.

Every case goes through the public entry points of paper_2310_13908_gb300, with
the surfaces, densities and regularization of the paper's method: the layer sums
over one capsule surface in both precisions, the sums over the upsampled grid and
by the FMM, the membrane force, whole capsule steps and a burst of served
requests. A program keeps one context (and one server), works on a stream of its
own, and holds its inputs in device memory, except where the entry point takes
host arrays (capsules, the server).

SK_FP32C is the 32-bit mode: its callers keep the velocities in 32 bits, and so do
these cases. SK_FP64 results, forces and node positions stay in 64 bits.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import capsule_inputs as ci
import paper_2310_13908_gb300 as sk
from capsule_inputs.workloads import build_request

ES, ED = 2.0, 20.0        # Skalak moduli (Sec. 4.3)
FMM_K, FMM_P, FMM_LLOYD = 128, 6, 10
EULER_DT = 1e-4


# ---- the cases ----------------------------------------------------------------

def _layer(name, shape, m, layer, precision, delta, probes=0, nodes=True):
    """One layer sum: targets are the surface's nodes and / or exterior probes."""
    c = {"kind": "layer", "shape": shape, "m": m, "layer": layer, "precision": precision,
         "delta": delta, "probes": probes, "nodes": nodes}
    return {"name": name, **c} if name else c


def listed():
    return [
        # a coarse capsule (N = 1,944), the smallest surface of the mix: latency and launches count
        _layer("sphere19_single_fp32c", "sphere", 19, "single", "fp32c", "2h"),
        _layer("sphere19_single_fp64", "sphere", 19, "single", "fp64", "2h"),
        # a red cell at an everyday resolution (N = 24,576): velocity from a traction, the
        # stresslet with the delta* of each target's patch, and the 64-bit sum of the same size
        _layer("cell65_single_fp32c", "cell", 65, "single", "fp32c", "2h"),
        _layer("cell65_double_fp32c", "cell", 65, "double", "fp32c", "star"),
        _layer("cell65_single_fp64", "cell", 65, "single", "fp64", "2h"),
        # a fine ellipsoid (N = 221,184): the stresslet at its nodes
        _layer("ellipsoid193_double_fp32c", "ellipsoid", 193, "double", "fp32c", "2h"),
        # the finest surface (N = 393,216) with 100,000 off-surface probes: the largest sum
        _layer("ellipsoid257_probes_single_fp32c", "ellipsoid", 257, "single", "fp32c", "2h",
               probes=100_000),
        # the paper's upsampled sum at m = 32: few targets (5,766), many sources (96,774)
        {"name": "upsampled32_fp32c", "kind": "upsampled", "m": 32, "precision": "fp32c"},
        # the single-level FMM over the nodes of a fine surface (N = 98,304)
        {"name": "fmm129_fp32c", "kind": "fmm", "m": 129, "precision": "fp32c"},
        # the membrane force of every time step, 128 x 128 nodes per patch
        {"name": "membrane129", "kind": "membrane", "m": 129},
        # a time-step loop: four explicit Euler steps of a membrane capsule in shear flow
        {"name": "capsule65_steps4", "kind": "capsule", "m": 65, "steps": 4, "precision": "fp32c"},
        # requests of uneven size that arrive together at the server
        {"name": "serve_burst24", "kind": "serve", "requests": 24, "mix": 4000, "n_min": 1536,
         "n_max": 98_304},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choices(["layer", "upsampled", "fmm", "membrane", "capsule", "serve"],
                       [7, 1, 1, 1, 1, 1])[0]
    if kind == "layer":
        precision = rng.choices(["fp32c", "fp64"], [3, 1])[0]
        fp64 = precision == "fp64"
        m = _log_int(rng, 9, 64 if fp64 else 192)
        where = rng.choice(["nodes", "nodes", "both", "probes"])
        probes = 0 if where == "nodes" else _log_int(rng, 100, 3_000 if fp64 else 40_000)
        # delta* is a rule for nodes: probes take the global delta
        delta = rng.choice(["1.5h", "2h", "3h"] + (["star"] if where == "nodes" else []))
        return _layer(None, rng.choice(["sphere", "cell", "ellipsoid"]), m,
                      rng.choice(["single", "double"]), precision, delta, probes=probes,
                      nodes=where != "probes")
    if kind == "upsampled":
        return {"kind": "upsampled", "m": rng.randint(8, 48), "precision": "fp32c"}
    if kind == "fmm":
        return {"kind": "fmm", "m": _log_int(rng, 65, 160), "precision": "fp32c"}
    if kind == "membrane":
        return {"kind": "membrane", "m": _log_int(rng, 9, 256)}
    if kind == "capsule":
        return {"kind": "capsule", "m": _log_int(rng, 17, 96), "steps": rng.randint(1, 8),
                "precision": "fp32c"}
    return {"kind": "serve", "requests": rng.randint(2, 40), "mix": rng.randrange(1 << 20),
            "n_min": 1536, "n_max": _log_int(rng, 6_000, 98_304)}


# ---- inputs ---------------------------------------------------------------------

_PRECISION = {"fp32c": sk.SK_FP32C, "fp64": sk.SK_FP64}
_kept: dict = {}


def _handle():
    """The program's context, its stream, and what it keeps on the device."""
    if "ctx" not in _kept:
        _kept["ctx"] = sk.Context(0)
        _kept["stream"] = torch.cuda.Stream()
    return _kept["ctx"].handle, _kept["stream"]


def _server():
    """The program's server, in a context of its own; it shares the GPU with the program's
    other work, so its kernel leaves soon after the last request."""
    if "server" not in _kept:
        _kept["server_ctx"] = sk.Context(0)
        _kept["server"] = sk.serve_create(_kept["server_ctx"].handle, max_slots=32,
                                           idle_exit_us=2_000)
    return _kept["server"]


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def _shape(kind, rng):
    if kind == "sphere":
        return ci.Sphere(1.0)
    if kind == "cell":
        return ci.EvansFungRBC(ci.random_rotation(rng))
    return ci.Ellipsoid(1.0, 0.8, 0.5)


def _layer_inputs(case, seed):
    """(X, w, normals, density, targets, delta) of one layer sum, as numpy arrays."""
    rng = np.random.default_rng(seed)
    shape = _shape(case["shape"], rng)
    s = ci.make_surface(shape, case["m"])
    dens = ci.sh_density(s.x0, rng, lmax=8)
    if case["shape"] == "sphere":  # uniform traction with noise
        dens = np.array([1.0, 0.0, 0.0]) + ci.gaussian_noise(s.N, 0.1, rng)
    parts = [s.X] if case["nodes"] else []
    if case["probes"]:
        parts.append(ci.exterior_probes(shape, case["probes"], s.h, rng)[0])
    delta = (ci.delta_star(s) if case["delta"] == "star"
             else np.array([float(case["delta"][:-1]) * s.h]))
    return s.X, s.w, s.n, dens, np.concatenate(parts), delta


def _nodes_inputs(case, seed):
    """Ellipsoid (1, 0.8, 0.5) surface and a density (upsampled sums, FMM)."""
    rng = np.random.default_rng(seed)
    s = ci.make_surface(ci.Ellipsoid(1.0, 0.8, 0.5), case["m"])
    return s, ci.sh_density(s.x0, rng, lmax=8)


def _membrane_inputs(case, seed):
    """Stress-free ellipsoid (0.9, 1, 1) and its stretched nodes."""
    rng = np.random.default_rng(seed)
    ref = ci.make_surface(ci.Ellipsoid(0.9, 1.0, 1.0), case["m"])
    return ref, ref.X * (1.0 + rng.uniform(-0.04, 0.04, 3))


def _mix(case):
    """The requests' kinds and sizes."""
    return ci.serving_mix(case["requests"], seed=case["mix"], n_min=case["n_min"],
                          n_max=case["n_max"])


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for spec in _mix(case):
        kind, params = spec["shape"]
        new = np.sort(rng.uniform(0.5, 1.0, 3))[::-1] if kind == "ellipsoid" else rng.normal(size=4)
        spec = dict(spec, shape=(kind, tuple(float(v) for v in new)), seed=int(rng.integers(1 << 31)))
        s, f, delta = build_request(spec)
        out.append((s.X, s.w, f, s.X, np.array([delta])))
    return out


class _Capsule:
    """A resident capsule with its membrane; released with the state."""

    def __init__(self, case, seed):
        ref, X = _membrane_inputs(case, seed)
        self.cap = sk.Capsule(_handle()[0], case["m"], X, ref.w, delta=None, mu=1.0,
                              precision=_PRECISION[case["precision"]])
        self.cap.set_membrane(ref.X, ES, ED)

    def __del__(self):
        if hasattr(self, "cap"):
            self.cap.close()


def prepare(case, seed):
    kind = case["kind"]
    ctx, stream = _handle()
    st = {"kind": kind, "ctx": ctx, "stream": stream, "case": case}
    if kind == "layer":
        X, w, n, dens, Y, delta = (_dev(a) for a in _layer_inputs(case, seed))
        st.update(X=X, w=w, n=n, dens=dens, Y=Y, delta=delta)
    elif kind == "upsampled":
        s, f = _nodes_inputs(case, seed)
        st.update(X=_dev(s.X), W=_dev(s.W), f=_dev(f))
    elif kind == "fmm":
        s, f = _nodes_inputs(case, seed)
        act = np.flatnonzero(s.w)
        st.update(X=_dev(s.X), w=_dev(s.w), f=_dev(f), delta=_dev([2.0 * s.h]),
                  centers=_dev(s.X[act[:: len(act) // FMM_K][:FMM_K]]))
    elif kind == "membrane":
        ref, X = _membrane_inputs(case, seed)
        st.update(X=_dev(X), ref=_dev(ref.X))
    elif kind == "capsule":
        st["capsule"] = _Capsule(case, seed)
    elif kind == "serve":
        st.update(server=_server(), requests=_requests(case, seed))
    else:
        raise ValueError(f"unknown kind {kind!r}")
    torch.cuda.synchronize()  # the inputs were made on another stream
    return st


# ---- one pass -------------------------------------------------------------------

def _kept_as(u, precision):
    """Velocities as the caller of that precision keeps them."""
    return u if precision == "fp64" else u.to(torch.float32)


def run(st):
    kind, case, ctx, stream = st["kind"], st["case"], st["ctx"], st["stream"]
    if kind == "serve":
        srv = st["server"]
        tickets = [(sk.serve_submit(srv, *r, 1.0), r[3].shape[0]) for r in st["requests"]]
        out = []
        for t, n in tickets:
            code, u, _ = sk.serve_poll(srv, t, n)
            if code != sk.SK_OK:
                raise RuntimeError(f"served request failed: {code}")
            out.append(u.astype(np.float32))
        return out
    if kind == "capsule":
        cap = st["capsule"].cap
        cap.step(case["steps"], EULER_DT, None, (sk.SK_FLOW_SHEAR, 1.0, 0.0, 0.0))
        return cap.positions()
    with torch.cuda.stream(stream):
        if kind == "layer":
            prec = _PRECISION[case["precision"]]
            if case["layer"] == "single":
                u = sk.stokes_sl_eval(ctx, prec, sk.SK_DEVICE, st["X"], st["w"], st["dens"],
                                      st["Y"], st["delta"], 1.0, stream=stream)
            else:
                u = sk.stokes_dl_eval(ctx, prec, sk.SK_DEVICE, st["X"], st["w"], st["n"],
                                      st["dens"], st["Y"], st["delta"], stream=stream)
            return _kept_as(u, case["precision"])
        if kind == "upsampled":
            u = sk.stokes_sl_eval_upsampled(ctx, _PRECISION[case["precision"]], sk.SK_DEVICE,
                                            case["m"], st["X"], st["W"], st["f"], 1.0,
                                            stream=stream)
            return _kept_as(u, case["precision"])
        if kind == "fmm":
            u = sk.stokes_sl_eval_fmm(ctx, sk.SK_DEVICE, st["X"], st["w"], st["f"], st["X"],
                                      st["delta"], 1.0, st["centers"], FMM_LLOYD, FMM_P,
                                      stream=stream, precision=_PRECISION[case["precision"]])
            return _kept_as(u, case["precision"])
        f, w = sk.membrane_force(ctx, case["m"], sk.SK_DEVICE, st["X"], st["ref"], ES, ED,
                                 weights=True, stream=stream)
        return f, w


# ---- what a pass cannot do without --------------------------------------------------

def _active(m):
    """Nodes with nonzero weight on the grid of order m (the same for every shape)."""
    return ci.make_surface(ci.Sphere(1.0), m).n_active


def _layer_work(n, n_active, n_tgt, n_delta, double, out_bytes):
    # 29 flops per single-layer pair and 33 per double-layer pair (FMA = 2, rsqrt = 1)
    return {"bytes": 8 * ((10 if double else 7) * n + 3 * n_tgt + n_delta) + 3 * out_bytes * n_tgt,
            "flops": (33 if double else 29) * n_tgt * n_active}


def work(case):
    kind = case["kind"]
    if kind == "serve":
        tot = {"bytes": 0, "flops": 0}
        for m in (spec["m"] for spec in _mix(case)):
            w = _layer_work(6 * (m - 1) ** 2, _active(m), 6 * (m - 1) ** 2, 1, False, 8)
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    m = case["m"]
    n = 6 * (m - 1) ** 2
    if kind == "layer":
        n_tgt = (n if case["nodes"] else 0) + case["probes"]
        return _layer_work(n, _active(m), n_tgt, n if case["delta"] == "star" else 1,
                           case["layer"] == "double", 8 if case["precision"] == "fp64" else 4)
    if kind == "upsampled":
        return _layer_work(n, _active(4 * m), n, 0, False, 4)
    if kind == "fmm":
        # every target against the surface points of each cluster's cube (or the sources, if
        # they are fewer)
        per_target = min(_active(m), FMM_K * (6 * FMM_P ** 2 - 12 * FMM_P + 8))
        return {"bytes": 8 * (7 * n + 3 * n) + 12 * n, "flops": 29 * n * per_target}
    # membrane force: 15 fields (two sets of tangents, the tension, their derivatives), each
    # with spline slopes, extension, differences and blending (about 120 operations per node)
    membrane = {"bytes": 8 * 10 * n, "flops": 15 * 120 * n}
    if kind == "membrane":
        return membrane
    one = _layer_work(n, _active(m), n, 0, False, 8)
    return {k: case["steps"] * (membrane[k] + one[k]) for k in one}


# ---- the same numbers in plain 64-bit torch and numpy ----------------------------------

def _sum64(double, X, w, n, dens, Y, delta, mu=1.0, pairs_at_once=1 << 24):
    """The regularized layer sum in 64 bits, target block by target block."""
    keep = w != 0
    X, w, dens = X[keep], w[keep], dens[keep]
    scale = -6.0 / (8.0 * math.pi) if double else 1.0 / (8.0 * math.pi * mu)
    g = dens * w[:, None] * scale
    if double:
        n = n[keep]
    delta = delta.expand(Y.shape[0])
    out = torch.empty_like(Y)
    step = max(1, pairs_at_once // X.shape[0])
    for a in range(0, Y.shape[0], step):
        y, dl = Y[a:a + step], delta[a:a + step]
        d = [y[:, c, None] - X[None, :, c] for c in range(3)]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        ri = r2.rsqrt()
        i, j = torch.nonzero(r2 < (7.0 * dl[:, None]) ** 2, as_tuple=True)
        rho = r2[i, j].sqrt() / dl[i]
        at0 = rho == 0
        p2, er = rho * rho, torch.erf(rho)
        ex = torch.exp(-p2) / math.sqrt(math.pi)
        gd = (d[0] * g[:, 0]).addcmul_(d[1], g[:, 1]).addcmul_(d[2], g[:, 2])
        b = ri * ri * ri
        if double:
            b *= ri * ri
            s3 = er - (2.0 / 9.0) * rho * (((8 * p2 - 36) * p2 + 6) * p2 + 9) * ex
            b[i, j] = torch.where(at0, 0.0, b[i, j] * s3)
            gd *= (d[0] * n[:, 0]).addcmul_(d[1], n[:, 1]).addcmul_(d[2], n[:, 2])
        else:
            s1 = er - (2.0 / 3.0) * rho * (2 * p2 - 5) * ex
            s2 = er - (2.0 / 3.0) * rho * ((4 * p2 - 14) * p2 + 3) * ex
            b[i, j] = torch.where(at0, 0.0, b[i, j] * s2)
            ri[i, j] = torch.where(at0, 16.0 / (3.0 * math.sqrt(math.pi)) / dl[i], ri[i, j] * s1)
        gd *= b
        u = torch.stack([(gd * d[c]).sum(1) for c in range(3)], 1)
        out[a:a + step] = u if double else u + ri @ g
    return out


def _spline_matrix(m):
    """Not-a-knot cubic spline through h, 2h, .. (m - 1) h, as the matrix that takes node
    values to values at h/4, 2h/4, .. (4m - 1) h/4 (end pieces continued)."""
    n = m - 1
    A = np.eye(n) * 4.0 + np.eye(n, k=1) + np.eye(n, k=-1)
    B = 6.0 * (np.eye(n, k=1) + np.eye(n, k=-1) - 2.0 * np.eye(n))
    A[0], A[-1], B[0], B[-1] = 0.0, 0.0, 0.0, 0.0
    A[0, :3] = A[-1, -3:] = (1.0, -2.0, 1.0)
    M = np.linalg.solve(A, B)  # second derivatives times h^2
    x = np.arange(1, 4 * m) / 4.0 - 1.0
    k = np.clip(np.floor(x).astype(int), 0, n - 2)
    t = (x - k)[:, None]
    eye = np.eye(n)
    return ((1 - t) * eye[k] + t * eye[k + 1]
            + ((1 - t) ** 3 - (1 - t)) / 6.0 * M[k] + (t ** 3 - t) / 6.0 * M[k + 1])


def _upsampled64(case, seed):
    s, f = _nodes_inputs(case, seed)
    m, nf = case["m"], 4 * case["m"] - 1
    S = _spline_matrix(m)
    G = np.concatenate([s.X, s.W[:, None], f], 1).reshape(6, m - 1, m - 1, 7)
    fine = np.einsum("ai,pijc,bj->pabc", S, G, S, optimize=True)
    grid = fine[..., :3]
    reach = np.zeros(6)  # largest distance to a grid neighbour, per patch
    for a, b in ((0, 1), (1, 0), (1, 1), (1, -1)):
        lo = grid[:, :nf - a, max(0, -b):nf - max(0, b)]
        hi = grid[:, a:, max(0, b):nf + min(0, b)]
        reach = np.maximum(reach, np.linalg.norm(hi - lo, axis=-1).reshape(6, -1).max(1))
    psi = ci.make_surface(ci.Sphere(1.0), 4 * m).psi
    fine = fine.reshape(-1, 7)
    w = psi * fine[:, 3] * (math.pi / (4 * m)) ** 2
    return _sum64(False, _dev(fine[:, :3]), _dev(w), None, _dev(fine[:, 4:]), _dev(s.X),
                  _dev(np.repeat(reach, (m - 1) ** 2)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "layer":
        X, w, n, dens, Y, delta = (_dev(a) for a in _layer_inputs(case, seed))
        return _sum64(case["layer"] == "double", X, w, n, dens, Y, delta)
    if kind == "upsampled":
        return _upsampled64(case, seed)
    if kind == "fmm":
        s, f = _nodes_inputs(case, seed)
        return _sum64(False, _dev(s.X), _dev(s.w), None, _dev(f), _dev(s.X), _dev([2.0 * s.h]))
    if kind == "serve":
        return [_sum64(False, _dev(X), _dev(w), None, _dev(f), _dev(Y), _dev(delta)).cpu().numpy()
                for X, w, f, Y, delta in _requests(case, seed)]
    # the finite-difference operator of the membrane has no short form
    return None
