"""The calls that users of this framework make, as cases to time and to compare.

Every case is one pass through the public entry points of `paper_1906_11029_gb300`:

* ``evolve``    one time slab on a device-resident state (``Tents.evolve``), 2D and 3D, FP64,
                FP32 and split FP32, with the default kernel variant or the one that the
                autotuner picks for small meshes;
* ``host``      the same slab from and to pinned host buffers (``Tents.evolve_host``);
* ``adjoint``   the differentiable evolve, forward and backward, with the gradients of a
                least-squares misfit w.r.t. the initial state and both materials;
* ``batch``     many small problems with several right-hand sides in one launch (``Batch``);
* ``exchange``  initial data in, energy and lattice values out;
* ``pitch``     the tent list of a mesh, pitched on the device.

Meshes are those of the repository's workloads: the unit square of the TE cavity, the perturbed
Kuhn cube of the (1,1,1) cavity mode, the cube graded towards one corner with an eps = 4 ball, and
the cube with random eps of the gradient problem.  A slab of height T is what a time loop calls
again and again, so the evolve cases step their state in place.

`exact` is a plain FP64 implementation of the method in torch: its own reference tables by
quadrature, its own pitcher and its own tent operator with dense tables.
"""
import functools
import json
import math

import numpy as np
import torch

import paper_1906_11029_gb300 as mtp

PRECISION = {"fp64": mtp.MTP_FP64, "fp32": mtp.MTP_FP32, "split": mtp.MTP_FP32_SPLIT}
CAUSALITY = 0.5


def listed():
    return [
        # the smallest whole problem: 128 triangles, one launch of a few tents per layer (latency)
        {"name": "square8_p2_fp64", "kind": "evolve", "mesh": "square", "n": 8, "p": 2, "precision": "fp64", "T": 0.5},
        # one step of a 2D convergence study at high order
        {"name": "square32_p4_fp64", "kind": "evolve", "mesh": "square", "n": 32, "p": 4, "precision": "fp64",
         "T": 0.125},
        # 3D cavity, default settings: layers hold fewer tents than the GPU has CTA slots
        {"name": "cavity16_p3_fp32", "kind": "evolve", "mesh": "cube", "n": 16, "p": 3, "precision": "fp32", "T": 0.25},
        # the same with the kernel variant that the autotuner picks for it
        {"name": "cavity16_p3_fp32_v2", "kind": "evolve", "mesh": "cube", "n": 16, "p": 3, "precision": "fp32",
         "T": 0.25, "variant": 2},
        # the headline workload: graded mesh, p = 4, layers wider than the GPU (throughput)
        {"name": "graded32_p4_fp32", "kind": "evolve", "mesh": "graded", "n": 32, "p": 4, "precision": "fp32",
         "T": 0.01},
        # split precision: FP32 arithmetic, hi + lo Taylor sums, FP64 state
        {"name": "cavity16_p3_split", "kind": "evolve", "mesh": "cube", "n": 16, "p": 3, "precision": "split",
         "T": 0.1},
        # full FP64 in 3D, the reference solution of an accuracy check
        {"name": "cavity8_p3_fp64", "kind": "evolve", "mesh": "cube", "n": 8, "p": 3, "precision": "fp64", "T": 0.1},
        # a solver whose state lives in host memory; odd mesh size, low order
        {"name": "host13_p2_fp32", "kind": "host", "mesh": "cube", "n": 13, "p": 2, "precision": "fp32", "T": 0.1},
        # material gradients of a misfit (inverse problem), forward and backward
        {"name": "adjoint8_p2_fp64", "kind": "adjoint", "mesh": "random_eps", "n": 8, "p": 2, "precision": "fp64",
         "T": 0.2},
        # many instances of mixed size (6..20) and degree (2..4), four right-hand sides each
        {"name": "batch8_rhs4_fp32", "kind": "batch", "count": 8, "pick": 4, "n_rhs": 4, "precision": "fp32",
         "T": 0.006},
        # initial data from lattice values, then energy and lattice readout, on the headline mesh
        {"name": "exchange32_p4_fp32", "kind": "exchange", "mesh": "graded", "n": 32, "p": 4, "precision": "fp32"},
        # the tent list of a cavity mesh, pitched on the device
        {"name": "pitch16", "kind": "pitch", "mesh": "cube", "n": 16, "p": 3, "precision": "fp32", "T": 0.25},
    ]


def draw(rng):
    """One more case of the same ranges; T makes its rough cost fall between a millisecond and about half a second."""
    kind = rng.choice(["square", "fp32", "fp32", "fp32", "variant", "split", "fp64", "host", "adjoint", "batch",
                       "exchange", "pitch"])

    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    ms = math.exp(rng.uniform(math.log(2.0), math.log(300.0)))
    if kind == "square":
        c = {"kind": "evolve", "mesh": "square", "n": log_int(3, 48), "p": rng.randint(1, 4),
             "precision": rng.choice(["fp64", "fp64", "fp32"])}
    elif kind == "fp32":
        c = {"kind": "evolve", "mesh": rng.choice(["cube", "graded"]), "n": log_int(3, 32), "p": rng.randint(2, 4),
             "precision": "fp32"}
    elif kind == "variant":
        c = {"kind": "evolve", "mesh": "cube", "n": log_int(5, 16), "p": rng.randint(2, 3), "precision": "fp32",
             "variant": 2}
    elif kind in ("split", "fp64"):
        top = 20 if kind == "split" else 12
        c = {"kind": "evolve", "mesh": rng.choice(["cube", "graded"]), "n": log_int(3, top), "p": rng.randint(2, 4 if kind == "split" else 3),
             "precision": kind}
    elif kind == "host":
        c = {"kind": "host", "mesh": "cube", "n": log_int(4, 24), "p": rng.randint(2, 4), "precision": "fp32"}
    elif kind == "adjoint":
        c = {"kind": "adjoint", "mesh": "random_eps", "n": log_int(3, 8), "p": rng.randint(1, 2), "precision": "fp64"}
    elif kind == "batch":
        c = {"kind": "batch", "count": rng.randint(2, 8), "pick": rng.randint(0, 9999), "n_rhs": rng.choice([1, 2, 4]),
             "precision": "fp32", "T": 0.01}
        c["T"] = round(min(0.05, max(0.001, 0.01 * ms / sum(c["n_rhs"] * _rough_ms(i) for i in _instances(c)))), 5)
        return c
    elif kind == "exchange":
        return {"kind": "exchange", "mesh": rng.choice(["cube", "graded"]), "n": log_int(4, 32), "p": rng.randint(1, 4),
                "precision": rng.choice(["fp32", "fp32", "fp64"])}
    else:
        c = {"kind": "pitch", "mesh": rng.choice(["cube", "graded"]), "n": log_int(3, 24), "p": 2,
             "precision": "fp32"}
    c["T"] = 0.1
    c["T"] = round(min(0.5, max(0.004, 0.1 * ms / _rough_ms(c))), 5)
    return c


def _rough_tents(c):
    """Tents and layers of a slab, by the size of the mesh (a slab has at least one tent for every vertex)."""
    n, T = c["n"], c["T"]
    if c["mesh"] == "square":
        return max((n + 1) ** 2, 6.5 * n ** 3 * T), max(4, 30 * n * T)
    return max((n + 1) ** 3, 17 * n ** 4 * T), max(8, (630 if c["mesh"] == "graded" else 410) * n * T)


def _rough_updates(c):
    dim = 2 if c["mesh"] == "square" else 3
    return _rough_tents(c)[0] * (6 if dim == 2 else 24) * _nf(dim) * _nb(dim, c["p"]) * 2 * c["p"] * (c["p"] + 1)


def _rough_ms(c):
    """Rough cost of a pass in milliseconds (one GPU): layers x latency of a tent, or updates / rate."""
    layers = _rough_tents(c)[1]
    if c["kind"] == "pitch":
        return 0.04 * layers
    stage = 9e-4 * c["p"] ** 2 * (0.1 if c["mesh"] == "square" else 1.0) * {"fp64": 18, "split": 1.5, "fp32": 1}[c["precision"]]
    passes = 5.0 if c["kind"] == "adjoint" else 1.0
    rate = {"fp64": 3e9, "split": 5e10, "fp32": 7e10}[c["precision"]]
    return passes * max(layers * 2 * c["p"] * (c["p"] + 1) * stage, 1e3 * _rough_updates(c) / rate)


# ---------------------------------------------------------------------------------------------
# problems
# ---------------------------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _nf(dim):
    return 3 if dim == 2 else 6


def _nb(dim, p):
    return (p + 1) * (p + 2) // 2 if dim == 2 else (p + 1) * (p + 2) * (p + 3) // 6


def _square_mesh(n):
    x = np.linspace(0.0, 1.0, n + 1)
    Y, X = np.meshgrid(x, x, indexing="ij")
    i, j = (a.T.ravel() for a in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
    a = i + (n + 1) * j
    b, c, d = a + 1, a + n + 2, a + n + 1
    el = np.stack([np.stack([a, b, c], 1), np.stack([a, c, d], 1)], 1).reshape(-1, 3)
    return np.stack([X.ravel(), Y.ravel()], 1), el.astype(np.int32)


def _cube_mesh(n, ratio=1.0, perturb=0.0):
    """Kuhn cube, optionally graded towards the origin, interior vertices optionally perturbed."""
    size = (ratio ** (1.0 / max(1, n - 1))) ** np.arange(n)
    x = np.concatenate([[0.0], np.cumsum(size / size.sum())])
    x[-1] = 1.0
    Z, Y, X = np.meshgrid(x, x, x, indexing="ij")
    verts = np.stack([X.ravel(), Y.ravel(), Z.ravel()], 1)
    k, j, i = (a.ravel() for a in np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij"))
    base = i + (n + 1) * (j + (n + 1) * k)
    step = (1, n + 1, (n + 1) * (n + 1))
    el = []
    for q in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        v1 = base + step[q[0]]
        v2 = v1 + step[q[1]]
        el.append(np.stack([base, v1, v2, v2 + step[q[2]]], 1))
    if perturb:
        inner = np.all((verts > 1e-12) & (verts < 1.0 - 1e-12), axis=1)
        shift = np.random.default_rng(11029).uniform(-perturb / n, perturb / n, size=verts.shape)
        verts[inner] += shift[inner]
    return verts, np.stack(el, 1).reshape(-1, 4).astype(np.int32)


def _problem(c, seed):
    """(dim, vertices, elements, eps, mu) of a case."""
    if c["mesh"] == "square":
        v, e = _square_mesh(c["n"])
    elif c["mesh"] == "cube":
        v, e = _cube_mesh(c["n"], perturb=0.15)
    elif c["mesh"] == "graded":
        v, e = _cube_mesh(c["n"], ratio=8.0)
    else:
        v, e = _cube_mesh(c["n"])
    eps = np.ones(len(e))
    if c["mesh"] == "graded":
        eps[np.linalg.norm(v[e].mean(axis=1) - 0.5, axis=1) <= 0.25] = 4.0
    elif c["mesh"] == "random_eps":
        eps = np.random.default_rng([1, int(seed)]).uniform(1.0, 3.0, len(e))
    if c["kind"] == "pitch":     # a tent list depends on the materials alone
        eps = np.random.default_rng(3).uniform(1.0, 1.5, len(e)) * 4.0 ** _octave(seed)
    return v.shape[1], v, e, eps, np.ones(len(e))


def _octave(seed):
    """Other seeds pitch the same mesh in other units of time (powers of two), so the list keeps its length."""
    return int(seed) % 13 - 6


def _instances(c):
    """The instances of a batch: sizes 6..20 and degrees 2..4, picked from the case alone."""
    rng = np.random.default_rng(c["pick"])
    return [{"kind": "evolve", "mesh": "plain", "n": int(rng.integers(6, 21)), "p": int(rng.choice([2, 3, 4])),
             "precision": c["precision"], "T": c["T"]} for _ in range(c["count"])]


def _lattice(dim, p):
    r = range(p + 1)
    if dim == 2:
        return np.array([(a, b) for b in r for a in r if a + b <= p], float) / p
    return np.array([(a, b, d) for d in r for b in r for a in r if a + b + d <= p], float) / p


def _initial(c, prob, seed, n_rhs=1):
    """FP64 lattice values [rhs][element][point][field] of y = (eps E, mu H) on the device: the cavity mode at a
    random phase and amplitude, or Gaussian pulses at random centres."""
    dim, v, e, eps, mu = prob
    dev = _device()
    rng = np.random.default_rng([2, int(seed)])
    P = torch.tensor(v[np.sort(e, axis=1)], device=dev)
    xi = torch.tensor(_lattice(dim, c["p"]), device=dev)
    x = P[:, None, 0] + torch.einsum("kl,elq->ekq", xi, P[:, 1:] - P[:, :1])
    ep, m = torch.tensor(eps, device=dev)[:, None], torch.tensor(mu, device=dev)[:, None]
    out = []
    for _ in range(n_rhs):
        t, amp = rng.uniform(0.0, 1.0), rng.uniform(0.5, 2.0)
        cs = [(torch.cos(math.pi * x[..., d]), torch.sin(math.pi * x[..., d])) for d in range(dim)]
        if c["mesh"] == "square":
            (cx, sx), (cy, sy) = cs
            w = math.sqrt(2.0) * math.pi * t
            a = amp * math.sin(w) / math.sqrt(2.0)
            y = [-a * ep * cx * sy, a * ep * sx * cy, amp * math.cos(w) * m * cx * cy]
        elif c["mesh"] == "cube":
            (cx, sx), (cy, sy), (cz, sz) = cs
            w = math.sqrt(3.0) * math.pi * t
            a, b = amp * math.cos(w), -amp * math.sin(w) / math.sqrt(3.0)
            y = [a * ep * cx * sy * sz, a * ep * sx * cy * sz, -2 * a * ep * sx * sy * cz,
                 -3 * b * m * sx * cy * cz, 3 * b * m * cx * sy * cz, 0 * m * cx * cy * sz]
        else:
            ctr = rng.uniform(0.3, 0.7, size=dim)
            width = max(0.05, 1.0 / c["n"])      # a pulse that the mesh can hold
            d = x - torch.tensor(ctr, device=dev)
            psi = amp * torch.exp(-(d * d).sum(-1) / width ** 2)
            zero = torch.zeros_like(psi)
            y = [-2.0 * d[..., 1] / width ** 2 * psi * ep, 2.0 * d[..., 0] / width ** 2 * psi * ep, zero, zero, zero, zero]
        out.append(torch.stack(y, -1))
    return torch.stack(out)


def _mesh(c, prob, n_rhs=1):
    dim, v, e, eps, mu = prob
    return mtp.Mesh(dim, v, e, eps, mu, p=c["p"], precision=PRECISION[c["precision"]], n_rhs=n_rhs)


# ---------------------------------------------------------------------------------------------
# what is measured
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    c = dict(case)
    s = {"case": c}
    if c["kind"] == "batch":
        tents, states = [], []
        for i, inst in enumerate(_instances(c)):
            prob = _problem(inst, seed)
            mesh = _mesh(inst, prob, c["n_rhs"])
            tents.append(mesh.pitch(inst["T"], CAUSALITY))
            states.append(mesh.state_from_lattice(_initial(inst, prob, seed * 64 + i, c["n_rhs"])))
        s["batch"], s["states"] = mtp.Batch(tents), states
        return s
    prob = _problem(c, seed)
    mesh = s["mesh"] = _mesh(c, prob)
    if c["kind"] == "pitch":
        s["T"] = c["T"] * 2.0 ** _octave(seed)
        return s
    vals = _initial(c, prob, seed)
    if c["kind"] == "exchange":
        s["vals"], s["state"] = vals, mesh.new_state()
        s["out"] = torch.empty_like(vals)
        return s
    s["tents"] = mesh.pitch(c["T"], CAUSALITY, device=True)
    if c.get("variant"):
        s["tents"].set_variant(c["variant"])
    state = mesh.state_from_lattice(vals)
    if c["kind"] == "evolve":
        s["state"] = state
    elif c["kind"] == "host":
        s["host"] = state.cpu().pin_memory()
    else:
        dim, _, _, eps, mu = prob
        s["Y0"] = state.requires_grad_(True)
        s["eps"] = torch.tensor(eps, device=state.device, requires_grad=True)
        s["mu"] = torch.tensor(mu, device=state.device, requires_grad=True)
        s["target"] = mesh.state_from_lattice(_initial(c, prob, seed + 7919))
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "evolve":
        s["tents"].evolve(s["state"])
        return s["state"]
    if kind == "host":
        s["tents"].evolve_host(s["host"], s["host"])
        return s["host"]
    if kind == "adjoint":
        YT = mtp.mtp_evolve_autograd(s["Y0"], s["eps"], s["mu"], s["tents"])
        misfit = 0.5 * (YT - s["target"]).square().sum()
        dY, de, dm = torch.autograd.grad(misfit, (s["Y0"], s["eps"], s["mu"]))
        return {"YT": YT.detach(), "dY0": dY, "deps": de, "dmu": dm}
    if kind == "batch":
        s["batch"].evolve(s["states"])
        return s["states"]
    if kind == "exchange":
        s["mesh"].state_from_lattice(s["vals"], s["state"])
        energy = s["mesh"].energy(s["state"])
        s["mesh"].state_to_lattice(s["state"], s["out"])
        return {"state": s["state"], "energy": energy, "lattice": s["out"]}
    return s["mesh"].pitch(s["T"], CAUSALITY, device=True).get()


@functools.lru_cache(maxsize=None)
def _updates(text):
    """(spacetime DOF updates, tents) of one pass of a case; for a seed's own materials those of one seed."""
    c = json.loads(text)
    t = _mesh(c, _problem(c, 6)).pitch(c["T"], CAUSALITY)   # octave 0
    return t.info["spacetime_dofs"], t.info["n_tents"]


def _flop_per_update(dim, p):
    """Dense, formulation-free count per DOF update: volume, facet traces and lifts, mass solve and M'."""
    nfb = p + 1 if dim == 2 else (p + 1) * (p + 2) // 2
    return 2.0 * (dim * _nb(dim, p) + 2 * dim * nfb + 2 * _nf(dim))


def work(case):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        bytes_ = flops = 0.0
        for inst in _instances(c):
            w = work(inst)
            bytes_ += c["n_rhs"] * w["bytes"]
            flops += c["n_rhs"] * w["flops"]
        return {"bytes": bytes_, "flops": flops}
    dim = 2 if c["mesh"] == "square" else 3
    n_el = 2 * c["n"] ** 2 if dim == 2 else 6 * c["n"] ** 3
    coef = n_el * _nf(dim) * _nb(dim, c["p"])
    size = 4 if c["precision"] == "fp32" else 8
    if kind == "exchange":
        return {"bytes": coef * (8 + size + 8), "flops": 4.0 * coef * _nb(dim, c["p"])}
    updates, tents = _updates(json.dumps(c, sort_keys=True))
    if kind == "pitch":
        # a vertex has about 14 neighbours (time, bound, index) that each of its tents looks at once
        return {"bytes": tents * (24.0 + 14 * 20.0), "flops": tents * 14.0}
    flops = updates * _flop_per_update(dim, c["p"])
    bytes_ = 2.0 * coef * size + 256.0 * n_el + 20.0 * tents
    if kind == "adjoint":   # forward, and in reverse the transposed operator beside the forward one
        return {"bytes": 2 * bytes_, "flops": 3 * flops}
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits, without the framework
# ---------------------------------------------------------------------------------------------
def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        if sum(_cost_s(inst, c["n_rhs"]) for inst in _instances(c)) > 20:
            return None
        out = []
        for i, inst in enumerate(_instances(c)):
            prob = _problem(inst, seed)
            sch = _Scheme(*prob, inst["p"])
            sch.pitch(inst["T"])
            out.append(sch.evolve(sch.from_lattice(_initial(inst, prob, seed * 64 + i, c["n_rhs"]))))
        return out
    prob = _problem(c, seed)
    if kind == "pitch":
        t = _pitch(*prob, c["T"] * 2.0 ** _octave(seed))
        return {"vertex": None, "t_bot": t["t_bot"], "t_top": t["t_top"], "layer": None, "layer_ptr": None}
    if kind != "exchange" and _cost_s(c, 4 if kind == "adjoint" else 1) > 20:
        return None
    sch = _Scheme(*prob, c["p"])
    vals = _initial(c, prob, seed)
    Y0 = sch.from_lattice(vals)
    if kind == "exchange":
        return {"state": Y0, "energy": sch.energy(Y0), "lattice": vals}
    sch.pitch(c["T"])
    if kind == "adjoint":
        target = sch.from_lattice(_initial(c, prob, seed + 7919))
        YT, dY, de, dm = sch.gradient(Y0, target)
        return {"YT": YT, "dY0": dY, "deps": de, "dmu": dm}
    return sch.evolve(Y0)


def _cost_s(c, times=1):
    """Rough seconds that the FP64 evolve below takes: arithmetic, or its torch calls."""
    dim = 2 if c["mesh"] == "square" else 3
    calls = _rough_tents(c)[1] * 2 * c["p"] * (c["p"] + 1) * 60 * (3 if c["kind"] == "adjoint" else 1)
    return max(times * _rough_updates(c) * _flop_per_update(dim, c["p"]) / 8e11, calls * 6e-6)


def _jacobi(n, alpha, t, s):
    """s^k P_k^(alpha, 0)(t / s) for k = 0..n."""
    H = [np.ones_like(t)]
    if n >= 1:
        H.append(0.5 * ((alpha + 2) * t + alpha * s))
    for k in range(2, n + 1):
        a1 = 2.0 * k * (k + alpha) * (2 * k + alpha - 2)
        b = 2 * k + alpha - 1
        a3 = 2.0 * (k + alpha - 1) * (k - 1) * (2 * k + alpha)
        H.append((b * ((2 * k + alpha) * (2 * k + alpha - 2) * t + alpha * alpha * s) * H[-1] - a3 * s * s * H[-2]) / a1)
    return H


def _quadrature(d, n):
    """Points and weights on the unit simplex: Gauss-Legendre in collapsed coordinates."""
    g, w = np.polynomial.legendre.leggauss(n)
    g, w = (g + 1) / 2, w / 2
    if d == 1:
        return g[:, None], w
    if d == 2:
        y, x = (a.ravel() for a in np.meshgrid(g, g, indexing="ij"))
        return np.stack([x * (1 - y), y], 1), np.outer(w * (1 - g), w).ravel()
    z, y, x = (a.ravel() for a in np.meshgrid(g, g, g, indexing="ij"))
    W = np.einsum("i,j,k->ijk", w * (1 - g) ** 2, w * (1 - g), w).ravel()
    return np.stack([x * (1 - y) * (1 - z), y * (1 - z), z], 1), W


def _dubiner(d, p, X):
    """Orthogonal Dubiner functions of P_p at the points X (real or complex), ordered by degree."""
    one = np.ones_like(X[:, 0])
    x, y, z = (X[:, i] if i < d else 0 * one for i in range(3))
    out = []
    if d == 1:
        out = [(i, f) for i, f in enumerate(_jacobi(p, 0, 2 * x - 1, one))]
    else:
        for i, hi in enumerate(_jacobi(p, 0, 2 * x + y + z - 1, 1 - y - z)):
            for j, hj in enumerate(_jacobi(p - i, 2 * i + 1, 2 * y + z - 1, 1 - z)):
                if d == 2:
                    out.append((i + j, hi * hj))
                else:
                    out += [(i + j + k, hi * hj * hk)
                            for k, hk in enumerate(_jacobi(p - i - j, 2 * i + 2 * j + 2, 2 * z - 1, one))]
    return np.stack([f for _, f in sorted(out, key=lambda a: a[0])])


def _basis(d, p, X, derivative=None):
    Q, w = _quadrature(d, p + 3)
    norm = 1.0 / np.sqrt(np.einsum("ak,k->a", _dubiner(d, p, Q) ** 2, w))
    if derivative is None:
        return norm[:, None] * _dubiner(d, p, X)
    step = 1e-30       # complex step: exact for polynomials
    Xc = X.astype(complex)
    Xc[:, derivative] += 1j * step
    return norm[:, None] * _dubiner(d, p, Xc).imag / step


def _tables(d, p):
    """S[j][l] (volume), Tr[f] (facet traces), L[j][f] (lifts) and the lattice Vandermonde."""
    X, w = _quadrature(d, p + 3)
    lam = np.concatenate([1 - X.sum(1, keepdims=True), X], 1).T
    psi = _basis(d, p, X)
    S = np.stack([np.stack([np.einsum("k,ak,bk->ab", w * lam[j], _basis(d, p, X, l), psi) for l in range(d)])
                  for j in range(d + 1)])
    Xf, wf = _quadrature(d - 1, p + 3)
    corner = np.concatenate([np.zeros((1, d)), np.eye(d)])
    chi = _basis(d - 1, p, Xf)
    Tr, L = [], np.zeros((d + 1, d + 1, psi.shape[0], chi.shape[0]))
    for f in range(d + 1):
        at = corner[[i for i in range(d + 1) if i != f]]
        Y = at[0] + Xf @ (at[1:] - at[0])
        tr = _basis(d, p, Y)
        Tr.append(np.einsum("k,ck,ak->ca", wf, chi, tr))
        lf = np.concatenate([1 - Y.sum(1, keepdims=True), Y], 1).T
        for j in range(d + 1):
            L[j, f] = np.einsum("k,ak,ck->ac", wf * lf[j], tr, chi)
    return S, np.stack(Tr), L, _basis(d, p, _lattice(d, p)).T


def _pitch(dim, v, e, eps, mu, T):
    """Tents by rounds: every strict local minimum of (tau, id) moves up to min over its neighbours of tau + bound.
    The operations are those of the rule, one rounding each, so ties fall as they have to."""
    s = np.sort(e.astype(np.int64), axis=1)
    nv = len(v)
    P = [[v[s[:, i], q] for q in range(dim)] for i in range(dim + 1)]
    sub = lambda a, b: [P[b][q] - P[a][q] for q in range(dim)]  # noqa: E731
    H = []
    if dim == 2:
        det = (P[1][0] - P[0][0]) * (P[2][1] - P[0][1]) - (P[2][0] - P[0][0]) * (P[1][1] - P[0][1])
        for i in range(3):
            d = sub(*[k for k in range(3) if k != i])
            H.append(np.abs(det) / np.sqrt(d[0] * d[0] + d[1] * d[1]))
    else:
        a, b, c = sub(0, 1), sub(0, 2), sub(0, 3)
        det = a[0] * (b[1] * c[2] - b[2] * c[1]) - a[1] * (b[0] * c[2] - b[2] * c[0]) + a[2] * (b[0] * c[1] - b[1] * c[0])
        for i in range(4):
            o = [k for k in range(4) if k != i]
            u, w = sub(o[0], o[1]), sub(o[0], o[2])
            x, y, z = u[1] * w[2] - u[2] * w[1], u[2] * w[0] - u[0] * w[2], u[0] * w[1] - u[1] * w[0]
            H.append(np.abs(det) / np.sqrt(x * x + y * y + z * z))
    k = np.full(nv, np.inf)
    for i in range(dim + 1):
        np.minimum.at(k, s[:, i], H[i])
    speed = 1.0 / np.sqrt(eps * mu)
    key = np.concatenate([s[:, i] * nv + s[:, j] for i in range(dim + 1) for j in range(i + 1, dim + 1)])
    uniq, inv = np.unique(key, return_inverse=True)
    cmax = np.zeros(len(uniq))
    np.maximum.at(cmax, inv.ravel(), np.tile(speed, len(key) // len(s)))
    a, b = uniq // nv, uniq % nv
    bab = (CAUSALITY * np.minimum(k[a], k[b])) / (float(dim) * cmax)
    src, dst, bnd = np.concatenate([a, b]), np.concatenate([b, a]), np.concatenate([bab, bab])
    order = np.lexsort((dst, src))
    src, dst, bnd = src[order], dst[order], bnd[order]
    start = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=nv))])[:-1]
    tau, out, before = np.zeros(nv), [], src < dst
    while True:
        ts, td = tau[src], tau[dst]
        sel = np.nonzero(np.logical_and.reduceat((ts < td) | ((ts == td) & before), start) & (tau < T))[0]
        if not len(sel):
            break
        new = np.minimum(T, np.minimum.reduceat(td + bnd, start)[sel])
        out.append((sel, tau[sel].copy(), new))
        tau[sel] = new
    ptr = np.concatenate([[0], np.cumsum([len(o[0]) for o in out])])
    return {"vertex": np.concatenate([o[0] for o in out]), "t_bot": np.concatenate([o[1] for o in out]),
            "t_top": np.concatenate([o[2] for o in out]), "ptr": ptr}


class _Scheme:
    """Mapped tent pitching with SAT stepping in FP64 torch; every layer's patches in one set of tensors, all six
    field components (2D: the TE ones embedded)."""

    def __init__(self, dim, v, e, eps, mu, p):
        self.dev = _device()
        t = lambda a, **k: torch.tensor(np.ascontiguousarray(a), device=self.dev, **k)  # noqa: E731
        self.dim, self.p, self.prob = dim, p, (dim, v, e, eps, mu)
        self.nb, self.q, self.m = _nb(dim, p), p + 1, 2 * p
        self.comp = [0, 1, 5] if dim == 2 else list(range(6))
        s = np.sort(e.astype(np.int64), axis=1)
        ne, nvx = s.shape
        X = v[s]
        J = np.swapaxes(X[:, 1:] - X[:, :1], 1, 2)
        det = np.abs(np.linalg.det(J))
        g = np.zeros((ne, nvx, 3))
        g[:, 1:, :dim] = np.linalg.inv(J)
        g[:, 0] = -g[:, 1:].sum(1)
        size = np.linalg.norm(g, axis=2)
        self.elems, self.glam = t(s), t(g)
        self.normal, self.area = t(-g / size[..., None]), t(det[:, None] * size)
        self.scale = t(1.0 / np.sqrt(det))
        self.eps, self.mu = t(eps), t(mu)
        # patches: entries (vertex, element), by vertex, then local index, then element
        vid, loc, el = s.T.ravel(), np.repeat(np.arange(nvx), ne), np.tile(np.arange(ne), nvx)
        order = np.lexsort((el, loc, vid))
        self.p_elem, self.p_loc = t(el[order]), t(loc[order])
        self.p_ptr = np.concatenate([[0], np.cumsum(np.bincount(vid, minlength=len(v)))])
        where = np.zeros((ne, nvx), np.int64)
        where[el[order], loc[order]] = np.arange(len(order))
        # neighbours across facets
        key = np.zeros((ne, nvx), np.int64)
        for f in range(nvx):
            for i in [i for i in range(nvx) if i != f]:
                key[:, f] = key[:, f] * len(v) + s[:, i]
        flat = key.ravel()
        o = np.argsort(flat, kind="stable")
        same = np.nonzero(flat[o[1:]] == flat[o[:-1]])[0]
        nbr = np.full(ne * nvx, -1)
        nbr[o[same]], nbr[o[same + 1]] = o[same + 1], o[same]
        # per patch entry and facet containing the vertex: the neighbour's entry and facet place, flat, or -1
        fac = np.array([[f for f in range(nvx) if f != j] for j in range(nvx)])
        nb_f = np.full((len(order), dim), -1)
        pe, pj, pv = el[order], loc[order], vid[order]
        for i in range(dim):
            f = fac[pj, i]
            n2 = nbr[pe * nvx + f]
            e2, f2 = n2 // nvx, n2 % nvx
            j2 = np.argmax(s[e2] == pv[:, None], axis=1)
            place = where[e2, j2] * dim + f2 - (f2 > j2)
            nb_f[:, i] = np.where(n2 >= 0, place, -1)
        self.p_nbr, self.fac = t(nb_f), t(fac)
        S, Tr, L, V = _tables(dim, p)
        self.V, self.Vinv = t(V), t(np.linalg.inv(V))
        self.into, self.lift = [], []
        for j in range(nvx):
            self.into.append(t(np.concatenate([S[j].reshape(-1, self.nb)] + [Tr[f] for f in fac[j]]).T))
            self.lift.append(t(np.concatenate([L[j, f].T for f in fac[j]])))
        self.nfb = Tr.shape[1]

    def from_lattice(self, vals):
        return torch.einsum("ak,rekf->refa", self.Vinv, vals) / self.scale[:, None, None]

    def energy(self, Y):
        nE = 2 if self.dim == 2 else 3
        d = Y.square().sum(-1)
        return (0.5 * (d[..., :nE].sum(-1) / self.eps + d[..., nE:].sum(-1) / self.mu).sum(-1)).cpu().numpy()

    def pitch(self, T):
        t = _pitch(*self.prob, T)
        self.tents = [(t["vertex"][a:b], t["t_bot"][a:b], t["t_top"][a:b]) for a, b in zip(t["ptr"][:-1], t["ptr"][1:])]

    def _layer_data(self, tau, layer):
        """Index tensors and time-dependent geometry of a layer's patches, entries sorted by local index."""
        vs, tb, tt = layer
        cnt = self.p_ptr[vs + 1] - self.p_ptr[vs]
        off = np.concatenate([[0], np.cumsum(cnt)])
        pos = np.arange(off[-1]) + np.repeat(self.p_ptr[vs] - off[:-1], cnt)
        to = lambda a: torch.from_numpy(a).to(self.dev)  # noqa: E731
        pos, dt = to(pos), to(np.repeat(tt - tb, cnt))
        shift = to(np.repeat(self.p_ptr[vs] - off[:-1], cnt))
        j = self.p_loc[pos]
        order = torch.argsort(j, stable=True)
        rank = torch.empty_like(order)
        rank[order] = torch.arange(len(order), device=self.dev)
        nb = self.p_nbr[pos]
        place = torch.where(nb >= 0, nb // self.dim - shift[:, None], 0)
        nb = torch.where(nb >= 0, rank[place] * self.dim + nb % self.dim, -1)[order]
        pos, dt, j = pos[order], dt[order], j[order]
        e = self.p_elem[pos]
        d = {"e": e, "dt": dt, "count": torch.bincount(j, minlength=self.dim + 1).tolist()}
        gl = self.glam[e]
        d["a"] = dt[:, None, None, None] * gl[:, 1:, :, None]
        d["g0"] = torch.einsum("ni,niq->nq", tau[self.elems[e]], gl)
        d["g1"] = dt[:, None] * gl[torch.arange(len(e), device=self.dev), j]
        f = self.fac[j]
        rows = e[:, None].expand_as(f)
        d["n"] = self.normal[rows, f].reshape(-1, 3, 1)
        d["lift"] = (dt[:, None] * self.area[rows, f] * self.scale[e][:, None])[:, None, :, None]
        d["scale"] = self.scale[e][:, None, None]
        d["wall"] = (nb < 0).reshape(-1)
        d["nbr"] = torch.where(nb < 0, torch.arange(nb.numel(), device=self.dev).view_as(nb), nb).reshape(-1)
        return d

    def _step(self, Y, d, eps, mu):
        """All SAT stages of a layer: Y [rhs][entry][6][basis] at the tent bottoms -> at the tent tops."""
        cross = lambda x, y: torch.linalg.cross(*torch.broadcast_tensors(x, y), dim=-2)  # noqa: E731
        R, N, nb, dim, nfb = Y.shape[0], Y.shape[1], self.nb, self.dim, self.nfb
        Z = torch.sqrt(mu / eps)[d["e"]][:, None].expand(N, dim).reshape(-1)
        Zm, Zp = Z[:, None, None], Z[d["nbr"]][:, None, None]
        mirror = torch.tensor([-1.0] * 3 + [1.0] * 3, dtype=Y.dtype, device=Y.device)[:, None]
        wall, n = d["wall"][:, None, None], d["n"]
        ep, m = eps[d["e"]][:, None, None], mu[d["e"]][:, None, None]

        def by_j(A, mats):
            parts = [x @ mat for x, mat in zip(A.split(d["count"], dim=1), mats)]
            return torch.cat(parts, 1)

        def operator(U):
            PT = by_j(U, self.into)
            P = PT[..., :dim * nb].view(R, N, 6, dim, nb)
            out = [0.0, 0.0]
            for l in range(dim):
                out[0] = out[0] - cross(d["a"][:, l], P[:, :, 3:, l])
                out[1] = out[1] + cross(d["a"][:, l], P[:, :, :3, l])
            um = (PT[..., dim * nb:].view(R, N, 6, dim, nfb).transpose(2, 3) * d["scale"][:, None]).reshape(R, -1, 6, nfb)
            up = torch.where(wall, um * mirror, um[:, d["nbr"]])
            tang = lambda w: w - (w * n).sum(-2, keepdim=True) * n  # noqa: E731
            Em, Ep, Hm, Hp = tang(um[:, :, :3]), tang(up[:, :, :3]), um[:, :, 3:], up[:, :, 3:]
            FE = (cross(Zm * Hm + Zp * Hp, n) + Em - Ep) / (Zm + Zp)
            Et = (Zp * Em + Zm * Ep + Zp * Zm * cross(Hm - Hp, n)) / (Zm + Zp)
            F = torch.cat([FE, -cross(Et, n)], -2).view(R, N, dim, 6, nfb).transpose(2, 3) * d["lift"]
            return torch.cat(out, -2) - by_j(F.reshape(R, N, 6, dim * nfb), self.lift)

        def solve(y, g):
            g = g[:, :, None]
            s = 1.0 / (ep * m - (g * g).sum(-2, keepdim=True))
            yE, yH = y[:, :, :3], y[:, :, 3:]
            flat = lambda w: w - g * ((g * w).sum(-2, keepdim=True) / (ep * m))  # noqa: E731
            return torch.cat([s * (m * flat(yE) - cross(g, yH)), s * (ep * flat(yH) + cross(g, yE))], -2)

        gd = d["g1"][:, :, None]
        for i in range(self.m):
            g = d["g0"] + (i / self.m) * d["g1"]
            U, c = solve(Y, g), 1.0
            for k in range(1, self.q + 1):
                Yk = operator(U)
                c = c / (self.m * k)
                Y = Y + c * Yk
                if k < self.q:
                    MU = torch.cat([-cross(U[:, :, 3:], gd), cross(U[:, :, :3], gd)], -2)
                    U = solve(Yk - k * MU, g)
        return Y

    def _embed(self, Y):
        out = torch.zeros(Y.shape[0], Y.shape[1], 6, self.nb, dtype=Y.dtype, device=Y.device)
        out[:, :, self.comp] = Y
        return out

    def _front(self):
        return torch.zeros(len(self.prob[1]), dtype=torch.float64, device=self.dev)

    def evolve(self, Y, each=None):
        Y, tau = self._embed(Y), self._front()
        for layer in self.tents:
            d = self._layer_data(tau, layer)
            if each is not None:
                each.append((d, Y[:, d["e"]]))
            Y[:, d["e"]] = self._step(Y[:, d["e"]], d, self.eps, self.mu)
            tau[torch.from_numpy(layer[0]).to(self.dev)] = torch.from_numpy(layer[2]).to(self.dev)
        return Y[:, :, self.comp]

    def gradient(self, Y0, target):
        tape = []
        YT = self.evolve(Y0, tape)
        lam = self._embed(YT - target)
        eps, mu = self.eps.clone().requires_grad_(True), self.mu.clone().requires_grad_(True)
        de, dm = torch.zeros_like(eps), torch.zeros_like(mu)
        for d, bottom in reversed(tape):
            y = bottom.clone().requires_grad_(True)
            top = self._step(y, d, eps, mu)
            gy, ge, gm = torch.autograd.grad(top, (y, eps, mu), lam[:, d["e"]])
            lam[:, d["e"]] = gy
            de += ge
            dm += gm
        return YT, lam[:, :, self.comp], de, dm
