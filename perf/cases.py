"""The calls that users of the library make, at the sizes they make them, as measurable cases.

Each case is one call of ``paper_2304_07006_gb300.Context`` on a synthetic molecule: atom-centred
quadrature grid with Becke weights, Cartesian Gaussian orbitals orthonormal on that grid, a density
and a polynomial Jastrow factor with U(-0.1, 0.1) coefficients.  Inputs and outputs are CUDA tensors,
and the context is kept, as in a program that updates orbitals or Jastrow parameters and builds
again.  ``exact`` evaluates the working equations in plain FP64 torch.

Keys of a case:
  call       "build" (closed shell), "rohf" (two spin densities), "batched", "two_body_K", "fold"
  precision  the context's precision: "fp64", "fp16x2" or "bf16x3"
  n_orb, n_grid, n_nuc, n_sets       sizes (n_sets Jastrow centre sets, shared cyclically)
  rank       occupied orbitals (two or more: with one the constant vanishes), or with correlated=True
             the rank of a random symmetric density
  outer      outer grid points of a partial sum (a resumable piece of a large build); 0 = all
  du         type of the Delta U output: "f64" or "f32"
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2304_07006_gb300 import Context

TERMS = np.array([(0, 0, 1), (0, 1, 1), (0, 2, 1), (1, 1, 1), (1, 2, 1),
                  (0, 0, 2), (0, 1, 2), (0, 2, 2), (1, 1, 2)], dtype=np.int32)
EXACT_FLOPS = 9e12   # FP64 operations beyond which exact() is left out (about 10 s on one GB300)


def _case(name, call, precision, n_orb, n_grid, n_nuc, n_sets, rank, correlated=False, outer=0, du="f64"):
    c = {"call": call, "precision": precision, "n_orb": n_orb, "n_grid": n_grid, "n_nuc": n_nuc,
         "n_sets": n_sets, "rank": rank, "correlated": correlated, "outer": outer, "du": du}
    return {"name": name, **c} if name else c


def listed():
    return [
        # H2-sized reference build, all FP64, two natural orbitals occupied: the smallest build, the one
        # new inputs are checked with
        _case("h2_fp64", "build", "fp64", 10, 2000, 2, 1, 2, correlated=True),
        # a small ragged molecule in the default precision: launches and latency count
        _case("small_fp16x2", "build", "fp16x2", 23, 3957, 3, 3, 3),
        # water-sized build in the alternative mixed precision
        _case("water_bf16x3", "build", "bf16x3", 58, 40000, 3, 3, 5),
        # the headline build: a diatomic in a large basis, the whole grid, default precision
        _case("n2_fp16x2", "build", "fp16x2", 120, 100000, 2, 2, 7),
        # one resumable piece of a build too long for one call: many orbitals, 8 nuclei, FP32 Delta U
        _case("large_piece_fp16x2", "build", "fp16x2", 200, 200000, 8, 2, 14, outer=2560, du="f32"),
        # open shell: separate alpha and beta densities
        _case("rohf_fp16x2", "rohf", "fp16x2", 40, 20000, 3, 3, 5),
        # a correlated (full-rank) reference density, odd sizes, four nuclei
        _case("correlated_fp16x2", "build", "fp16x2", 65, 24001, 4, 4, 65, correlated=True),
        # several molecules or Jastrow parameter sets of uneven size in one call (sizes: see _instances)
        {"name": "batch8_fp16x2", "call": "batched", "precision": "fp16x2", "n_inst": 8, "sizes": 4,
         "n_orb_lo": 20, "n_orb_hi": 90, "n_grid_lo": 3000, "n_grid_hi": 20000},
        # FP64 reference of a water-sized build on some of its outer points (how a mixed build is verified)
        _case("water_fp64_piece", "build", "fp64", 58, 40000, 3, 3, 5, outer=512),
        # the two-body integrals K on the smallest molecule, all FP64
        _case("k_h2_fp64", "two_body_K", "fp64", 10, 2000, 2, 1, 0),
        # K on a larger molecule in the default precision
        _case("k_mid_fp16x2", "two_body_K", "fp16x2", 30, 8000, 3, 3, 0),
        # freezing the core of a finished build
        {"name": "fold_n120", "call": "fold", "precision": "fp16x2", "n_orb": 120, "n_core": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "mixed", "mixed", "mixed", "piece", "rohf", "batched", "fp64_piece", "K", "K", "fold"])
    while True:
        nuc = rng.randint(1, 4)
        if kind == "fp64":
            n, g = _log_int(rng, 6, 24), _log_int(rng, 1000, 4000)
            c = _case(None, "build", "fp64", n, g, nuc, nuc, rng.randint(2, max(2, n // 5)))
        elif kind == "mixed":
            n, g = _log_int(rng, 10, 120), _log_int(rng, 2000, 100000)
            corr = rng.random() < 0.3
            c = _case(None, "build", rng.choice(["fp16x2", "fp16x2", "bf16x3"]), n, g, nuc, nuc,
                      rng.randint(2, n) if corr else rng.randint(2, max(2, n // 8)), correlated=corr,
                      du=rng.choice(["f64", "f64", "f32"]))
        elif kind == "piece":
            n, g = _log_int(rng, 100, 200), _log_int(rng, 60000, 200000)
            nuc = rng.randint(2, 8)
            c = _case(None, "build", "fp16x2", n, g, nuc, min(2, nuc), rng.randint(5, 14),
                      outer=rng.randint(500, 4000), du="f32")
        elif kind == "rohf":
            n, g = _log_int(rng, 15, 70), _log_int(rng, 4000, 40000)
            c = _case(None, "rohf", "fp16x2", n, g, nuc, nuc, rng.randint(2, max(2, n // 8)))
        elif kind == "batched":
            lo, glo = rng.randint(10, 40), rng.randint(3000, 10000)
            c = {"call": "batched", "precision": "fp16x2", "n_inst": rng.randint(2, 8), "sizes": rng.randint(0, 10 ** 6),
                 "n_orb_lo": lo, "n_orb_hi": rng.randint(lo, 90), "n_grid_lo": glo, "n_grid_hi": rng.randint(glo, 20000)}
        elif kind == "fp64_piece":
            n, g = _log_int(rng, 20, 80), _log_int(rng, 10000, 60000)
            c = _case(None, "build", "fp64", n, g, nuc, nuc, rng.randint(2, max(2, n // 8)), outer=rng.randint(64, 1024))
        elif kind == "K":
            n, g = _log_int(rng, 8, 48), _log_int(rng, 1500, 12000)
            c = _case(None, "two_body_K", rng.choice(["fp64", "fp16x2"]), n, g, nuc, nuc, 0)
        else:
            n = rng.randint(24, 120)
            c = {"call": "fold", "precision": "fp16x2", "n_orb": n, "n_core": rng.randint(0, min(8, n // 8))}
        # at most about a second: FP64 work runs near 0.7 TFLOP/s, mixed work near 300
        f = work(c)["flops"]
        slow = c["precision"] == "fp64" or c["call"] == "two_body_K"
        if f <= (3e11 if slow else 3e14):
            return c


# ----------------------------------------------------------------------------- synthetic molecules

def _centres(rng, n_nuc):
    out, radius = [], 1.2 + 0.45 * n_nuc
    while len(out) < n_nuc:
        p = rng.uniform(-radius, radius, 3)
        if np.linalg.norm(p) <= radius and all(np.linalg.norm(p - q) > 1.3 for q in out):
            out.append(p)
    return np.array(out)


def _grid(centres, n_grid, dev):
    """Radial x angular grids around every nucleus with Becke weights; the points of smallest weight
    are dropped until n_grid are left."""
    n_at = len(centres)
    n_theta, n_phi = (5, 10) if n_grid < 6000 else (10, 20)
    n_rad = max(4, -(-n_grid // (n_at * n_theta * n_phi)))
    t = np.arange(1, n_rad + 1) * math.pi / (n_rad + 1)
    x = np.cos(t)
    wx = math.pi / (n_rad + 1) * np.sin(t)
    lg = np.log(2.0 / (1.0 - x))
    r = (1.0 + x) ** 0.6 * lg / math.log(2.0)
    dr = (0.6 * (1.0 + x) ** -0.4 * lg + (1.0 + x) ** 0.6 / (1.0 - x)) / math.log(2.0)
    ct, wt = np.polynomial.legendre.leggauss(n_theta)
    ph = 2.0 * math.pi * (np.arange(n_phi) + 0.5) / n_phi
    st = np.sqrt(1.0 - ct * ct)
    ang = np.stack([np.outer(st, np.cos(ph)), np.outer(st, np.sin(ph)), np.outer(ct, np.ones(n_phi))], -1).reshape(-1, 3)
    wa = np.outer(wt, np.full(n_phi, 2.0 * math.pi / n_phi)).reshape(-1)
    C = torch.tensor(centres, device=dev)
    local = torch.tensor((r[:, None, None] * ang).reshape(-1, 3), device=dev)
    wl = torch.tensor(((wx * dr * r * r)[:, None] * wa).reshape(-1), device=dev)
    pts = (C[:, None, :] + local).reshape(-1, 3)
    w = wl.repeat(n_at)
    if n_at > 1:
        d = torch.linalg.vector_norm(pts[:, None, :] - C, dim=-1)
        cell = torch.ones_like(d)
        for a in range(n_at):
            for b in range(n_at):
                if a != b:
                    mu = (d[:, a] - d[:, b]) / float(np.linalg.norm(centres[a] - centres[b]))
                    for _ in range(3):
                        mu = 1.5 * mu - 0.5 * mu ** 3
                    cell[:, a] *= 0.5 * (1.0 - mu)
        owner = torch.arange(n_at, device=dev).repeat_interleave(local.shape[0])
        w = w * cell.gather(1, owner[:, None])[:, 0] / cell.sum(1)
    keep = torch.sort(torch.argsort(w, descending=True, stable=True)[:n_grid]).values
    return pts[keep].contiguous(), w[keep].contiguous()


_CART = {0: [(0, 0, 0)], 1: [(1, 0, 0), (0, 1, 0), (0, 0, 1)],
         2: [(2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1)]}


def _shells(n_nuc, n_func):
    """Even-tempered s, p and d shells, shared out over the nuclei in turn."""
    out, total, k = [], 0, 0
    used = [[0, 0, 0] for _ in range(n_nuc)]
    while total < n_func:
        a, L = k % n_nuc, (0, 1, 0, 2, 0, 1)[(k // n_nuc) % 6]
        out.append((a, L, (0.08, 0.15, 0.3)[L] * 2.4 ** used[a][L]))
        used[a][L] += 1
        total += len(_CART[L])
        k += 1
    return out


def _orbitals(pts, w, centres, n_orb, rng, gradients):
    shells = _shells(len(centres), n_orb + n_orb // 4 + 2)
    C = torch.tensor(centres, device=pts.device)
    cols, grads = [], []
    for a, L, alpha in shells:
        d = pts - C[a]
        g = torch.exp(-alpha * (d * d).sum(1))
        for ijk in _CART[L]:
            mono = [d[:, x] ** ijk[x] for x in range(3)]
            cols.append(mono[0] * mono[1] * mono[2] * g)
            if gradients:
                for x in range(3):
                    k = ijk[x]
                    dk = (k * d[:, x] ** (k - 1) if k else 0.0) - 2.0 * alpha * d[:, x] ** (k + 1)
                    grads.append(dk * mono[(x + 1) % 3] * mono[(x + 2) % 3] * g)
    chi = torch.stack(cols, 1)
    norm = (chi * chi * w[:, None]).sum(0).sqrt()
    chi = chi / norm
    s, U = np.linalg.eigh((chi.T @ (chi * w[:, None])).cpu().numpy())
    q, _ = np.linalg.qr(rng.standard_normal((n_orb, n_orb)))
    T = (U[:, -n_orb:] / np.sqrt(s[-n_orb:])) @ q   # orthonormal, randomly rotated
    T = torch.tensor(T, device=pts.device)
    phi = (chi @ T).contiguous()
    dphi = None
    if gradients:
        dchi = torch.stack(grads, 1).reshape(pts.shape[0], -1, 3) / norm[None, :, None]
        dphi = torch.einsum("gmx,mo->gox", dchi, T).contiguous()
    return phi, dphi


def _molecule(rng, n_orb, n_grid, n_nuc, n_sets, gradients=False):
    dev = torch.device("cuda", 0)
    centres = _centres(rng, n_nuc)
    pts, w = _grid(centres, n_grid, dev)
    phi, dphi = _orbitals(pts, w, centres, n_orb, rng, gradients)
    return {"nuc_xyz": centres, "nuc_set": np.arange(n_nuc, dtype=np.int32) % n_sets, "terms": TERMS,
            "coef": rng.uniform(-0.1, 0.1, (n_sets, len(TERMS))), "grid": pts, "weights": w, "phi": phi, "dphi": dphi}


def _density(rng, n_orb, rank, correlated, dev):
    g = np.zeros((n_orb, n_orb))
    if correlated:
        q, _ = np.linalg.qr(rng.standard_normal((n_orb, n_orb)))
        occ = np.zeros(n_orb)
        occ[:rank] = rng.uniform(0.02, 1.0, rank)
        g = (q * occ) @ q.T
        g = 0.5 * (g + g.T)
    else:
        g[np.arange(rank), np.arange(rank)] = 1.0
    return torch.tensor(g, device=dev)


def _instances(case):
    """(n_orb, n_grid, n_nuc) of the instances of a batched case."""
    r = random.Random(case["sizes"])
    return [(r.randint(case["n_orb_lo"], case["n_orb_hi"]), r.randint(case["n_grid_lo"], case["n_grid_hi"]), r.randint(1, 4))
            for _ in range(case["n_inst"])]


# ----------------------------------------------------------------------------- the calls

def _inputs(case, seed):
    rng = np.random.default_rng([int(seed), 77])
    dev = torch.device("cuda", 0)
    call = case["call"]
    if call == "fold":
        # the outputs of a build: Delta U with its 8-fold symmetry and symmetric Delta h
        n, k = case["n_orb"], 24
        f = torch.tensor(rng.standard_normal((k, n, n)), device=dev)
        f = (f + f.transpose(1, 2)).reshape(k, n * n)
        h = torch.tensor(rng.standard_normal((n, n)), device=dev)
        core = sorted(int(c) for c in rng.choice(n // 2, case["n_core"], replace=False))
        return {"dU": (f.T @ f / (4.0 * k)).reshape(n, n, n, n).contiguous(), "dh": (h + h.T).contiguous(), "core": core}
    if call == "batched":
        out = []
        for n, g, nuc in _instances(case):
            m = _molecule(rng, n, g, nuc, nuc)
            m["gamma"] = _density(rng, n, max(2, n // 10), False, dev)
            out.append(m)
        return {"instances": out}
    n = case["n_orb"]
    m = _molecule(rng, n, case["n_grid"], case["n_nuc"], case["n_sets"], gradients=call == "two_body_K")
    if call == "build":
        m["gamma"] = _density(rng, n, case["rank"], case["correlated"], dev)
    elif call == "rohf":
        m["gamma_a"] = _density(rng, n, case["rank"], False, dev)
        m["gamma_b"] = _density(rng, n, max(1, case["rank"] - 1), False, dev)
    return m


def prepare(case, seed):
    s = _inputs(case, seed)
    dev, f64 = torch.device("cuda", 0), torch.float64
    s["call"] = case["call"]
    s["ctx"] = ctx = Context(case["precision"], device=0)

    def empty(*shape, dtype=f64):
        return torch.empty(shape, dtype=dtype, device=dev)

    if case["call"] == "batched":
        for m in s["instances"]:
            n = m["phi"].shape[1]
            m["dU"], m["dh"], m["e0"] = empty(n, n, n, n), empty(n, n), empty(1)
        return s
    n = case["n_orb"]
    if case["call"] == "fold":
        na = n - case["n_core"]
        s["out"] = {"dh_fc": empty(na, na), "dU_act": empty(na, na, na, na), "e_core": empty(1)}
        return s
    ctx.set_jastrow(s["nuc_xyz"], s["nuc_set"], s["terms"], s["coef"])
    if case["outer"]:
        ctx.set_outer_range(0, case["outer"])
    if case["call"] == "build":
        s["out"] = {"dh": empty(n, n), "e0": empty(1)}
        if case["du"] == "f32":
            s["out"]["dU_f32"] = empty(n, n, n, n, dtype=torch.float32)
        else:
            s["out"]["dU"] = empty(n, n, n, n)
    elif case["call"] == "rohf":
        s["out"] = {k: empty(n, n, n, n) for k in ("dU_aa", "dU_ab", "dU_bb")}
        s["out"] |= {"dh_a": empty(n, n), "dh_b": empty(n, n), "e0": empty(1)}
    else:
        s["out"] = empty(n, n, n, n)
    return s


def run(state):
    s = state
    ctx, call = s["ctx"], s["call"]
    if call == "build":
        ctx.build(s["grid"], s["weights"], s["phi"], s["gamma"], **s["out"])
        return s["out"]
    if call == "rohf":
        return ctx.build_rohf(s["grid"], s["weights"], s["phi"], s["gamma_a"], s["gamma_b"], **s["out"])
    if call == "batched":
        return ctx.build_batched(s["instances"])
    if call == "two_body_K":
        return ctx.two_body_K(s["grid"], s["weights"], s["phi"], s["dphi"], out=s["out"])
    return ctx.frozen_core_fold(s["dU"], s["dh"], s["core"], **s["out"])


# ----------------------------------------------------------------------------- work

def _build_work(n, g, outer, n_nuc, du_bytes, n_du, spins):
    npair = n * (n + 1) / 2
    flops = 6.0 * outer * g * npair              # step (b)
    flops += spins * 8.0 * outer * npair ** 2    # step (d)
    flops += 12.0 * outer * n ** 3               # step (c)
    nbytes = 8.0 * (g * (4 + n) + spins * n * n)         # grid, weights, orbitals, densities
    return nbytes + n_du * du_bytes * n ** 4 + 8.0 * (spins * n * n + 1), flops


def work(case):
    call = case["call"]
    if call == "fold":
        n, na = case["n_orb"], case["n_orb"] - case["n_core"]
        return {"bytes": 16.0 * na ** 4 + 16.0 * na * na, "flops": 4.0 * na * na * max(1, case["n_core"])}
    if call == "batched":
        parts = [_build_work(n, g, g, nuc, 8, 1, 1) for n, g, nuc in _instances(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n, g = case["n_orb"], case["n_grid"]
    outer = case["outer"] or g
    if call == "two_body_K":
        npair = n * (n + 1) / 2
        # V (three components), W and the contraction over (outer point, component)
        return {"bytes": 8.0 * (g * (4 + 4 * n) + n ** 4), "flops": 8.0 * outer * g * npair + 8.0 * outer * n * n * npair}
    spin = call == "rohf"
    b, f = _build_work(n, g, outer, case["n_nuc"], 4 if case["du"] == "f32" else 8, 3 if spin else 1, 2 if spin else 1)
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- plain FP64 evaluation

def _pow(a, k):
    return torch.ones_like(a) if k == 0 else (a if k == 1 else a ** k)


def _jastrow(ri, rj, m, laplacian):
    """nabla_1 u (3 arrays) and, if asked, nabla_1^2 u for all pairs of ri and rj; unit vectors and 2/r
    terms are 0 below 1e-14 bohr."""
    d = [ri[:, None, x] - rj[None, :, x] for x in range(3)]
    r12 = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).sqrt()
    i12 = torch.where(r12 < 1e-14, 0.0, 1.0 / r12.clamp_min(1e-14))
    b = r12 / (1.0 + r12)
    bp = 1.0 / (1.0 + r12) ** 2
    bpp = -2.0 / (1.0 + r12) ** 3
    hb = torch.zeros_like(r12)                   # factor of the electron-electron unit vector
    g = [torch.zeros_like(r12) for _ in range(3)]
    lap = torch.zeros_like(r12) if laplacian else None
    for I, R in enumerate(torch.tensor(m["nuc_xyz"], device=ri.device)):
        v = ri - R
        d1 = torch.linalg.vector_norm(v, dim=1)
        i1 = torch.where(d1 < 1e-14, 0.0, 1.0 / d1.clamp_min(1e-14))
        e1 = v * i1[:, None]
        a1 = (d1 / (1.0 + d1))[:, None]
        ap = (1.0 / (1.0 + d1) ** 2)[:, None]
        app = (-2.0 / (1.0 + d1) ** 3)[:, None]
        d2 = torch.linalg.vector_norm(rj - R, dim=1)
        a2 = (d2 / (1.0 + d2))[None, :]
        ga = torch.zeros_like(r12)
        for o in range(3):
            P, Pa, Paa = 0.0, 0.0, 0.0
            for (p, q, oo), c in zip(m["terms"].tolist(), m["coef"][m["nuc_set"][I]].tolist()):
                if oo != o:
                    continue
                P = P + c * (_pow(a1, p) * _pow(a2, q) + _pow(a1, q) * _pow(a2, p))
                for s, t in ((p, q), (q, p)):    # a1^s a2^t
                    if s >= 1:
                        Pa = Pa + c * s * _pow(a1, s - 1) * _pow(a2, t)
                    if s >= 2:
                        Paa = Paa + c * s * (s - 1) * _pow(a1, s - 2) * _pow(a2, t)
            if isinstance(P, float):
                continue
            Q, Qb, Qbb = _pow(b, o), (o * _pow(b, o - 1) if o else 0.0), (2.0 if o == 2 else 0.0)
            ga += Pa * Q
            if o:
                hb += P * Qb
            if laplacian:
                lap += Q * (Paa * ap * ap + Pa * (app + 2.0 * ap * i1[:, None]))
                if o:
                    cos = (e1[:, 0, None] * d[0] + e1[:, 1, None] * d[1] + e1[:, 2, None] * d[2]) * i12
                    lap += P * (Qbb * bp * bp + Qb * (bpp + 2.0 * bp * i12)) + 2.0 * Pa * ap * Qb * bp * cos
        for x in range(3):
            g[x] += ga * ap * e1[:, x, None]
    hb = hb * bp * i12
    for x in range(3):
        g[x] += hb * d[x]
    return g, lap


def _fields(m, i0, i1, laplacian=False):
    """V_x (and the field of lap u + |grad u|^2) of outer points [i0, i1): [x][i][pair]; packed pairs."""
    n = m["phi"].shape[1]
    p, q = torch.triu_indices(n, n, device=m["phi"].device)
    V = torch.zeros(4 if laplacian else 3, i1 - i0, len(p), dtype=torch.float64, device=p.device)
    step = max(256, int(6e7 / (i1 - i0 + len(p))))
    for j0 in range(0, m["phi"].shape[0], step):
        f, w = m["phi"][j0:j0 + step], m["weights"][j0:j0 + step]
        rho = w[:, None] * f[:, p] * f[:, q]
        g, lap = _jastrow(m["grid"][i0:i1], m["grid"][j0:j0 + step], m, laplacian)
        if laplacian:
            g = g + [lap + g[0] * g[0] + g[1] * g[1] + g[2] * g[2]]
        for x, gx in enumerate(g):
            V[x].addmm_(gx, rho)
    return V, p, q


def _blocks(n_outer, n_orb):
    step = int(max(32, min(2048, 4e8 / (8.0 * n_orb * n_orb * 12))))
    return [(i, min(i + step, n_outer)) for i in range(0, n_outer, step)]


def _full(packed, p, q, n):
    out = torch.empty(packed.shape[:-1] + (n, n), dtype=packed.dtype, device=packed.device)
    out[..., p, q] = packed
    out[..., q, p] = packed
    return out


def _assemble(m, n_outer, direct, exchange):
    """f^t[pq][rs] = sum_i rho_pq A^t_rs + V_pq . B^t_rs (all N^2 x N^2) for every exchange density t, with
    the direct density `direct`."""
    n = m["phi"].shape[1]
    f = [torch.zeros(n * n, n * n, dtype=torch.float64, device=direct.device) for _ in exchange]
    for i0, i1 in _blocks(n_outer, n):
        V, p, q = _fields(m, i0, i1)
        V = _full(V, p, q, n)                                     # [x][i][N][N]
        phi, w = m["phi"][i0:i1], m["weights"][i0:i1]
        rho = w[:, None, None] * phi[:, :, None] * phi[:, None, :]
        W = (V * direct).sum((2, 3))
        Vt = (W[:, :, None, None] * V).sum(0)
        Wt = (rho * direct).sum((1, 2))
        k = i1 - i0
        for t, gx in enumerate(exchange):
            X = gx @ V
            A = Vt - (V @ X).sum(0)
            Z = rho @ X
            B = 0.5 * Wt[None, :, None, None] * V - Z - Z.transpose(2, 3)
            f[t] += rho.reshape(k, -1).T @ A.reshape(k, -1)
            for x in range(3):
                f[t] += V[x].reshape(k, -1).T @ B[x].reshape(k, -1)
    return f


def exact(case, seed):
    if case["call"] == "fold":
        s = _inputs(case, seed)
        act = [k for k in range(case["n_orb"]) if k not in s["core"]]
        a = torch.tensor(act, device=s["dU"].device)
        U, h = s["dU"], s["dh"]
        hf = h[a][:, a].clone()
        e = torch.zeros(1, dtype=torch.float64, device=U.device)
        for c in s["core"]:
            hf += 2.0 * U[:, :, c, c][a][:, a] - U[:, c, c, :][a][:, a]
            e += 2.0 * h[c, c]
            for d in s["core"]:
                e += 2.0 * U[c, c, d, d] - U[c, d, d, c]
        return {"dh_fc": hf, "dU_act": U[a][:, a][:, :, a][:, :, :, a].contiguous(), "e_core": e}
    if work(case)["flops"] > EXACT_FLOPS:
        return None
    if case["call"] == "batched":
        return None
    m = _inputs(case, seed)
    n = case["n_orb"]
    n_outer = case["outer"] or case["n_grid"]
    if case["call"] == "two_body_K":
        S = torch.zeros(n * n, n * n, dtype=torch.float64, device=m["phi"].device)
        for i0, i1 in _blocks(n_outer, n):
            V, p, q = _fields(m, i0, i1, laplacian=True)
            V = _full(V, p, q, n).reshape(4, i1 - i0, n * n)
            wp = m["weights"][i0:i1, None] * m["phi"][i0:i1]
            S += 0.5 * (wp[:, :, None] * m["phi"][i0:i1, None, :]).reshape(i1 - i0, -1).T @ V[3]
            for x in range(3):
                S += (wp[:, :, None] * m["dphi"][i0:i1, None, :, x]).reshape(i1 - i0, -1).T @ V[x]
        return (S + S.T).reshape(n, n, n, n)
    if case["call"] == "rohf":
        ga, gb = m["gamma_a"], m["gamma_b"]
        fa, fb = _assemble(m, n_outer, ga + gb, [ga, gb])
        aa, bb, ab = ((-(x + y.T)).reshape(n, n, n, n) for x, y in ((fa, fa), (fb, fb), (fb, fa)))

        def onebody(U, cross, g, go):
            return -0.5 * (torch.einsum("pqrs,rs->pq", U, g) + torch.einsum("pqrs,rs->pq", cross, go)
                           - torch.einsum("psrq,rs->pq", U, g))
        ha, hb = onebody(aa, ab, ga, gb), onebody(bb, ab.permute(2, 3, 0, 1), gb, ga)
        return {"dU_aa": aa, "dU_ab": ab, "dU_bb": bb, "dh_a": ha, "dh_b": hb,
                "e0": (-((ha * ga).sum() + (hb * gb).sum()) / 3.0).reshape(1)}
    g = m["gamma"]
    f, = _assemble(m, n_outer, 2.0 * g, [g])
    dU = (-(f + f.T)).reshape(n, n, n, n)
    dh = -0.5 * (2.0 * torch.einsum("pqrs,rs->pq", dU, g) - torch.einsum("psrq,rs->pq", dU, g))
    out = {"dh": dh, "e0": (-2.0 / 3.0 * (dh * g).sum()).reshape(1)}
    out["dU_f32" if case["du"] == "f32" else "dU"] = dU
    return out
