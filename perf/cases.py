"""Cases for timing the framework through its public entry points.

A case is one call that an AFQMC program makes with one trial and one
Hamiltonian: the overlap, the force bias, the local energy, all three in one
pass, the one-body density matrix, a propagation step, a batch of uneven
systems, or a gradient of the control-variate network. The sizes are those of
the repository's workloads (`synth.CONFIGS`, the batched recipe, the network of
the control-variate run) and odd sizes between them; `draw` gives more of the
same ranges.

Integrals are at a chemical scale (mean on-site repulsion 1 Ha, a Cholesky
spectrum exp(-g / (n_chol / 6))), as those of a molecule are. Every input,
Hamiltonian and trial included, is made from the seed; large arrays are made on
the GPU and handed over as the entry points take them. `exact` evaluates the
same quantities in 64 bits with plain torch.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2406_08314_gb300 import cv, msd
from paper_2406_08314_gb300.synth import System

DEV = "cuda:0"
C128 = torch.complex128

_CU2O2 = dict(M=108, na=16, nb=16, core=8, act=16, level=6, n_chol=400)
_FE2S2 = dict(M=160, na=30, nb=30, core=15, act=20, level=6, n_chol=800)
_SMALL = dict(M=20, na=5, nb=5, core=0, act=10, level=4, n_chol=60)


def listed():
    return [
        # the smallest call: one overlap of a handful of walkers, all latency
        dict(name="overlap_small", op="overlap", prec="fp64", **_SMALL, n_det=100, n_w=16),
        # the smallest full measurement of a walker set
        dict(name="evaluate_small", op="evaluate", prec="mixed", **_SMALL, n_det=100, n_w=16),
        # the copper-oxo-shaped trial at the paper's walker count, both precisions
        dict(name="evaluate_cu2o2", op="evaluate", prec="mixed", **_CU2O2, n_det=10000, n_w=640),
        dict(name="evaluate_cu2o2_fp64", op="evaluate", prec="fp64", **_CU2O2, n_det=10000, n_w=640),
        # the iron-sulfur-shaped trial: the benchmark's step
        dict(name="evaluate_fe2s2", op="evaluate", prec="mixed", **_FE2S2, n_det=120000, n_w=640),
        # the same trial in the default precision, energies of one block of walkers
        dict(name="energy_fe2s2_fp64", op="energy", prec="fp64", **_FE2S2, n_det=120000, n_w=64),
        # the paper's largest expansion in its few-walker regime
        dict(name="evaluate_1e6_few", op="evaluate", prec="mixed", **_CU2O2, n_det=1000000, n_w=10),
        # one phaseless AFQMC step with re-orthonormalisation
        dict(name="propagate_cu2o2", op="propagate", prec="fp64", **_CU2O2, n_det=10000, n_w=640, order=6, qr=True),
        # importance sampling between measurements: force bias, unequal spins, ragged sizes
        dict(name="force_bias_odd", op="force_bias", prec="mixed", M=131, na=23, nb=19, core=11, act=19, level=5,
             n_chol=523, n_det=20011, n_w=97),
        # the property estimator, unequal spins, ragged sizes
        dict(name="rdm_odd_fp64", op="rdm", prec="fp64", M=87, na=13, nb=11, core=5, act=15, level=5, n_chol=301,
             n_det=3001, n_w=211),
        # uneven systems evaluated together
        dict(name="batch_uneven", op="batch", prec="mixed", n_sys=6, m_lo=40, m_hi=160, det_lo=1000, det_hi=100000,
             n_w=128, shape_seed=0),
        # one gradient of the control-variate network on a training batch
        dict(name="network_grad", op="network", n_in=6912, width=256, n_w=512),
    ]


def draw(rng):
    """One more case of the listed ranges; no costlier than the largest listed one."""
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    op = rng.choice(["overlap", "force_bias", "evaluate", "evaluate", "energy", "rdm", "propagate", "batch", "network"])
    if op == "network":
        return dict(op=op, n_in=64 * log(16, 120), width=256, n_w=log(64, 2048))
    if op == "batch":
        return dict(op=op, prec=rng.choice(["mixed", "mixed", "fp64"]), n_sys=rng.randint(2, 6), m_lo=30, m_hi=rng.randint(50, 120),
                    det_lo=300, det_hi=log(1000, 30000), n_w=log(8, 64), shape_seed=rng.randint(1, 10 ** 6))
    prec = rng.choice(["mixed", "fp64"])
    M = rng.randint(20, 160)
    na = rng.randint(4, max(4, min(32, M // 5)))
    nb = max(3, na - rng.choice([0, 0, 1, 2, 3]))
    ae = rng.randint(3, min(nb, 12))                    # active electrons of the smaller spin
    core = nb - ae
    holes = na - core                                   # the larger spin's
    parts = rng.randint(3, max(3, min(9, 112 // holes, M - na)))
    act = min(holes + parts, M - core)
    level = rng.randint(3, 6)
    c = dict(op=op, prec=prec, M=M, na=na, nb=nb, core=core, act=act, level=level,
             n_chol=min(rng.randint(3 * M, 5 * M), M * (M + 1) // 2), n_det=0, n_w=log(1, 640))
    c["n_det"] = max(2, min(log(50, 100000), _pair_count(c) // 2))
    if op == "propagate":
        c |= dict(order=rng.randint(4, 8), qr=rng.random() < 0.5)
    top = max(_cost(x) for x in listed() if x["op"] not in ("network", "batch"))
    while _cost(c) > top and c["n_w"] > 1:
        c["n_w"] = c["n_w"] * 2 // 3
    return c


def _cost(c):
    """Rough relative time: FP64 work counts for more than the mixed path's."""
    w = work(c)
    return w["flops"] * (8.0 if c["prec"] == "fp64" or c["op"] == "propagate" else 1.0)


# ------------------------------------------------------------------- inputs
def _levels(n, c):
    """(active occupied, active virtual, highest level) of one spin."""
    o = n - c["core"]
    v = c["act"] - o
    return o, v, min(o, v, c["level"], 6)


def _pair_count(c):
    cnt = []
    for n in (c["na"], c["nb"]):
        o, v, k = _levels(n, c)
        cnt.append([math.comb(o, i) * math.comb(v, i) for i in range(k + 1)])
    return sum(a * b for i, a in enumerate(cnt[0]) for j, b in enumerate(cnt[1]) if 1 <= i + j <= c["level"])


def _strings(n, c):
    """Every excitation string of one spin up to the highest level, by level:
    holes and particles (orbital numbers, [n_k][k]) and the sign of sorting."""
    o, v, kmax = _levels(n, c)
    out = []
    for k in range(kmax + 1):
        h = np.array(list(itertools.combinations(range(c["core"], n), k)), np.int64).reshape(math.comb(o, k), k)
        p = np.array(list(itertools.combinations(range(n, c["core"] + c["act"]), k)), np.int64).reshape(math.comb(v, k), k)
        hh, pp = np.repeat(h, len(p), 0), np.tile(p, (len(h), 1))
        inv = sum((n - 1 - hh[:, i]) - (k - 1 - i) for i in range(k)) if k else np.zeros(len(hh), np.int64)
        out.append((hh, pp, np.where(inv % 2, -1.0, 1.0)))
    return out


def _occupations(n, strings):
    occ = []
    for h, p, _ in strings:
        k = h.shape[1]
        rows = np.tile(np.arange(n), (len(h), 1))
        if k:
            np.put_along_axis(rows, h, p, 1)
        occ.append(np.sort(rows, 1))
    return np.concatenate(occ).astype(np.int32)


def _trial(c, rng):
    """CI trial of distinct excitation pairs, uniform over all pairs with
    total level 1..level, sorted by level; |c_I| = (I + 1)^-1.2, random signs.
    Also the string numbers of every determinant."""
    sa, sb = _strings(c["na"], c), _strings(c["nb"], c)
    na, nb = [len(x[2]) for x in sa], [len(x[2]) for x in sb]
    oa, ob = np.cumsum([0] + na), np.cumsum([0] + nb)
    cls = [(i, j) for i in range(len(na)) for j in range(len(nb)) if 1 <= i + j <= c["level"]]
    w = np.array([float(na[i]) * nb[j] for i, j in cls])
    ca, cb = np.array([i for i, _ in cls]), np.array([j for _, j in cls])
    keys = np.zeros(0, np.int64)
    want = c["n_det"] - 1
    while keys.size < want:
        t = rng.choice(len(cls), size=int((want - keys.size) * 1.2) + 16, p=w / w.sum())
        i, j = ca[t], cb[t]
        a = oa[i] + (rng.random(t.size) * np.array(na)[i]).astype(np.int64)
        b = ob[j] + (rng.random(t.size) * np.array(nb)[j]).astype(np.int64)
        both = np.concatenate([keys, a * ob[-1] + b])
        _, first = np.unique(both, return_index=True)
        keys = both[np.sort(first)][:want]
    a, b = keys // ob[-1], keys % ob[-1]
    lv = (np.searchsorted(oa, a, "right") - 1) + (np.searchsorted(ob, b, "right") - 1)
    order = np.argsort(lv, kind="stable")
    a, b = np.concatenate([[0], a[order]]), np.concatenate([[0], b[order]])
    coeff = (np.arange(c["n_det"]) + 1.0) ** -1.2 * rng.choice([-1.0, 1.0], size=c["n_det"])
    coeff[0] = abs(coeff[0])
    coeff /= np.linalg.norm(coeff)
    return coeff, _occupations(c["na"], sa)[a], _occupations(c["nb"], sb)[b], a, b


def _inputs(c, seed):
    """The system (host arrays) and its walkers (on the GPU)."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    M, G = c["M"], c["n_chol"]

    def randn(*shape):
        return torch.randn(shape, dtype=torch.float64, device=DEV, generator=gen)

    h = torch.triu(randn(M, M))
    h = (h + torch.triu(h, 1).T) / M
    L = randn(G, M, M)
    L = L + L.transpose(1, 2)
    L /= torch.linalg.vector_norm(L, dim=(1, 2), keepdim=True)
    L *= torch.exp(-torch.arange(G, device=DEV, dtype=torch.float64) / (G / 6.0))[:, None, None]
    d = torch.diagonal(L, dim1=1, dim2=2)
    L /= math.sqrt(float((d * d).sum(0).mean()))        # mean (pp|pp) = 1 Ha
    coeff, occ_a, occ_b, a, b = _trial(c, rng)
    hn = h.cpu().numpy()
    s = System(M, c["na"], c["nb"], np.stack([hn, hn]), 0.0, L.cpu().numpy(), coeff, occ_a, occ_b, c["core"], c["act"])
    walkers = []
    for n in (c["na"], c["nb"]):
        phi = torch.complex(randn(c["n_w"], M, n), randn(c["n_w"], M, n)) * (0.1 / math.sqrt(2.0))
        phi[:, torch.arange(n), torch.arange(n)] += 1.0
        walkers.append(_orthonormal(phi))
    x = randn(c["n_w"], G)
    return s, walkers[0], walkers[1], x, (h, L, a, b)


def _orthonormal(phi):
    """Q of phi = Q R with a positive diagonal of R (Cholesky of phi^H phi)."""
    r = torch.linalg.cholesky(phi.mH @ phi)             # lower, phi^H phi = r r^H
    return torch.linalg.solve_triangular(r.mH, phi, upper=True, left=False).contiguous()


def _members(c):
    """The cases of a batch: M uniform, M // 6 electrons per spin, n_det
    log-uniform, 4 M Cholesky vectors, min(N, 8) active electrons in twice as
    many orbitals. The shapes belong to the case, the values to the seed."""
    r = np.random.default_rng(c["shape_seed"])
    out = []
    for _ in range(c["n_sys"]):
        M = int(r.integers(c["m_lo"], c["m_hi"] + 1))
        n = M // 6
        e = min(n, 8)
        k = dict(op="evaluate", prec=c["prec"], M=M, na=n, nb=n, core=n - e, act=2 * e, level=6, n_chol=4 * M, n_w=c["n_w"])
        nd = int(round(math.exp(r.uniform(math.log(c["det_lo"]), math.log(c["det_hi"])))))
        out.append(dict(k, n_det=min(nd, _pair_count(k) // 2)))
    return out


def _network_inputs(c, seed):
    """Rows of a Green's function near the identity, and standardised targets."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    x = 0.07 * torch.randn((c["n_w"], c["n_in"]), device=DEV, generator=gen)
    x[:, ::217] += 1.0
    t = torch.randn((c["n_w"],), device=DEV, generator=gen)
    return x, t


def prepare(case, seed):
    c = dict(case)
    if c["op"] == "network":
        x, t = _network_inputs(c, seed)
        return dict(c=c, net=cv.MLP(c["n_in"], c["width"], device=0, seed=seed), x=x, t=t)
    if c["op"] == "batch":
        ctxs, walkers = [], []
        for i, m in enumerate(_members(c)):
            s, pa, pb, _, _ = _inputs(m, seed * 64 + i)
            ctxs.append(msd.Context(s, c["prec"], device=0))
            walkers.append((pa, pb))
        b = msd.Batch(ctxs)
        return dict(c=c, batch=b, walkers=walkers, outs=b.outputs(walkers))
    s, pa, pb, x, _ = _inputs(c, seed)
    st = dict(c=c, ctx=msd.Context(s, c["prec"], device=0), pa=pa, pb=pb)
    if c["op"] == "propagate":
        st |= dict(x=x, w=torch.ones(c["n_w"], dtype=torch.float64, device=DEV))
    return st


def run(state):
    op = state["c"]["op"]
    if op == "network":
        return state["net"].grad(state["x"], state["t"])
    if op == "batch":
        return state["batch"].evaluate(state["walkers"], state["outs"])
    ctx, pa, pb = state["ctx"], state["pa"], state["pb"]
    if op == "overlap":
        return ctx.overlap(pa, pb)
    if op == "force_bias":
        return ctx.force_bias(pa, pb, ovlp=True)
    if op == "energy":
        return ctx.local_energy(pa, pb, ovlp=True)
    if op == "evaluate":
        return ctx.evaluate(pa, pb)
    if op == "rdm":
        return ctx.rdm1(pa, pb)
    # a step works on its walkers in place: from the same walkers each time
    pa, pb, w = pa.clone(), pb.clone(), state["w"].clone()
    ratio = ctx.propagate(pa, pb, w, state["x"], 0.005, state["c"]["order"], state["c"]["qr"])
    return pa, pb, w, ratio


# --------------------------------------------------------------------- work
def work(case):
    """Bytes: walkers, Hamiltonian and determinant tables in, results out,
    once each. Flops: the reference inverse, a minor per string, a product
    pair per determinant, and the contractions with the Cholesky vectors that
    the quantity needs."""
    c = dict(case)
    if c["op"] == "network":
        p = c["width"] * (c["n_in"] + 2 * c["width"] + 4) + 1
        layers = c["width"] * (c["n_in"] + 2 * c["width"])
        return dict(bytes=4.0 * (2 * p + c["n_w"] * (c["n_in"] + 1)),
                    flops=2.0 * c["n_w"] * (2 * layers + 2 * c["width"] ** 2))
    if c["op"] == "batch":
        ws = [work(m) for m in _members(c)]
        return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))
    M, G, nw, nd = c["M"], c["n_chol"], c["n_w"], c["n_det"]
    tri = G * M * (M + 1) / 2.0                         # L is symmetric
    walkers = 16.0 * nw * M * (c["na"] + c["nb"])
    by = walkers + nd * (8.0 + 8.0)
    fl = 0.0
    rows, X = 0, []
    for n in (c["na"], c["nb"]):
        o, v, k = _levels(n, c)
        rows += n + v
        X.append(o * v)
        strings = sum(math.comb(o, i) * math.comb(v, i) for i in range(1, k + 1))
        fl += nw * 8.0 * (4.0 / 3.0 * n ** 3 + (M - n) * n * n)
        fl += nw * 8.0 * 4.0 * min(strings, nd)
    fl += nw * 4.0 * nd * 2.0
    bias = 4.0 * nw * G * rows * M
    energy = 0.0
    for n in (c["na"], c["nb"]):
        o, v, _ = _levels(n, c)
        energy += 4.0 * nw * n * (M - n) * G * (n + v)              # G L on the occupied rows
        energy += 8.0 * nw * G * (n * n * v + o * n * v)            # Lambda, Xi
    energy += 8.0 * nw * G * (X[0] * (X[0] + 1) / 2.0 + X[1] * (X[1] + 1) / 2.0 + X[0] * X[1])
    energy += nw * nd * 8.0 * 20.0                                  # opposite-spin terms at level ~2 x 2
    op = c["op"]
    if op == "overlap":
        return dict(bytes=by + 16.0 * nw, flops=fl)
    if op == "rdm":
        return dict(bytes=by + 32.0 * nw * M * M, flops=fl + 8.0 * nw * M * (X[0] + X[1]))
    by += 8.0 * tri
    if op == "force_bias":
        return dict(bytes=by + 16.0 * nw * (G + 1), flops=fl + bias)
    if op == "energy":
        return dict(bytes=by + 32.0 * nw, flops=fl + energy)
    if op == "evaluate":
        return dict(bytes=by + 16.0 * nw * (G + 2), flops=fl + bias + energy)
    step = 4.0 * nw * M * (M + 1) / 2.0 * G + nw * M * M * (c["na"] + c["nb"]) * (8.0 + 8.0 * c["order"])
    return dict(bytes=by + walkers + nw * (8.0 * G + 16.0 + 16.0), flops=2.0 * fl + bias + step)


# -------------------------------------------------------------------- exact
def _wick(c, seed_inputs, phi_a, phi_b, want):
    """Overlap, force bias, density matrix and local energy by the
    generalized Wick theorem in 64 bits, for a block of walkers."""
    s, _, _, _, (h, L, ia, ib) = seed_inputs
    nw, M, G = phi_a.shape[0], c["M"], c["n_chol"]
    coeff = torch.from_numpy(s.coeff).to(DEV)
    ids = [torch.from_numpy(ia).to(DEV), torch.from_numpy(ib).to(DEV)]
    need_b = want != "overlap"
    sp = []
    for n, phi in ((c["na"], phi_a), (c["nb"], phi_b)):
        st = _strings(n, c)
        o, v, _ = _levels(n, c)
        S = phi[:, :n]
        theta = torch.linalg.solve(S, phi, left=False)               # phi S^-1, [w][M][n]
        g = theta.transpose(1, 2).contiguous()                       # G[occ_j][r]
        A = g[:, c["core"]:n, n:c["core"] + c["act"]]                # [w][holes][particles]
        r, B = [], []
        for hh, pp, sg in st:
            k = hh.shape[1]
            sgn = torch.from_numpy(sg).to(DEV)
            if k == 0:
                r.append(torch.ones((nw, 1), dtype=C128, device=DEV))
                B.append(torch.zeros((nw, 1, o * v), dtype=C128, device=DEV) if need_b else None)
                continue
            hi = torch.from_numpy(hh - c["core"]).to(DEV)
            pi = torch.from_numpy(pp - n).to(DEV)
            minor = A[:, hi[:, :, None], pi[:, None, :]]             # [w][s][k][k]
            r.append(torch.linalg.det(minor) * sgn)
            if need_b:
                x = (hi[:, None, :] * v + pi[:, :, None]).reshape(1, -1, k * k).expand(nw, -1, -1)
                d = torch.zeros((nw, len(hh), o * v), dtype=C128, device=DEV)
                B.append(d.scatter_(2, x, torch.linalg.inv(minor).reshape(nw, -1, k * k)))
        sp.append(dict(n=n, o=o, v=v, g=g, det=torch.linalg.det(S), r=torch.cat(r, 1), B=torch.cat(B, 1) if need_b else None))
    a, b = sp
    Cm = torch.sparse_coo_tensor(torch.stack(ids), coeff, (a["r"].shape[1], b["r"].shape[1])).coalesce().to_sparse_csr()
    Ct = torch.sparse_coo_tensor(torch.stack(ids[::-1]), coeff, (b["r"].shape[1], a["r"].shape[1])).coalesce().to_sparse_csr()

    def times(m, z):                                                 # real sparse [p][q] on complex [q][t]
        return torch.view_as_complex((m @ torch.view_as_real(z.contiguous()).reshape(z.shape[0], -1)).reshape(m.shape[0], -1, 2))

    wa = a["r"] * times(Cm, b["r"].T).T
    wb = b["r"] * times(Ct, a["r"].T).T
    R = wa.sum(1)
    out = dict(ovlp=a["det"] * b["det"] * R)
    if want == "overlap":
        return out
    gts = []
    for q, w in ((a, wa), (b, wb)):
        n, core, act = q["n"], c["core"], c["act"]
        cof = (w[:, None, :] @ q["B"]).reshape(nw, q["o"], q["v"]) / R[:, None, None]   # [h][p]
        y = cof.transpose(1, 2) @ q["g"][:, core:n]                  # [p][c]
        gt = torch.zeros((nw, M, M), dtype=C128, device=DEV)
        gt[:, :n] = q["g"] - q["g"][:, :, n:core + act] @ y
        gt[:, n:core + act] += y
        gts.append(gt)
    out["rdm"] = torch.stack(gts, 1)
    if want == "rdm":
        return out
    t = torch.view_as_real((gts[0] + gts[1]).reshape(nw, M * M))
    Lf = L.reshape(G, M * M)
    out["vbias"] = torch.complex(t[..., 0] @ Lf.T, t[..., 1] @ Lf.T)
    if want == "force_bias":
        return out
    for q in sp:
        n, core, act, o, v = q["n"], c["core"], c["act"], q["o"], q["v"]
        cols = torch.cat([torch.arange(n), torch.arange(n, core + act)]).to(DEV)
        X = o * v
        for mats in ("h", "L"):
            m = h[None] if mats == "h" else L
            k = m.shape[0]
            rt = m[:, :, cols].permute(1, 0, 2).reshape(M, -1)       # [r][(g, col)]
            gv = torch.view_as_real(q["g"].reshape(nw * n, M))
            F = torch.complex(gv[..., 0] @ rt, gv[..., 1] @ rt).reshape(nw, n, k, -1).transpose(1, 2)
            T, FP = F[..., :n], F[..., n:]
            lam = FP - T @ q["g"][:, None, :, n:core + act]          # [w][g][j][p]
            v0 = torch.diagonal(T, dim1=2, dim2=3).sum(-1)
            if mats == "h":
                q["e1"], q["Y"] = v0[:, 0], lam[:, 0, core:].reshape(nw, X)
            else:
                q["v0"] = v0
                q["x"] = (T * T.transpose(2, 3)).sum((1, 2, 3))
                q["xi"] = (T[:, :, core:] @ lam).sum(1).reshape(nw, X)
                q["lam"] = lam[:, :, core:].reshape(nw, k, X).contiguous()
    V0 = a["v0"] + b["v0"]
    E = a["e1"] + b["e1"] + 0.5 * (V0 * V0).sum(1) - 0.5 * (a["x"] + b["x"])
    num = torch.zeros(nw, dtype=C128, device=DEV)
    for q, w in ((a, wa), (b, wb)):
        o, v = q["o"], q["v"]
        Y = q["Y"] + (V0[:, None, :] @ q["lam"])[:, 0] - q["xi"]
        K = q["lam"].transpose(1, 2) @ q["lam"]
        K = K - K.reshape(nw, o, v, o, v).transpose(2, 4).reshape(nw, o * v, o * v)
        e = (q["B"] @ Y[:, :, None])[..., 0] + 0.5 * ((q["B"] @ K) * q["B"]).sum(-1)
        num += (w * e).sum(1)
    Kab = a["lam"].transpose(1, 2) @ b["lam"]
    for i in range(nw):
        ub = times(Cm, b["r"][i, :, None] * b["B"][i])               # [alpha string][Xb]
        num[i] += ((a["r"][i, :, None] * (a["B"][i] @ Kab[i])) * ub).sum()
    out["e_loc"] = E + num / R
    return out


def _blocks(c, inputs, pa, pb, want):
    strings = sum(len(x[2]) for n in (c["na"], c["nb"]) for x in _strings(n, c))
    X = max(_levels(n, c)[0] * _levels(n, c)[1] for n in (c["na"], c["nb"]))
    per = 16.0 * (strings * (3 * X + 80) + (c["na"] + 8) * 2.5 * c["n_chol"] * (c["na"] + 10) + 8 * c["M"] ** 2)
    step = int(max(1, min(c["n_w"], 2.0e10 // per)))
    parts = [_wick(c, inputs, pa[i:i + step], pb[i:i + step], want) for i in range(0, c["n_w"], step)]
    return {k: torch.cat([p[k] for p in parts]) for k in parts[0]}


def _exact_step(c, inputs):
    s, pa, pb, x, (h, L, _, _) = inputs
    dt, G, M, nw = 0.005, c["n_chol"], c["M"], c["n_w"]
    old = _blocks(c, inputs, pa, pb, "force_bias")
    xbar = -1j * math.sqrt(dt) * old["vbias"]
    f = 1j * math.sqrt(dt) * (x - xbar)
    Lf = L.reshape(G, M * M)
    V = torch.complex(f.real @ Lf, f.imag @ Lf).reshape(nw, M, M)
    lf = L.permute(1, 0, 2).reshape(M, -1)
    ev, U = torch.linalg.eigh(h - 0.5 * (lf @ lf.T))
    E = ((U * torch.exp(-0.5 * dt * ev)) @ U.T).to(C128)
    new = []
    for phi in (pa, pb):
        t = E @ phi
        acc = t.clone()
        for k in range(1, c["order"] + 1):
            t = V @ t / k
            acc += t
        new.append(E @ acc)
    S = _blocks(c, inputs, new[0], new[1], "overlap")["ovlp"] / old["ovlp"]
    expo = (x * xbar - 0.5 * xbar * xbar).sum(1)
    w = S.abs() * torch.exp(expo.real) * torch.clamp(S.real / S.abs(), min=0)
    if c["qr"]:
        new = [_orthonormal(p) for p in new]
    return new[0], new[1], w, S


def _exact_network(c, seed):
    x, t = _network_inputs(c, seed)
    n, w = c["n_in"], c["width"]
    p = torch.from_numpy(_initial_parameters(n, w, seed)).to(DEV).double().requires_grad_()
    cut, at = [], 0
    for shape in ((w, n), (w,), (w, w), (w,), (w, w), (w,), (w,), (1,)):
        size = math.prod(shape)
        cut.append(p[at:at + size].reshape(shape))
        at += size
    z = x.double()
    for k in range(3):
        z = torch.nn.functional.gelu(z @ cut[2 * k].T + cut[2 * k + 1])
    loss = ((z @ cut[6] + cut[7] - t.double()) ** 2).mean()
    return loss.detach().reshape(1), torch.autograd.grad(loss, p)[0]


def _initial_parameters(n, w, seed):
    """The network's documented start: He-normal hidden weights, zero biases."""
    rng = np.random.default_rng(seed)
    parts = [rng.standard_normal(w * n) * np.sqrt(2.0 / n), np.zeros(w)]
    for _ in range(2):
        parts += [rng.standard_normal(w * w) * np.sqrt(2.0 / w), np.zeros(w)]
    parts += [rng.standard_normal(w) * np.sqrt(1.0 / w), np.zeros(1)]
    return np.concatenate(parts).astype(np.float32)


def exact(case, seed):
    c = dict(case)
    if c["op"] == "network":
        return _exact_network(c, seed)
    if c["op"] == "batch":
        out = []
        for i, m in enumerate(_members(c)):
            e = exact(m, seed * 64 + i)
            out.append(e)
        return out
    inputs = _inputs(c, seed)
    if c["op"] == "propagate":
        return _exact_step(c, inputs)
    want = c["op"]
    e = _blocks(c, inputs, inputs[1], inputs[2], want)
    if want == "overlap":
        return e["ovlp"]
    if want == "rdm":
        return e["rdm"]
    if want == "force_bias":
        return e["vbias"], e["ovlp"]
    if want == "energy":
        return e["e_loc"], e["ovlp"]
    return e["ovlp"], e["vbias"], e["e_loc"]
