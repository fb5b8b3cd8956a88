"""Performance cases of the walker-batched Slater-Jastrow DMC library.

Each case is one pass through the public entry points of
``paper_2504_07948_gb300.qmc`` on a seeded water cluster of ``synth``:

* ``dmc``      qmc_dmc steps at fixed population (with or without forces);
* ``vmc``      qmc_vmc sweeps with the E_L trace;
* ``evaluate`` qmc_evaluate: orbitals, FP64 inverses and E_L from scratch (the
  periodic rebuild of the incremental state);
* ``eloc``     qmc_eval_cached: the estimators from the maintained state;
* ``forces``   qmc_force_vjp: per-walker ionic derivatives and their weighted
  sum (the backward pass of the autograd function);
* ``batch``    qmc_batch_dmc with forces over clusters of uneven size.

Numbers of the mixed form carry FP32 accuracy and are returned as float32;
those of the FP64 form stay float64.  ``exact`` evaluates the fixed-configuration
paths in plain float64 torch; the sampling paths (chains of accept / reject
decisions) and determinant expansions have no such value.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2504_07948_gb300 import qmc as Q
from paper_2504_07948_gb300 import synth

TAU = 0.005


def _case(path, waters, walkers, precision, steps=1, delay=1, forces=False, dets=0, pp=False, warp=False, name=None):
    c = dict(path=path, waters=waters, walkers=walkers, precision=precision, steps=steps, delay=delay, forces=forces,
             dets=dets, pp=pp, warp=warp)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # the smallest production run: one water, energies only, a short block of DMC steps (launches and latency)
        _case("dmc", 1, 512, "fp64", steps=4, name="water1_dmc_fp64"),
        # the headline workload: 6-water cluster, 2048 walkers, FP64, DMC with forces every step
        _case("dmc", 6, 2048, "fp64", steps=2, forces=True, name="water6_dmc_forces_fp64"),
        # equilibration and sampling of the same cluster in the mixed form
        _case("vmc", 6, 2048, "mixed", steps=2, name="water6_vmc_mixed"),
        # the large cluster: delayed updates of rank 32, walker-tiled sweep
        _case("vmc", 32, 1024, "mixed", steps=1, delay=32, name="water32_vmc_mixed"),
        # the periodic FP64 rebuild and E_L of the large cluster
        _case("evaluate", 32, 256, "mixed", delay=32, name="water32_evaluate_mixed"),
        # a small ragged evaluation: odd walker count, 15 electrons per spin (geometry scans, tests)
        _case("evaluate", 3, 77, "fp64", name="water3_evaluate_fp64"),
        # force labels of the 6-water cluster in the mixed form (fused force kernel)
        _case("forces", 6, 2048, "mixed", name="water6_forces_mixed"),
        # forces of a large determinant, mixed (tensor-core GEMM path)
        _case("forces", 32, 512, "mixed", delay=32, name="water32_forces_mixed"),
        # forces of a large determinant, FP64
        _case("forces", 32, 256, "fp64", name="water32_forces_fp64"),
        # 10^4-determinant expansion: sampling by the table method
        _case("vmc", 6, 256, "mixed", dets=10_000, name="water6_msd10k_vmc_mixed"),
        # valence Hamiltonian: E_L with the non-local pseudopotential of every O
        _case("eloc", 32, 512, "mixed", delay=32, pp=True, name="water32_pp_eloc_mixed"),
        # many molecules of uneven size stepped together, forces on
        _case("batch", 16, 64, "fp64", steps=1, forces=True, name="uneven_batch_dmc_forces_fp64"),
    ]


def _spread(rng, lo, hi):
    """A whole number, uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of one listed kind: other cluster sizes, walker counts and options, its work at most the listed one's."""
    kind = rng.choice(listed())
    c = {k: v for k, v in kind.items() if k != "name"}
    if c["path"] == "batch":
        c["waters"] = rng.randint(2, 16)        # number of systems
        c["walkers"] = _spread(rng, 5, 64)
        c["forces"] = rng.random() < 0.7
        return c
    if c["dets"]:
        c["waters"] = rng.randint(3, 6)
        c["dets"] = _spread(rng, 100, 10_000)
    elif kind["waters"] <= 6:
        c["waters"] = rng.randint(1, 8)
    else:
        c["waters"] = rng.randint(9, 32)
        if c["path"] == "vmc":
            c["delay"] = rng.choice([8, 16, 32])
    if c["path"] == "dmc":
        c["forces"] = rng.random() < 0.6
        c["steps"] = rng.randint(1, 4)
    if c["path"] == "forces" and not c["dets"]:
        c["warp"] = rng.random() < 0.25
        c["pp"] = not c["warp"] and rng.random() < 0.25
    if c["path"] in ("evaluate", "eloc"):
        c["pp"] = rng.random() < 0.4 if c["path"] == "evaluate" else True
        c["precision"] = rng.choice(["fp64", "mixed"]) if c["path"] == "evaluate" else "mixed"
    c["walkers"] = _spread(rng, 24, 2048)
    top = max(work(x)["flops"] for x in listed() if x["path"] == c["path"] and x["precision"] == kind["precision"])
    while c["walkers"] > 8 and work(c)["flops"] > top:
        c["walkers"] = c["walkers"] * 9 // 10
    return c


@functools.lru_cache(maxsize=32)
def _system(waters, dets=0, pp=False):
    s = synth.water_system(waters)
    if pp:
        s = synth.with_pseudopotential(s)
    return synth.with_multidet(s, dets) if dets else s


def _batch_sizes(n):
    return [int(m) for m in synth.uneven_cluster_sizes(64)[:n]]


def _handle(system, case, seed):
    return Q.QMC(system, precision=case["precision"], recompute_period=100, seed=1 + seed % (1 << 31), cap_factor=2,
                 delay_rank=case["delay"], fixed_population=True, space_warp=case["warp"])


def _walkers(system, n, seed):
    return synth.initial_walkers(system, n, seed=seed)


def _weights(case, seed):
    rng = np.random.default_rng([seed, 1])
    return rng.normal(size=(2, case["walkers"]))


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    if case["path"] == "batch":
        systems = [_system(m) for m in _batch_sizes(case["waters"])]
        members = []
        for i, s in enumerate(systems):
            m = _handle(s, case, seed + 17 * i)
            m.set_walkers(_walkers(s, case["walkers"], [seed, i]))
            members.append(m)
        e = []
        for m in members:
            el = np.zeros(case["walkers"])
            Q.qmc_eval_cached(m.h, eloc=el)
            e.append(float(np.median(el)))
        return dict(case=case, members=members, batch=Q.Batch(members), e_trial=np.array(e),
                    R=[_empty(case["walkers"], s.n_elec, 3) for s in systems])
    s = _system(case["waters"], case["dets"], case["pp"])
    W, N, nn = case["walkers"], s.n_elec, s.n_nuc
    g = _handle(s, case, seed)
    g.set_walkers(_walkers(s, W, seed))
    st = dict(case=case, g=g)
    if case["path"] == "dmc":
        el = np.zeros(W)
        Q.qmc_eval_cached(g.h, eloc=el)
        st.update(e_trial=float(np.median(el)), R=_empty(W, N, 3))
    elif case["path"] == "vmc":
        st.update(trace=_empty(case["steps"], W), R=_empty(W, N, 3))
    elif case["path"] in ("evaluate", "eloc"):
        st.update(out=[_empty(W), _empty(W), _empty(W), _empty(W, N, 3)])
    else:
        gE, gL = torch.from_numpy(_weights(case, seed)).cuda()
        st.update(gE=gE, gL=gL, dR=_empty(nn, 3), pw=_empty(W, 2, nn, 3))
    return st


def _num(case, *xs):
    return [x.float() for x in xs] if case["precision"] == "mixed" else list(xs)


def run(state):
    case = state["case"]
    path = case["path"]
    if path == "batch":
        for m in state["members"]:
            Q.qmc_reset_estimators(m.h)
        out = state["batch"].dmc(case["steps"], TAU, state["e_trial"], forces_every=1 if case["forces"] else 0)
        for m, R in zip(state["members"], state["R"]):
            Q.qmc_get_walkers(m.h, R)
        res = [out["e_step"], out["pop"], torch.cat([R.reshape(-1) for R in state["R"]])]
        if case["forces"]:
            res.append(np.concatenate([m.force_estimate(Q.QMC_EST_DMC)[0] for m in state["members"]]))
        return res
    g = state["g"]
    if path == "dmc":
        Q.qmc_reset_estimators(g.h)
        out = g.dmc(case["steps"], TAU, state["e_trial"], forces_every=1 if case["forces"] else 0)
        state["e_trial"] = float(out["e_trial"][-1])   # the next block goes on from here
        Q.qmc_get_walkers(g.h, state["R"])
        res = [out["e_step"], out["pop"], out["e_trial"], state["R"]]
        if case["forces"]:
            res.append(g.force_estimate(Q.QMC_EST_DMC)[0])
        return res
    if path == "vmc":
        Q.qmc_vmc(g.h, case["steps"], TAU, 0, state["trace"])
        Q.qmc_get_walkers(g.h, state["R"])
        return _num(case, state["trace"], state["R"])
    if path in ("evaluate", "eloc"):
        logpsi, sign, el, grad = state["out"]
        (Q.qmc_evaluate if path == "evaluate" else Q.qmc_eval_cached)(g.h, logpsi, sign, el, grad)
        return [sign.to(torch.int32)] + _num(case, logpsi, el, grad)
    Q.qmc_force_vjp(g.h, state["gE"], state["gL"], state["dR"], state["pw"])
    return _num(case, state["dR"], state["pw"])


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def _work_one(s, case):
    """(flops, bytes) of a pass over one system: the dense products of the method (contraction, ratio and update of every
    move; E_L; the adjoint's products), and positions, inverses, coefficients and outputs once each."""
    W, N, nb, nn = case["walkers"], s.n_elec, s.n_basis, s.n_nuc
    path, steps = case["path"], case["steps"]
    item = 8 if case["precision"] == "fp64" else 4
    ns = (s.n_up, s.n_dn)
    n2, n3 = sum(n * n for n in ns), sum(n ** 3 for n in ns)
    sweep = sum(n * (10.0 * n * nb + 14.0 * n + 2.0 * n * n) for n in ns)
    eloc = 8.0 * n2 + 30.0 * N * (N + nn)
    if case["pp"]:   # u_k and chi(r') . u_k at twelve points of one nucleus per electron
        eloc += sum(2.0 * n * n * nb for n in ns) + 24.0 * N * nb
    force = sum(4.0 * n * n * nb + 2.0 * n ** 3 for n in ns) + 30.0 * N * nb
    table = 0.0
    if case["dets"]:   # virtual orbitals of a move and its table row, two small determinants per string of the moved spin
        nv = 20
        table = N * (10.0 * nv * nb + 4.0 * nv * s.n_up + 60.0 * case["dets"])
    pos, inv, coef = 24.0 * N * W, item * n2 * W, item * sum(ns) * nb
    if path in ("dmc", "vmc", "batch"):
        flops = steps * (sweep + table + eloc + (force if case["forces"] else 0.0)) * W
        return flops, 2 * pos + 2 * inv + coef + 8.0 * W * steps
    if path == "evaluate":
        return (10.0 * sum(n * n * nb for n in ns) + 2.0 * n3 + eloc) * W, 2 * pos + inv + coef + 24.0 * W
    if path == "eloc":
        return eloc * W, 2 * pos + 5 * inv + coef + 24.0 * W
    return force * W, pos + 5 * inv + coef + 48.0 * nn * W + 16.0 * W


def work(case):
    if case["path"] == "batch":
        parts = [_work_one(_system(m), case) for m in _batch_sizes(case["waters"])]
    else:
        parts = [_work_one(_system(case["waters"], 0, case["pp"]), case)]
    return {"flops": sum(p[0] for p in parts), "bytes": sum(p[1] for p in parts)}


# ---------------------------------------------------------------------------
# plain float64 values of the fixed-configuration paths
# ---------------------------------------------------------------------------

def _basis_tables(s):
    """Per shell padded primitives (alpha, normalised coefficient), per function its shell and its angular polynomial
    P(x) = p0 + p . x + x H x / 2."""
    shells = len(s.shell_l)
    width = int(max(s.shell_nprim))
    al, cn = np.zeros((shells, width)), np.zeros((shells, width))
    fn_shell, p0, p1, H = [], [], [], []
    off = 0
    r3 = math.sqrt(3.0)
    for k in range(shells):
        l, n = int(s.shell_l[k]), int(s.shell_nprim[k])
        a, c = s.alpha[off:off + n], s.coef[off:off + n].copy()
        off += n
        S = (2.0 * np.sqrt(a[:, None] * a[None, :]) / (a[:, None] + a[None, :])) ** (l + 1.5)
        norm = (2.0 * a / math.pi) ** 0.75 * (4.0 * a) ** (0.5 * l) / math.sqrt((1.0, 1.0, 3.0)[l])
        al[k, :n] = a
        cn[k, :n] = c * norm / math.sqrt(c @ S @ c)
        if l == 0:
            polys = [(1.0, np.zeros(3), np.zeros((3, 3)))]
        elif l == 1:
            polys = [(0.0, np.eye(3)[q], np.zeros((3, 3))) for q in range(3)]
        else:
            def sym(i, j, v):
                h = np.zeros((3, 3))
                h[i, j] = h[j, i] = v
                return h
            if s.shell_pure[k]:
                hs = [sym(0, 1, r3), sym(1, 2, r3), np.diag([-1.0, -1.0, 2.0]), sym(0, 2, r3), np.diag([r3, -r3, 0.0])]
            else:
                hs = [np.diag([2.0, 0, 0]), sym(0, 1, r3), sym(0, 2, r3), np.diag([0, 2.0, 0]), sym(1, 2, r3),
                      np.diag([0, 0, 2.0])]
            polys = [(0.0, np.zeros(3), h) for h in hs]
        for a0, a1, h in polys:
            fn_shell.append(k); p0.append(a0); p1.append(a1); H.append(h)
    t = lambda x: torch.as_tensor(np.array(x), dtype=torch.float64, device="cuda")  # noqa: E731
    ctr = torch.as_tensor(np.asarray(s.shell_center, dtype=np.int64), device="cuda")
    fs = torch.as_tensor(np.array(fn_shell), device="cuda")
    return dict(al=t(al), cn=t(cn), ctr=ctr, fs=fs, p0=t(p0), p1=t(p1), H=t(np.array(H)))


def _orbitals(s, T, r, nuc, derivs):
    """Orbital values [W, M, n_mo_used] at points r [W, M, 3] (nuclei [W, n_nuc, 3]); with derivs also gradients
    [W, M, 3, .] and Laplacians."""
    n = max(s.n_up, s.n_dn)
    C = torch.as_tensor(s.C[:n].T.copy(), device="cuda")   # [n_basis, n]
    x = r[:, :, None, :] - nuc[:, None, :, :]
    x = x[:, :, T["ctr"]]                                  # per shell
    t = (x * x).sum(-1)
    e = T["cn"] * torch.exp(-T["al"] * t[..., None])
    f0 = e.sum(-1)[..., T["fs"]]
    xf = x[:, :, T["fs"]]
    Hx = torch.einsum("wmfc,fcd->wmfd", xf, T["H"])
    P = T["p0"] + (xf * (T["p1"] + 0.5 * Hx)).sum(-1)
    val = (P * f0) @ C
    if not derivs:
        return val
    f1 = -(T["al"] * e).sum(-1)[..., T["fs"]]
    f2 = (T["al"] ** 2 * e).sum(-1)[..., T["fs"]]
    tf = t[..., T["fs"]]
    gP = T["p1"] + Hx
    trH = T["H"].diagonal(dim1=1, dim2=2).sum(-1)
    grad = torch.stack([(2.0 * P * xf[..., c] * f1 + gP[..., c] * f0) @ C for c in range(3)], dim=2)
    lap = (P * (6.0 * f1 + 4.0 * tf * f2) + 4.0 * (gP * xf).sum(-1) * f1 + trH * f0) @ C
    return val, grad, lap


def _pair(a, b, r):
    q = 1.0 / (1.0 + b * r)
    return a * r * q, a * q * q, -2.0 * a * b * q ** 3


def _like_spin(s):
    up = torch.arange(s.n_elec, device="cuda") < s.n_up
    return torch.where(up[:, None] == up[None, :], s.a_par, s.a_anti).to(torch.float64)


def _jastrow(s, r, nuc):
    """J, its gradient and Laplacian per electron, and the pair distances."""
    N = s.n_elec
    eye = torch.eye(N, device="cuda", dtype=torch.float64)
    d = r[:, :, None, :] - r[:, None, :, :]
    ree = ((d * d).sum(-1) + eye).sqrt()                   # ones on the diagonal, masked below
    off = 1.0 - eye
    u, du, d2u = _pair(_like_spin(s) * off, s.b_ee, ree)
    x = r[:, :, None, :] - nuc[:, None, :, :]
    ren = (x * x).sum(-1).sqrt()
    a_en = torch.as_tensor(s.a_en, device="cuda")
    v, dv, d2v = _pair(a_en, s.b_en, ren)
    J = 0.5 * u.sum((1, 2)) + v.sum((1, 2))
    g = ((du / ree)[..., None] * d).sum(2) + ((dv / ren)[..., None] * x).sum(2)
    lap = (d2u + 2.0 * du / ree).sum(2) + (d2v + 2.0 * dv / ren).sum(2)
    return J, g, lap, ree, ren, off


def _philox(c, key):
    """Philox4x32-10 of counters c [..., 4] (uint64 arrays holding 32-bit words)."""
    m = np.uint64(0xFFFFFFFF)
    x = [c[..., k].astype(np.uint64) for k in range(4)]
    k0, k1 = np.uint64(key & 0xFFFFFFFF), np.uint64(key >> 32)
    for r in range(10):
        if r:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m, (k1 + np.uint64(0xBB67AE85)) & m
        p0, p1 = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(p1 >> np.uint64(32)) ^ x[1] ^ k0, p1 & m, (p0 >> np.uint64(32)) ^ x[3] ^ k1, p0 & m]
    return x


def _rotations(s, walkers, seed):
    """Shoemake rotations [len(walkers), n_nuc, 3, 3] of the quadrature rule at sweep counter 0."""
    c = np.zeros((len(walkers), s.n_nuc, 4), dtype=np.uint64)
    c[..., 1] = np.arange(s.n_nuc, dtype=np.uint64)[None, :]
    c[..., 2] = np.asarray(walkers, dtype=np.uint64)[:, None]
    c[..., 3] = 3
    u = [(w.astype(np.float64) + 0.5) * 2.0 ** -32 for w in _philox(c, seed)[:3]]
    a, b = np.sqrt(1.0 - u[0]), np.sqrt(u[0])
    x, y = a * np.sin(2 * np.pi * u[1]), a * np.cos(2 * np.pi * u[1])
    z, w = b * np.sin(2 * np.pi * u[2]), b * np.cos(2 * np.pi * u[2])
    m = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                  2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                  2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], axis=-1)
    return torch.as_tensor(m.reshape(len(walkers), s.n_nuc, 3, 3), device="cuda")


def _radial_pp(s, k, r):
    return float(s.pp_beta[k]) * r ** (int(s.pp_n[k]) - 2) * torch.exp(-float(s.pp_alpha[k]) * r * r)


def _nonlocal(s, T, r, nuc, inv, rot):
    """Non-local pseudopotential energy per walker (locality approximation)."""
    W, N = r.shape[:2]
    quad, qw = (torch.as_tensor(v, device="cuda") for v in (s.pp_quad, s.pp_qw))
    x = r[:, :, None, :] - nuc[:, None, :, :]
    dist = (x * x).sum(-1).sqrt()
    rcut = torch.as_tensor(s.pp_rcut, device="cuda")
    w, i, a = torch.nonzero(dist < rcut, as_tuple=True)
    if w.numel() == 0:
        return r.new_zeros(W)
    x, dist = x[w, i, a], dist[w, i, a]
    dq = torch.einsum("pcd,qd->pqc", rot[w, a], quad)
    cos = (dq * x[:, None, :]).sum(-1) / dist[:, None]
    pts = nuc[w, a][:, None, :] + dist[:, None, None] * dq            # [pairs, nq, 3]
    phi = _orbitals(s, T, pts, nuc[w], False)
    det = torch.zeros_like(cos)
    for spin, (n, i0) in enumerate(((s.n_up, 0), (s.n_dn, s.n_up))):
        sel = torch.nonzero((i >= i0) & (i < i0 + n)).squeeze(1)
        if sel.numel():
            col = inv[spin][w[sel], :, i[sel] - i0]                   # A^-1 e_i
            det = det.index_copy(0, sel, torch.einsum("pqj,pj->pq", phi[sel][..., :n], col))
    mask = (torch.arange(N, device="cuda")[None, :] != i[:, None]).to(torch.float64)[:, None, :]
    amp = _like_spin(s)[i][:, None, :] * mask
    rj = r[w][:, None, :, :]

    def u_of(p):                                                      # Jastrow terms of electron i placed at p
        d2 = ((p[:, :, None, :] - rj) ** 2).sum(-1)
        ree = (d2 + (1.0 - mask)).sqrt()
        ren = ((p[:, :, None, :] - nuc[w][:, None, :, :]) ** 2).sum(-1).sqrt()
        a_en = torch.as_tensor(s.a_en, device="cuda")
        return _pair(amp, s.b_ee, ree)[0].sum(-1) + _pair(a_en, s.b_en, ren)[0].sum(-1)

    ratio = det * torch.exp(u_of(pts) - u_of(r[w, i][:, None, :]))
    legendre = (torch.ones_like(cos), cos, 1.5 * cos ** 2 - 0.5, 2.5 * cos ** 3 - 1.5 * cos)
    weight = torch.zeros_like(cos)
    for k in range(len(s.pp_l)):
        l = int(s.pp_l[k])
        if l >= 0:
            here = (a == int(s.pp_nuc[k])).to(torch.float64) * _radial_pp(s, k, dist)
            weight = weight + (2 * l + 1) * here[:, None] * legendre[l]
    return r.new_zeros(W).index_add(0, w, (weight * ratio * qw).sum(-1))


def _local_energy(s, T, r, nuc, rot):
    """ln|psi|, sign, E_L and grad ln|psi| of walkers r [W, N, 3] at nuclei [W, n_nuc, 3]."""
    phi, dphi, lphi = _orbitals(s, T, r, nuc, True)
    J, gJ, lJ, ree, ren, off = _jastrow(s, r, nuc)
    logdet, sign, gD, lD, inv = 0.0, 1.0, [], [], []
    for n, i0 in ((s.n_up, 0), (s.n_dn, s.n_up)):
        A = phi[:, i0:i0 + n, :n]
        sg, ld = torch.linalg.slogdet(A)
        Ai = torch.linalg.inv(A)
        logdet, sign = logdet + ld, sign * sg
        gD.append(torch.einsum("wicj,wji->wic", dphi[:, i0:i0 + n, :, :n], Ai))
        lD.append(torch.einsum("wij,wji->wi", lphi[:, i0:i0 + n, :n], Ai))
        inv.append(Ai)
    gD, lD = torch.cat(gD, 1), torch.cat(lD, 1)
    Z = torch.as_tensor(s.Z, device="cuda")
    kin = -0.5 * (lD + lJ + 2.0 * (gJ * gD).sum(-1) + (gJ * gJ).sum(-1)).sum(1)
    pot = 0.5 * (off / ree).sum((1, 2)) - (Z / ren).sum((1, 2))
    dn = nuc[:, :, None, :] - nuc[:, None, :, :]
    upper = torch.triu(torch.ones(s.n_nuc, s.n_nuc, device="cuda", dtype=torch.float64), 1)
    rnn = ((dn * dn).sum(-1) + (1.0 - upper)).sqrt()
    pot = pot + (Z[:, None] * Z[None, :] * upper / rnn).sum((1, 2))
    if rot is not None:
        for k in range(len(s.pp_l)):
            if int(s.pp_l[k]) < 0:
                pot = pot + _radial_pp(s, k, ren[:, :, int(s.pp_nuc[k])]).sum(1)
        pot = pot + _nonlocal(s, T, r, nuc, inv, rot)
    return J + logdet, sign, kin + pot, gJ + gD


def _warp(r, nuc, dE, dL, gE, gL):
    """Space-warped ionic derivatives from the plain ones and the electron-coordinate ones (weights |r - R|^-4)."""
    x = r[:, :, None, :] - nuc[:, None, :, :]
    d2 = (x * x).sum(-1)
    F = d2 ** -2
    S = F.sum(-1, keepdim=True)
    om = F / S
    gF = -4.0 * x * (F / d2)[..., None]
    gom = (gF - om[..., None] * gF.sum(2, keepdim=True)) / S[..., None]
    return (dE + torch.einsum("wia,wic->wac", om, gE),
            dL + torch.einsum("wia,wic->wac", om, gL) + 0.5 * gom.sum(1))


def exact(case, seed):
    if case["path"] not in ("evaluate", "eloc", "forces") or case["dets"]:
        return None
    s = _system(case["waters"], 0, case["pp"])
    T = _basis_tables(s)
    R = torch.from_numpy(np.ascontiguousarray(_walkers(s, case["walkers"], seed))).cuda()
    W = case["walkers"]
    chunk = max(1, 400_000 // (s.n_elec * s.n_basis))
    forces = case["path"] == "forces"
    parts = []
    for w0 in range(0, W, chunk):
        r = R[w0:w0 + chunk].clone()
        nuc = torch.as_tensor(s.R, device="cuda").expand(r.shape[0], -1, -1).clone()
        rot = _rotations(s, np.arange(w0, w0 + r.shape[0]), 1 + seed % (1 << 31)) if case["pp"] else None
        if forces:
            nuc.requires_grad_(True)
            r.requires_grad_(case["warp"])
        with torch.set_grad_enabled(forces):
            logpsi, sign, el, grad = _local_energy(s, T, r, nuc, rot)
        if not forces:
            parts.append((sign.to(torch.int32), logpsi, el, grad))
            continue
        leaves = [nuc, r] if case["warp"] else [nuc]
        gE = torch.autograd.grad(el.sum(), leaves, retain_graph=True)
        gL = torch.autograd.grad(logpsi.sum(), leaves)
        dE, dL = gE[0], gL[0]
        if case["warp"]:
            dE, dL = _warp(r.detach(), nuc.detach(), dE, dL, gE[1], gL[1])
        parts.append((dE, dL))
    cols = [torch.cat(c) for c in zip(*parts)]
    if not forces:
        return cols
    g = torch.from_numpy(_weights(case, seed)).cuda()
    return [torch.einsum("w,wac->ac", g[0], cols[0]) + torch.einsum("w,wac->ac", g[1], cols[1]),
            torch.stack(cols, dim=1)]
