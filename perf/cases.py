"""What the performance of this framework is measured on.

The cases are the calls of an XTRG run (arXiv:1801.00142): one beta doubling of
an MPO thermal state followed by its row of thermodynamics, in each arithmetic
and over the bond dimensions that a cooling schedule passes through; the
observables and the entanglement of a state on their own; a Taylor step
between grid points; a small batch of interleaved grids from the series
initialisation on; and the tensor-core contraction primitive that the
doublings are built from.  Bonds go up to 256: beyond, a doubling that meets a
rank-deficient basis takes exact splits of several seconds each.

The states are thermal-like MPOs made here from the seed, without this
repository's code: a Trotter product of XXZ gates, its bond cut to the D
largest weights, brought to right-canonical form.  Bond profile, spectrum and
gauge freedom are those of a state that a doubling returns.  The gauge of a
compressed MPO is arbitrary (degenerate singular values), so the new state is
returned as what does not depend on it: the dense operator of a short chain,
the thermodynamics and the magnetisation moments of a long one.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1801_00142_gb300 import _lib
from paper_1801_00142_gb300.batch import run_batch
from paper_1801_00142_gb300.engine import XTRG
from paper_1801_00142_gb300.hamiltonians import magnetization_power, xxz_chain

DEV = "cuda:0"


def listed():
    return [
        # one contraction of a short or young chain (bonds of a few tens): latency
        {"name": "gemm_small", "kind": "gemm", "M": 60, "N": 44, "K": 52, "batch": 1,
         "planes": 3, "nprod": 6, "splitk": 1, "nn": False},
        # a batched substep with ragged edges, B row-major, in the 16-bit split
        {"name": "gemm_nn_ragged", "kind": "gemm", "M": 250, "N": 330, "K": 201, "batch": 33,
         "planes": 2, "nprod": 3, "splitk": 1, "nn": True},
        # the two-site contraction C_E at D* = 256: 1024 x 1024 x 256^2
        {"name": "gemm_ce", "kind": "gemm", "M": 1024, "N": 1024, "K": 65536, "batch": 1,
         "planes": 3, "nprod": 6, "splitk": 4, "nn": False},
        # whole runs of interleaved tau0 grids, series initialisation included
        {"name": "batch_zshift", "kind": "batch", "L": 10, "D": 32, "grids": 4, "doublings": 2,
         "sweeps": 2},
        # FP64 doubling of a short chain without truncation (the parity sizes)
        {"name": "double_fp64_dense", "kind": "dense", "L": 7, "D": 64, "sweeps": 1,
         "prec": "fp64", "keep": True, "hot": False},
        # FP64 doubling early in a schedule, below beta = 1/4, where bonds are small
        {"name": "double_fp64_early", "kind": "double", "L": 32, "D": 40, "sweeps": 1,
         "prec": "fp64", "keep": True, "hot": False},
        # the smallest chains and bonds of the batched workload: launches count
        {"name": "double_x6_small", "kind": "double", "L": 16, "D": 64, "sweeps": 4,
         "prec": "bf16x6", "keep": True, "hot": True},
        # the headline step: 64 sites, D* = 256, 4 sweeps
        {"name": "double_x6_headline", "kind": "double", "L": 64, "D": 256, "sweeps": 4,
         "prec": "bf16x6", "keep": True, "hot": True},
        # the 16-bit split; bonds that are no multiple of a tile, the halves rebuilt
        # instead of resident
        {"name": "double_x3_ragged", "kind": "double", "L": 20, "D": 173, "sweeps": 2,
         "prec": "bf16x3", "keep": False, "hot": True},
        # a Taylor step between two grid points
        {"name": "settn_step", "kind": "settn", "L": 8, "D": 24, "order": 3, "sweeps": 1,
         "hot": False},
        # the row of a saturated state with the Hermiticity diagnostic (the default)
        {"name": "observables", "kind": "observables", "L": 64, "D": 256},
        # entanglement profile of a state
        {"name": "entanglement", "kind": "entanglement", "L": 12, "D": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "batch", "dense", "fp64", "mixed", "mixed", "mixed",
                       "settn", "observables", "entanglement"])
    if kind == "gemm":
        M, N = _log_int(rng, 17, 1100), _log_int(rng, 17, 1100)
        K = _log_int(rng, 16, min(65536, 60000000000 // (M * N)))
        batch = _log_int(rng, 1, max(1, min(64, 100000000 // (M * N + (M + N) * K))))
        planes, nprod = rng.choice([(3, 6), (3, 6), (2, 3), (3, 1)])
        return {"kind": kind, "M": M, "N": N, "K": K, "batch": batch, "planes": planes,
                "nprod": nprod, "splitk": rng.choice([1, 1, 2, 3, 8]), "nn": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": kind, "L": rng.randint(6, 10), "D": rng.randint(20, 32),
                "grids": rng.randint(2, 4), "doublings": rng.randint(1, 2), "sweeps": 2}
    if kind == "dense":
        prec = rng.choice(["fp64", "fp64", "bf16x6"])
        return {"kind": kind, "L": rng.randint(4, 7), "D": 64, "sweeps": 1, "prec": prec,
                "keep": rng.random() < 0.5, "hot": prec != "fp64"}
    if kind == "fp64":
        return {"kind": "double", "L": rng.randint(6, 32), "D": rng.randint(12, 40), "sweeps": 1,
                "prec": "fp64", "keep": True, "hot": False}
    if kind == "mixed":
        keep = rng.random() < 0.7
        return {"kind": "double", "L": _log_int(rng, 8, 64), "D": _log_int(rng, 40, 256),
                "sweeps": rng.randint(1, 4 if keep else 2),
                "prec": rng.choice(["bf16x6", "bf16x6", "bf16x3"]), "keep": keep, "hot": True}
    if kind == "settn":
        return {"kind": kind, "L": rng.randint(5, 9), "D": rng.randint(12, 24),
                "order": rng.randint(2, 4), "sweeps": 1, "hot": False}
    if kind == "observables":
        return {"kind": kind, "L": _log_int(rng, 8, 64), "D": _log_int(rng, 16, 256)}
    return {"kind": kind, "L": rng.randint(6, 12), "D": rng.randint(12, 64)}


# ------------------------------------------------------------------ inputs
def _rng(case, seed):
    return np.random.default_rng([seed, 1801])


def _gate(Delta, step):
    """Schmidt factors of exp(-step h), h = Sx Sx + Sy Sy + Delta Sz Sz: X[s][t][a], Y[a][s][t]."""
    sz, sp = np.diag([0.5, -0.5]), np.array([[0.0, 1.0], [0.0, 0.0]])
    h = 0.5 * (np.kron(sp, sp.T) + np.kron(sp.T, sp)) + Delta * np.kron(sz, sz)
    w, v = np.linalg.eigh(h)
    g = (v * np.exp(-step * w)) @ v.T
    g = g.reshape(2, 2, 2, 2).transpose(0, 2, 1, 3).reshape(4, 4)
    u, s, vt = np.linalg.svd(g)
    r = np.sqrt(s)
    return (u * r).reshape(2, 2, 4), (r[:, None] * vt).reshape(4, 2, 2), s


def _thermal_state(L, D, Delta, beta):
    """Right-canonical sites [Dl][2][2][Dr] (torch, on the GPU) and the log of the norm."""
    layers = max(1, math.ceil(math.log(D, 4) - 1e-9))
    X, Y, s = _gate(Delta, beta / layers)
    ident_l, ident_r = np.zeros((4, 2, 2)), np.zeros((2, 2, 4))
    ident_l[0], ident_r[:, :, 0] = np.eye(2), np.eye(2)
    # the D heaviest index tuples of the bond of a product of `layers` steps
    w = np.ones(1)
    for _ in range(layers):
        w = (w[:, None] * s[None, :]).reshape(-1)
    keep = torch.from_numpy(np.sort(np.argsort(-w, kind="stable")[:D])).to(DEV)

    def layered(i):
        # the step applies the gates on (i, i+1) with i odd first, then those with i even
        left = Y if i > 0 else ident_l
        right = X if i < L - 1 else ident_r
        T = (np.einsum("sua,but->bsta", right, left) if i % 2 == 0
             else np.einsum("bsu,uta->bsta", left, right))
        T = torch.from_numpy(np.ascontiguousarray(T)).to(DEV)
        P = T
        for _ in range(layers - 1):
            P = torch.einsum("lsur,mutp->lmstrp", P, T).reshape(
                P.shape[0] * 4, 2, 2, P.shape[3] * 4)
        P = P[:1] if i == 0 else P[keep]
        return (P[..., :1] if i == L - 1 else P[..., keep]).contiguous()

    kinds = {}
    sites = []
    for i in range(L):
        key = (i == 0, i == L - 1, i % 2)
        if key not in kinds:
            kinds[key] = layered(i)
        sites.append(kinds[key])
    # bonds near the left end: at most 4^i
    for i in range(L - 1):
        dl, dr = sites[i].shape[0], sites[i].shape[3]
        if 4 * dl >= dr:
            break
        m = sites[i].reshape(4 * dl, dr)
        sites[i] = torch.eye(4 * dl, dtype=torch.float64, device=DEV).reshape(dl, 2, 2, 4 * dl)
        sites[i + 1] = torch.einsum("ab,bstc->astc", m, sites[i + 1])
    lnc = 0.0
    for i in range(L - 1, 0, -1):
        dl = sites[i].shape[0]
        q, r = torch.linalg.qr(sites[i].reshape(dl, -1).T)
        k = q.shape[1]
        nrm = float(r.norm())
        lnc += math.log(nrm)
        sites[i] = q.T.reshape(k, 2, 2, -1).contiguous()
        sites[i - 1] = torch.einsum("astb,cb->astc", sites[i - 1], r / nrm)
    nrm = float(sites[0].norm())
    sites[0] = sites[0] / nrm
    return sites, lnc + math.log(nrm)


def _physics(case, seed):
    """Coupling and inverse temperature of the state, from the seed: the
    tensor-core doublings start at beta = 1/4 and the bonds they need grow as
    the chain cools; the FP64 ones come before them."""
    r = _rng(case, seed)
    Delta = float(r.uniform(0.1, 1.5))
    z = float(r.uniform(0.0, 1.0))
    if case.get("hot", True):
        return Delta, 2.0 ** z * max(0.25, case["D"] / 256)
    return Delta, 2.0 ** (z - 4.0)


def _gemm_inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    M, N, K, b = case["M"], case["N"], case["K"], case["batch"]
    kw = dict(generator=g, device=DEV, dtype=torch.float64)
    # operands of a contraction over a fused bond: weights fall along it
    fall = torch.exp2(-6.0 * torch.arange(K, device=DEV, dtype=torch.float64) / K)
    A = torch.randn(b, M, K, **kw).mul_(fall)
    B = torch.randn(b, K, N, **kw) if case["nn"] else torch.randn(b, N, K, **kw)
    return A, B


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B = _gemm_inputs(case, seed)
        size = (_lib.xtrg_tc_gemm_nn_workspace_bytes if case["nn"]
                else _lib.xtrg_tc_gemm_workspace_bytes)
        n = size(case["M"], case["N"], case["K"], case["batch"], case["planes"], case["splitk"])
        ws = torch.empty(n + 256, dtype=torch.uint8, device=DEV)
        C = torch.empty(case["batch"], case["M"], case["N"], dtype=torch.float64, device=DEV)
        return {"case": case, "A": A, "B": B, "C": C, "ws": ws,
                "ptr": (ws.data_ptr() + 255) // 256 * 256, "bytes": n}
    if kind == "batch":
        return {"case": case, "items": _batch_items(case, seed)}
    Delta, beta = _physics(case, seed)
    sites, lnc = _thermal_state(case["L"], case["D"], Delta, beta)
    eng = XTRG.xxz(case["L"], 1.0, Delta, tau0=2.0 ** -12, dstar=case["D"],
                   sweeps=case.get("sweeps", 4), prec=case.get("prec", "fp64"),
                   beta_switch=0.0, keep_parts=case.get("keep", True), device=DEV)
    eng.set_state([s.cpu().numpy() for s in sites], lnc, beta, right_canonical=True)
    state = {"case": case, "eng": eng}
    if kind in ("double", "dense", "settn"):
        # a step is the doubling and its thermodynamics; the diagnostic of
        # Hermiticity is a case of its own
        eng.set_herm_check(False)
        state["ckpt"] = eng.checkpoint()
        state["beta"] = beta
        state["m2"] = magnetization_power(case["L"], 2)
    return state


def _batch_items(case, seed):
    r = _rng(case, seed)
    Delta = float(r.uniform(0.1, 1.5))
    first = 2.0 ** (-7.0 + float(r.uniform(0.0, 1.0)))
    dims, sites = xxz_chain(case["L"], 1.0, Delta)
    return [(dims, sites, case["doublings"],
             dict(tau0=first * 2.0 ** (k / case["grids"]), order=4, dstar=case["D"],
                  sweeps=case["sweeps"])) for k in range(case["grids"])]


ROW = ("beta", "lnZ", "f", "u", "c")


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gemm":
        call = _lib.xtrg_tc_gemm_nn if case["nn"] else _lib.xtrg_tc_gemm
        C = state["C"]
        call(state["A"].data_ptr(), state["B"].data_ptr(), C.data_ptr(), case["M"], case["N"],
             case["K"], case["batch"], case["planes"], case["nprod"], case["splitk"],
             state["ptr"], state["bytes"], torch.cuda.current_stream().cuda_stream)
        return C.float()   # FP32-accurate values in an FP64 array: a program keeps 32 bits
    if kind == "batch":
        runs = run_batch(state["items"])
        return {k: np.array([[row[k] for row in rows] for rows in runs]) for k in ROW}
    eng = state["eng"]
    if kind == "observables":
        o = eng.observables()
        return {k: o[k] for k in ROW + ("herm_defect", "max_bond")}
    if kind == "entanglement":
        return eng.entanglement()
    eng.restore(state["ckpt"])
    if kind == "settn":
        eng.settn_step(state["beta"], case["order"])
        o = eng.observables()
        return {k: o[k] for k in ROW + ("max_bond",)}
    eng.double()
    o = eng.observables()
    # c is a difference of numbers some 10^2 times as large: of a state that
    # carries 24 bits it says less than u and the moment
    row = ROW if case["prec"] == "fp64" else ROW[:-1]
    out = {k: o[k] for k in row + ("lnZ2", "max_bond")}
    if kind == "double":
        out["m2"] = eng.expectation(*state["m2"])
        return out
    sites, lnc, _ = eng.get_state()
    v = sites[0][0]
    for w in sites[1:]:
        v = np.einsum("stb,buvc->sutvc", v, w, optimize=True).reshape(
            v.shape[0] * 2, v.shape[1] * 2, w.shape[3])
    rho = v[:, :, 0] * math.exp(lnc)
    # the operator in the precision of its arithmetic
    out["rho"] = rho if case["prec"] == "fp64" else rho.astype(np.float32)
    return out


# ------------------------------------------------------------------ work
def _bonds(L, D):
    return [min(D, 4 ** min(i, L - i, 8)) for i in range(L + 1)]


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K, b = (case[k] for k in ("M", "N", "K", "batch"))
        return {"bytes": 8.0 * b * (M * K + N * K + M * N), "flops": 2.0 * b * M * N * K}
    L = case["L"]
    d = _bonds(L, case["D"])
    site = sum(8.0 * d[i] * 4 * d[i + 1] for i in range(L))
    if kind == "observables":
        # E and H E transfers of Tr rho, Tr H rho, Tr H^2 rho (bond 5) and the
        # two D x D transfers of the Hermiticity diagnostic
        fl = sum(2.0 * d[i] * 4 * d[i + 1] * (1 + 5 + 25) +
                 2 * 2.0 * 4 * d[i] * d[i + 1] * (d[i] + d[i + 1]) for i in range(L))
        return {"bytes": site, "flops": fl}
    if kind == "entanglement":
        # one orthogonalisation and one split of every site
        return {"bytes": site, "flops": sum(6.0 * 4 * d[i] * d[i + 1] * d[i + 1]
                                            for i in range(L))}
    halves = []   # cost of the half of the environment at each site, and its update
    for i in range(L):
        l, r = d[i], d[i + 1]
        half = 8.0 * l * l * l * r + 8.0 * l * l * r * r * 2
        halves.append((half, 8.0 * l * r * r * r))
    once = sum(h + e for h, e in halves)
    upd = 0.0
    for i in range(L - 1):
        upd += 32.0 * d[i] * d[i + 2] * d[i + 1] ** 2 + halves[i][0] + halves[i][1]
    if kind == "settn":
        # each term: H (bond 5) times the last one; then the sum of the terms
        # against the compressed MPO
        fl = 0.0
        for i in range(L - 1):
            term = 2 * (8.0 * d[i] ** 2 * 5 * d[i + 1] + 16.0 * d[i] * d[i + 1] ** 2 * 5 +
                        16.0 * 5 * d[i] * d[i + 1] * d[i + 2])
            fl += case["order"] * term + (case["order"] + 1) * 48.0 * d[i] * d[i + 1] * d[i + 2]
        return {"bytes": 2 * site, "flops": 2 * case["sweeps"] * fl}
    if kind == "batch":
        return {"bytes": case["grids"] * site,
                "flops": case["grids"] * case["doublings"] * (once + 2 * case["sweeps"] * upd)}
    return {"bytes": 2 * site, "flops": once + 2 * case["sweeps"] * upd}


# ------------------------------------------------------------------ exact


def _xxz_mpo(L, Delta):
    """Automaton MPO of sum Sx Sx + Sy Sy + Delta Sz Sz, bond 5."""
    sz, sp, one = np.diag([0.5, -0.5]), np.array([[0.0, 1.0], [0.0, 0.0]]), np.eye(2)
    W = np.zeros((5, 2, 2, 5))
    W[0, :, :, 0] = one
    W[0, :, :, 1], W[1, :, :, 4] = 0.5 * sp, sp.T
    W[0, :, :, 2], W[2, :, :, 4] = 0.5 * sp.T, sp
    W[0, :, :, 3], W[3, :, :, 4] = Delta * sz, sz
    W[4, :, :, 4] = one
    return [W[:1] if i == 0 else W[..., 4:] if i == L - 1 else W for i in range(L)]


def _operator(sites):
    """Dense operator of a short MPO."""
    v = torch.ones(1, 1, 1, dtype=torch.float64, device=DEV)
    for w in sites:
        w = torch.as_tensor(w, device=DEV, dtype=torch.float64)
        v = torch.einsum("stb,buvc->sutvc", v, w).reshape(
            v.shape[0] * 2, v.shape[1] * 2, w.shape[3])
    return v[:, :, 0]


def _m2_plain(L):
    """MPO of (sum Sz)^2, bond 3: index counts the factors already placed."""
    m = np.diag([0.5, -0.5])
    W = np.zeros((3, 2, 2, 3))
    for p in range(3):
        W[p, :, :, p] = np.eye(2)
    W[0, :, :, 1], W[1, :, :, 2], W[0, :, :, 2] = 2.0 * m, m, m @ m
    return [W[:1] if i == 0 else W[..., 2:] if i == L - 1 else W for i in range(L)]


def _mean(ops, layer, square):
    """Log-scaled Tr(O R) with R = rho^T rho (square) or rho: (mantissa, log)."""
    E, ln = None, 0.0
    for O, w in zip(ops, layer):
        O = torch.as_tensor(np.ascontiguousarray(O), device=DEV, dtype=torch.float64)
        if square:
            # R[s][u] = sum_t w[t][s] w[t][u];  Tr(O R) = sum O[u][s] R[s][u]
            if E is None:
                E = torch.ones(1, 1, 1, dtype=torch.float64, device=DEV)
            X = torch.einsum("hab,atsc->hbtsc", E, w)
            X = torch.einsum("husk,hbtsc->kbtuc", O, X)
            E = torch.einsum("kbtuc,btud->kcd", X, w)
        else:
            if E is None:
                E = torch.ones(1, 1, dtype=torch.float64, device=DEV)
            X = torch.einsum("ha,astc->hstc", E, w)
            E = torch.einsum("htsk,hstc->kc", O, X)
        m = float(E.abs().max())
        E, ln = E / m, ln + math.log(m)
    return float(E.reshape(-1)[0]), ln


def _row(sites, lnc, beta, Delta, square, m2):
    L = len(sites)
    one = [np.eye(2).reshape(1, 2, 2, 1)] * L
    H = _xxz_mpo(L, Delta)
    HH = [np.einsum("asub,cutd->acstbd", W, W).reshape(W.shape[0] ** 2, 2, 2, W.shape[3] ** 2)
          for W in H]
    t0, l0 = _mean(one, sites, square)
    lnZ = math.log(t0) + l0 + (2.0 * lnc if square else lnc)
    avg = []
    for ops in (H, HH) + ((_m2_plain(L),) if m2 else ()):
        t, ln = _mean(ops, sites, square)
        avg.append(t / t0 * math.exp(ln - l0))
    out = {"beta": beta, "lnZ": lnZ, "f": -lnZ / (L * beta), "u": avg[0] / L,
           "c": beta * beta * (avg[1] - avg[0] ** 2) / L}
    if m2:
        out["m2"] = avg[2]
    return out


def _batch_exact(case, seed):
    L, nd = case["L"], case["doublings"]
    items = _batch_items(case, seed)
    Delta = float(_rng(case, seed).uniform(0.1, 1.5))
    e = torch.linalg.eigvalsh(_operator(_xxz_mpo(L, Delta)).cpu()).numpy()
    out = {k: [] for k in ROW}
    for _, _, _, kw in items:
        rows = []
        for n in range(nd + 1):
            b = kw["tau0"] * 2.0 ** n
            # rho(tau0) is the series to 4th order, doubled n times
            x = -kw["tau0"] * e
            p = (1 + x * (1 + x / 2 * (1 + x / 3 * (1 + x / 4)))) ** (2.0 ** n)
            Z = p.sum()
            e1, e2 = (p * e).sum() / Z, (p * e * e).sum() / Z
            rows.append((b, math.log(Z), -math.log(Z) / (L * b), e1 / L,
                         b * b * (e2 - e1 * e1) / L))
        for k, name in enumerate(ROW):
            out[name].append([r[k] for r in rows])
    return {k: np.array(v) for k, v in out.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B = _gemm_inputs(case, seed)
        return torch.matmul(A, B if case["nn"] else B.transpose(1, 2))
    if kind == "batch":
        return _batch_exact(case, seed)
    if case.get("prec") == "bf16x3":
        return None   # off by the noise of 16-bit operands, drawn anew by any order of the sums
    Delta, beta = _physics(case, seed)
    sites, lnc = _thermal_state(case["L"], case["D"], Delta, beta)
    L = case["L"]
    if kind == "observables":
        out = _row(sites, lnc, beta, Delta, False, False)
        E = F = torch.ones(1, 1, dtype=torch.float64, device=DEV)
        for w in sites:
            E = torch.einsum("btsc,btsd->cd", torch.einsum("ab,atsc->btsc", E, w), w)
            F = torch.einsum("btsc,bstd->cd", torch.einsum("ab,atsc->btsc", F, w), w)
        ratio = float(F[0, 0]) / float(E[0, 0])
        out["herm_defect"] = math.sqrt(max(0.0, 2.0 - 2.0 * ratio))
        out["max_bond"] = None
        return out
    if kind == "entanglement":
        S, c = [], sites[0]
        for i in range(L - 1):
            m = c.reshape(-1, c.shape[3])
            u, s, vt = torch.linalg.svd(m.cpu(), full_matrices=False)
            p = s.numpy() ** 2
            p = p[p > 0] / p.sum()
            S.append(float(-(p * np.log(p)).sum()))
            c = torch.einsum("ab,bstc->astc", (s[:, None] * vt).to(DEV), sites[i + 1])
        return S
    if kind == "settn":
        rho, H = _operator(sites) * math.exp(lnc), _operator(_xxz_mpo(L, Delta))
        term, new = rho, rho
        for k in range(1, case["order"] + 1):
            term = H @ term * (-beta / k)
            new = new + term
        Z = float(new.trace())
        e1, e2 = float((H @ new).trace()) / Z, float((H @ (H @ new)).trace()) / Z
        b = 2.0 * beta
        return {"beta": b, "lnZ": math.log(Z), "f": -math.log(Z) / (L * b), "u": e1 / L,
                "c": b * b * (e2 - e1 * e1) / L, "max_bond": None}
    out = _row(sites, lnc, 2.0 * beta, Delta, True, kind == "double")
    out["lnZ2"] = out["max_bond"] = None
    if case["prec"] != "fp64":
        del out["c"]
    if kind == "dense":
        rho = _operator(sites) * math.exp(lnc)
        out["rho"] = rho.T @ rho
    return out
