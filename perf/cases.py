"""The calls that a user of this package makes, at the sizes it is made for.

A case is one call on one problem: sigma = H.c on a tensor-product space (FP64,
FP32 or a tensor-core type), sigma on a pruned space, a bounded Davidson run, the
set-up of a space, the overlaps of CI vectors, or the string weights and
coefficient distribution of a selection step. Sizes are those of the workloads
and the serving stream in ``tbsci_inputs`` (norb 8 to 24; 50 to 40,000 strings
per spin), with the largest sigma cut in alpha strings so that a pass stays
within a second or so. Coefficients are normal deviates under string weights
that spread over about two decades per spin, as in a correlated wavefunction,
and each vector has unit norm.

Spaces of 10,000 strings and more and the tensor-core types are autotuned once
per shape, as bench.py and a user with a large space do; the context keeps the
shape for later spaces of the same size. Everything else runs untuned.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2503_10335_gb300 as tb
from tbsci_inputs import orbital_irreps, selected_strings, synth_hamiltonian, synth_hamiltonian_symmetric

_DTYPES = {"f64": (torch.float64, tb.TBSCI_F64), "f32": (torch.float32, tb.TBSCI_F32),
           "tf32": (torch.float32, tb.TBSCI_F32_TC_TF32), "bf16": (torch.float32, tb.TBSCI_F32_TC_BF16)}
_context = []
_tuned = set()


def listed():
    return [
        # the smallest full space (4,900 determinants): one launch, latency
        {"name": "sigma_fci8_f64", "call": "sigma", "norb": 8, "na": 4, "nb": 4, "la": 0, "lb": 0, "nvec": 1,
         "dtype": "f64"},
        # a small solve of the serving stream: distinct alpha and beta sets, two roots
        {"name": "sigma_sel12_f64", "call": "sigma", "norb": 12, "na": 6, "nb": 6, "la": 250, "lb": 260, "nvec": 2,
         "dtype": "f64"},
        # the 9.0M-determinant selected space with its three roots: the ordinary solve
        {"name": "sigma_sel16_f64", "call": "sigma", "norb": 16, "na": 8, "nb": 8, "la": 3000, "lb": 3000, "nvec": 3,
         "dtype": "f64"},
        # the same in the low-precision phase of a mixed solve
        {"name": "sigma_sel16_f32", "call": "sigma", "norb": 16, "na": 8, "nb": 8, "la": 3000, "lb": 3000, "nvec": 3,
         "dtype": "f32"},
        # the full norb-16 space (165.6M determinants) in the two tensor-core types
        {"name": "sigma_fci16_tf32", "call": "sigma", "norb": 16, "na": 8, "nb": 8, "la": 0, "lb": 0, "nvec": 1,
         "dtype": "tf32"},
        {"name": "sigma_fci16_bf16", "call": "sigma", "norb": 16, "na": 8, "nb": 8, "la": 0, "lb": 0, "nvec": 1,
         "dtype": "bf16"},
        # norb 24 with the 40,000 beta strings of the large selected space: rows longer than shared memory
        {"name": "sigma_sel24_f64", "call": "sigma", "norb": 24, "na": 12, "nb": 12, "la": 10000, "lb": 40000,
         "nvec": 1, "dtype": "f64"},
        {"name": "sigma_sel24_f32", "call": "sigma", "norb": 24, "na": 12, "nb": 12, "la": 20000, "lb": 40000,
         "nvec": 1, "dtype": "f32"},
        # one irrep of a symmetric full space (norb 14, D2h): sigma of a blocked solve
        {"name": "sigma_sym14_f64", "call": "pruned", "norb": 14, "na": 7, "nb": 7, "la": 0, "lb": 0, "nvec": 1,
         "dtype": "f64", "cap": -1},
        # a whole FP64 Davidson call, three roots, bounded at 20 iterations (two restarts)
        {"name": "davidson_sel16", "call": "davidson", "norb": 16, "na": 8, "nb": 8, "la": 1200, "lb": 1100,
         "nroots": 3, "iterations": 20},
        # set-up of a space: strings, link tables, Hamiltonian values, schedules, then its diagonal
        {"name": "setup_sel24", "call": "setup", "norb": 24, "na": 12, "nb": 12, "la": 4000, "lb": 5000},
        # string weights and coefficient distribution of a converged vector: a step of the selection loop
        {"name": "select_sel16", "call": "select", "norb": 16, "na": 8, "nb": 8, "la": 3000, "lb": 3000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["sigma", "sigma", "sigma", "sigma", "tc", "long", "pruned", "davidson", "setup", "select"])
    if call == "long":  # rows of 20,000 to 40,000 beta strings
        n = rng.choice([20, 22, 24])
        ne = n // 2 - rng.choice([0, 0, 1])
        return {"call": "sigma", "norb": n, "na": ne, "nb": ne, "la": _log(rng, 1500, 9000),
                "lb": _log(rng, 20000, 40000), "nvec": 1, "dtype": rng.choice(["f64", "f32"])}
    if call == "tc":
        n = rng.choice([10, 12, 13, 14, 15, 16])
        na, nb = n // 2, n // 2 - rng.choice([0, 1])
        top = math.comb(n, nb)
        full = rng.random() < 0.5 and top <= 6435
        return {"call": "sigma", "norb": n, "na": na, "nb": nb, "la": 0 if full else min(math.comb(n, na), _log(rng, 200, 6000)),
                "lb": 0 if full else min(top, _log(rng, 200, 6000)), "nvec": rng.choice([1, 2, 3]),
                "dtype": rng.choice(["tf32", "bf16"])}
    n = rng.choice([8, 10, 11, 12, 14, 15, 16])
    na = n // 2
    nb = na - rng.choice([0, 0, 1])
    la = min(math.comb(n, na), _log(rng, 50, 3000))
    lb = min(math.comb(n, nb), _log(rng, 50, 3000))
    case = {"call": call, "norb": n, "na": na, "nb": nb, "la": la, "lb": lb}
    if call == "sigma":
        case.update(nvec=rng.randint(1, 5), dtype=rng.choice(["f64", "f64", "f32"]))
    elif call == "pruned":
        case.update(nvec=rng.randint(1, 3), dtype=rng.choice(["f64", "f64", "f32"]), cap=rng.choice([-1, 4, 5]))
    elif call == "davidson":
        case.update(la=min(la, 1200), lb=min(lb, 1200), nroots=rng.randint(1, 3), iterations=rng.randint(10, 24))
    return case


def _ctx():
    if not _context:
        _context.append(tb.Context(0))
    return _context[0]


def _inputs(case, seed):
    """Integrals and string selections of a case (None: the full string space)."""
    n = case["norb"]
    irreps = None
    if case["call"] == "pruned" and case["cap"] < 0:
        irreps = orbital_irreps(n, 100 + n, 8)  # the molecule's point group: the same for every geometry
        h, eri, _ = synth_hamiltonian_symmetric(n, seed + 1, irreps)
    else:
        h, eri, _ = synth_hamiltonian(n, seed + 1)
    # a pruned space keeps its determinants from one geometry to the next, so its vectors have one length
    pick = n if case["call"] == "pruned" else seed
    alpha = selected_strings(n, case["na"], case["la"], pick + 2) if case["la"] else None
    beta = selected_strings(n, case["nb"], case["lb"], pick + 3) if case["lb"] else None
    return h, eri, 0.5, alpha, beta, irreps


def _sorted_strings(n, ne, sel):
    if sel is not None:
        return np.sort(sel.astype(np.int64))
    s = np.arange(1 << n, dtype=np.int64)
    return s[np.bitwise_count(s) == ne]


def _space(case, seed):
    h, eri, ecore, alpha, beta, irreps = _inputs(case, seed)
    return tb.Space(_ctx(), case["norb"], case["na"], case["nb"], h, eri, ecore, alpha=alpha, beta=beta), irreps


def _cap_rows(case, alpha, beta):
    """Per alpha string the beta strings within `cap` excitations in all of the aufbau determinant (CSR)."""
    la = np.bitwise_count(alpha >> case["na"]).astype(np.int64)
    lb = np.bitwise_count(beta >> case["nb"]).astype(np.int64)
    keep = la[:, None] + lb[None, :] <= case["cap"]
    off = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    return off, np.nonzero(keep)[1].astype(np.int32)


def _irrep_mask(case, alpha, beta, irreps):
    def of(strings):
        g = np.zeros(len(strings), dtype=np.int64)
        for i in range(case["norb"]):
            g ^= np.where((strings >> i) & 1, int(irreps[i]), 0)
        return g
    return of(alpha)[:, None] == of(beta)[None, :]


def _vectors(nvec, la, lb, seed, dtype):
    g = torch.Generator(device="cuda").manual_seed(seed + 4)
    c = torch.randn((nvec, la, lb), generator=g, device="cuda", dtype=dtype)
    for axis, length in ((1, la), (2, lb)):
        w = torch.pow(10.0, -2.0 * torch.rand(length, generator=g, device="cuda", dtype=torch.float32) ** 2).to(dtype)
        c *= w[None, :, None] if axis == 1 else w[None, None, :]
    for v in range(nvec):
        c[v] /= torch.linalg.vector_norm(c[v])
    return c


def prepare(case, seed):
    seed = int(seed) % (1 << 30)
    call = case["call"]
    if call == "setup":
        return {"case": case, "inputs": _inputs(case, seed)}
    sp, irreps = _space(case, seed)
    state = {"case": case, "space": sp}
    if call == "davidson":
        return state
    dt, kind = _DTYPES[case.get("dtype", "f64")]
    c = _vectors(case.get("nvec", 1), sp.la, sp.lb, seed, dt)
    if call == "pruned":
        alpha, beta = (s.astype(np.int64) for s in sp.strings())
        if case["cap"] < 0:
            pr = sp.symmetry_block(irreps, 0)
            keep = torch.from_numpy(_irrep_mask(case, alpha, beta, irreps)).cuda()
            c = c[:, keep]
        else:
            off, cols = _cap_rows(case, alpha, beta)
            pr = sp.prune(off, cols)
            rows = torch.from_numpy(np.repeat(np.arange(sp.la), np.diff(off))).cuda()
            c = c[:, rows, torch.from_numpy(cols).cuda().long()]
        state.update(pruned=pr, c=c.contiguous())
        return state
    if call == "sigma" and (max(sp.la, sp.lb) >= 10000 or case["dtype"] in ("tf32", "bf16")):
        key = (case["dtype"], case["norb"], sp.la, sp.lb)
        if key not in _tuned:
            out = torch.empty_like(c)
            tb.tbsci_sigma_autotune(_ctx().handle, sp.ham, sp.ta, sp.tb, c, out, c.shape[0], kind)
            _tuned.add(key)
    state["c"] = c
    if call == "select":
        state["c_hf"] = float(c.abs().max())
    return state


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "setup":
        h, eri, ecore, alpha, beta, _ = state["inputs"]
        sp = tb.Space(_ctx(), case["norb"], case["na"], case["nb"], h, eri, ecore, alpha=alpha, beta=beta)
        a, b = sp.strings()
        counts = sp.counts()
        out = {"alpha": a.view(np.int64), "beta": b.view(np.int64), "nnz_aa": counts["nnz_aa"],
               "nnz_bb": counts["nnz_bb"], "nnz_ab": counts["nnz_ab"], "diagonal": sp.diagonal()}
        sp.close()
        return out
    sp = state["space"]
    if call == "davidson":
        e, _, v = sp.davidson(case["nroots"], want_vectors=True, max_iter=case["iterations"], tol_energy=1e-15,
                              tol_residual=1e-14, check=False)
        return {"energies": e, "vectors": v}
    c = state["c"]
    if call == "pruned":
        return state["pruned"].sigma(c)
    if call == "select":
        wa, wb = sp.string_weights(c)
        _, counts = sp.coefficient_histogram(c, state["c_hf"])
        return {"alpha_weights": wa, "beta_weights": wb, "counts": counts}
    return sp.sigma(c, dtype=_DTYPES[case["dtype"]][1])


def work(case):
    """Two flops per non-zero of H and vector; c read once and sigma written once. For the other
    calls the vector work or the tables that the call returns or fills."""
    call = case["call"]
    la = case["la"] or math.comb(case["norb"], case["na"])
    lb = case["lb"] or math.comb(case["norb"], case["nb"])
    if call == "select":
        return {"bytes": 8.0 * la * lb, "flops": 2.0 * la * lb}
    sp, irreps = _space(case, 7)
    k = sp.counts()
    if call == "setup":
        links = k["nnz_aa"] // max(1, sp.lb) + k["nnz_bb"] // max(1, sp.la)
        sp.close()
        return {"bytes": 16.0 * links + 8.0 * la * lb, "flops": 2.0 * la * lb * case["na"]}
    nnz, ndet = float(k["nnz"]), float(k["ndet"])
    if call == "davidson":
        sp.close()
        steps, n = case["iterations"], case["nroots"]
        # per iteration: nroots sigma, the basis against the new vectors (Rayleigh columns,
        # Gram-Schmidt) and twice into the Ritz vectors and images, at a half-full basis
        basis = 4 * n
        return {"bytes": steps * ndet * 8.0 * (6 * basis + 8 * n), "flops": steps * n * (2.0 * nnz + 10.0 * basis * ndet)}
    size = 4 if case["dtype"] != "f64" else 8
    if call == "pruned":
        alpha, beta = (s.astype(np.int64) for s in sp.strings())
        kept = int(_irrep_mask(case, alpha, beta, irreps).sum()) if case["cap"] < 0 else int(_cap_rows(case, alpha, beta)[0][-1])
        # the couplings that stay inside the space: its share of the TPB space's
        nnz, ndet = nnz * (kept / ndet) ** 2, float(kept)
    sp.close()
    return {"bytes": 2.0 * case["nvec"] * ndet * size, "flops": 2.0 * case["nvec"] * nnz}


# ---------------------------------------------------------------- 64-bit values

def _parity(strings, x, y):
    """(-1)^(occupied orbitals strictly between x and y)."""
    lo, hi = np.minimum(x, y), np.maximum(x, y)
    between = ((np.int64(1) << hi) - 1) & ~((np.int64(1) << (lo + 1)) - 1)
    return 1.0 - 2.0 * (np.bitwise_count(strings & between) & 1)


def _lowbit(x):
    return np.bitwise_count((x & -x) - 1).astype(np.int64)


def _one_spin(n, strings, h, eri):
    """Dense one-spin string Hamiltonian (diagonal included) by the Slater-Condon rules."""
    m = len(strings)
    occ = ((strings[:, None] >> np.arange(n)) & 1).astype(np.float64)
    coul = np.einsum("iijj->ij", eri)
    exch = np.einsum("ijji->ij", eri)
    H = np.zeros((m, m))
    H[np.arange(m), np.arange(m)] = occ @ np.diag(h) + 0.5 * np.einsum("ki,ij,kj->k", occ, coul - exch, occ)
    singles = [[] for _ in range(3)]
    mean = np.einsum("pqkk->pqk", eri) - np.einsum("pkkq->pqk", eri)
    for lo in range(0, m, 1024):
        part = strings[lo:lo + 1024]
        diff = part[:, None] ^ strings[None, :]
        cnt = np.bitwise_count(diff)
        i, j = np.nonzero(cnt == 2)
        si, sj = part[i], strings[j]
        p, q = _lowbit(si & ~sj), _lowbit(sj & ~si)  # <si| a+_p a_q |sj>
        sg = _parity(sj, p, q)
        H[lo + i, j] = sg * (h[p, q] + np.einsum("kx,kx->k", mean[p, q], occ[j]))
        for dst, v in zip(singles, ((lo + i), j, sg * (1 + np.minimum(p, q) * n + np.maximum(p, q)))):
            dst.append(v)
        i, j = np.nonzero(cnt == 4)
        si, sj = part[i], strings[j]
        new, old = si & ~sj, sj & ~si
        p, q = _lowbit(new), _lowbit(old)
        r, s = _lowbit(new & (new - 1)), _lowbit(old & (old - 1))
        mid = sj ^ (np.int64(1) << q) ^ (np.int64(1) << p)
        sg = _parity(sj, p, q) * _parity(mid, r, s)
        H[lo + i, j] = sg * (eri[p, q, r, s] - eri[p, s, r, q])
    return H, tuple(np.concatenate(x) for x in singles), occ


def _sigma_exact(n, alpha, beta, h, eri, ecore, c):
    """sigma of c [nvec, la, lb] (FP64, on the GPU): H_a x 1 + 1 x H_b + sum (pq|rs) E^a_pq E^b_rs."""
    Ha, (ia, ja, ka), occ_a = _one_spin(n, alpha, h, eri)
    Hb, (ib, jb, kb), occ_b = _one_spin(n, beta, h, eri)
    dev = "cuda"
    cu = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)  # noqa: E731
    out = ecore * c + cu(Ha) @ c + c @ cu(Hb).T
    del Ha, Hb
    Ib, Jb, Kb = cu(ib), cu(jb), cu(kb)
    pair_b, sign_b = Kb.abs().long() - 1, Kb.sign()
    eri2 = cu(eri.reshape(n * n, n * n))
    occb = cu(occ_b)
    lb = len(beta)
    pair_a, sign_a = np.abs(ka).astype(np.int64) - 1, np.sign(ka)

    def beta_side(row):  # sum_rs (pq|rs) E^b_rs as a sparse matrix, its diagonal apart
        w = torch.sparse_coo_tensor(torch.stack([Ib, Jb]), sign_b * row[pair_b], (lb, lb), check_invariants=False)
        return w.to_sparse_csr(), occb @ row[torch.arange(n, device=dev) * (n + 1)]

    for p in range(n):
        for q in range(p, n):
            if p == q:
                rows = src = np.nonzero(occ_a[:, p])[0]
                sg = np.ones(len(rows))
            else:
                at = np.nonzero(pair_a == p * n + q)[0]
                rows, src, sg = ia[at], ja[at], sign_a[at]
            if not len(rows):
                continue
            w, d = beta_side(eri2[p * n + q])
            for v in range(c.shape[0]):
                x = c[v][cu(src)] * cu(sg)[:, None]
                y = x * d
                if len(ib):
                    y += torch.sparse.mm(w, x.T.contiguous()).T
                out[v].index_add_(0, cu(rows), y)
    return out


def exact(case, seed):
    seed = int(seed) % (1 << 30)
    call = case["call"]
    if call == "davidson":
        return None
    n = case["norb"]
    h, eri, ecore, alpha, beta, irreps = _inputs(case, seed)
    alpha, beta = _sorted_strings(n, case["na"], alpha), _sorted_strings(n, case["nb"], beta)
    la, lb = len(alpha), len(beta)
    if call == "select":
        c = _vectors(1, la, lb, seed, torch.float64)[0]
        sq = c * c
        return {"alpha_weights": sq.sum(1) / sq.sum(), "beta_weights": sq.sum(0) / sq.sum(), "counts": None}
    if call == "setup":
        occ_a = ((alpha[:, None] >> np.arange(n)) & 1).astype(np.float64)
        occ_b = ((beta[:, None] >> np.arange(n)) & 1).astype(np.float64)
        coul, exch = np.einsum("iijj->ij", eri), np.einsum("ijji->ij", eri)
        ea, eb = (o @ np.diag(h) + 0.5 * np.einsum("ki,ij,kj->k", o, coul - exch, o) for o in (occ_a, occ_b))
        d = ecore + ea[:, None] + eb[None, :] + occ_a @ coul @ occ_b.T
        return {"alpha": None, "beta": None, "nnz_aa": None, "nnz_bb": None, "nnz_ab": None, "diagonal": d.reshape(-1)}
    if la * lb > 50_000_000:
        return None
    c = _vectors(case["nvec"], la, lb, seed, _DTYPES[case["dtype"]][0]).double()
    if call == "sigma":
        return _sigma_exact(n, alpha, beta, h, eri, ecore, c)
    if case["cap"] < 0:
        keep = torch.from_numpy(_irrep_mask(case, alpha, beta, irreps)).cuda()
    else:
        off, cols = _cap_rows(case, alpha, beta)
        keep = torch.zeros((la, lb), dtype=torch.bool, device="cuda")
        keep[torch.from_numpy(np.repeat(np.arange(la), np.diff(off))).cuda(), torch.from_numpy(cols).cuda().long()] = True
    return _sigma_exact(n, alpha, beta, h, eri, ecore, c * keep)[:, keep]
