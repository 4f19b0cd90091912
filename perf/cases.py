"""What this framework is used for, as cases that can be timed and compared.

A case is one call (or one step of a loop) of a program that evolves matrix product states with
this library, through its public entry points: the contraction engines on device buffers, the
allocation-free correlator, and whole calls on a simulation handle (quench from a product state,
one step of a saturated state with its observables, a batch of simulations, the observables of a
large state).  Outputs of a handle are what does not depend on the gauge of the Schmidt vectors:
densities, currents, every bond's spectrum (descending), the bond dimensions and, in the
particle-number-blocked form, every bond's charges (ascending).  The site tensors themselves are
fixed only up to a phase per Schmidt vector and a rotation among equal singular values, so they
are compared through these.

The calls on a handle run in FP64 or in exact-digit arithmetic.  The mixed path's own engine, split
3xTF32 with FP32 accumulation, is here as single products: a whole mixed step turns a change of one
FP64 rounding anywhere into differences of FP32 size (1e-6, measured), and its other kernels are those
of the exact-digit steps.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import workloads
from paper_2401_05301_gb300 import SuperSiteTEBD, TEBD, load
from paper_2401_05301_gb300.binding import batch_step


def listed():
    return [
        # One bond's correlator inside a latency-critical loop: the smallest call of the library.
        {"name": "correlator_chi24_d4", "kind": "correlator", "chl": 24, "chm": 24, "chr": 24, "d": 4},
        # theta~ = X B_{i+2} of an interior triple at chi = 256, d = 4, on each contraction engine; the
        # FP64 one as the rebuild B_i = C V1^+ (a conjugate-transposed operand), with ragged sizes.
        {"name": "zgemm_fp64_rebuild_ragged", "kind": "zgemm", "precision": 0, "opB": 1, "M": 1000, "N": 250, "K": 3990},
        {"name": "zgemm_tf32_theta", "kind": "zgemm", "precision": 1, "opB": 0, "M": 4096, "N": 1024, "K": 256},
        {"name": "zgemm_exact_theta", "kind": "zgemm", "precision": 2, "opB": 0, "M": 4096, "N": 1024, "K": 256},
        # The first steps of an eight-site quench against which small-chain studies are checked: bonds
        # of 1 to 30, so a step is bound by launches and by the host's decisions.
        {"name": "quench_L8_d4_fp64", "kind": "quench", "form": "dense", "L": 8, "n_max": 3, "chi": 256,
         "steps": 4, "dt": 0.01, "precision": 0, "w_cut": 0.0},
        # The paper's kind of run (d = 5, chi_max = 40, cuts of 1e-12, dt = 0.05 pi / 2) on a shorter
        # chain in its particle-number-symmetric form: many small charge blocks.
        {"name": "quench_L41_d5_chi40_u1_fp64", "kind": "quench", "form": "u1", "L": 41, "n_max": 4, "chi": 40,
         "steps": 4, "dt": 0.025 * math.pi, "precision": 0, "w_cut": 1e-12},
        # The paper's super sites (d_e = 16 here) on the same kind of run.
        {"name": "quench_L20_d4_chi32_supersite_exact", "kind": "quench", "form": "supersite", "L": 20, "n_max": 3,
         "chi": 32, "steps": 2, "dt": 0.02, "precision": 2, "w_cut": 1e-12},
        # One step and its observables of a saturated chain, dense form, FP64 on the CUDA cores, odd chi.
        {"name": "step_L12_d4_chi61_fp64", "kind": "step", "form": "dense", "L": 12, "n_max": 3, "chi": 61,
         "precision": 0, "graph": 0},
        # The same at chi = 256 (the truncating L = 32 workload's bonds) with exact-digit products.
        {"name": "step_L14_d4_chi256_exact", "kind": "step", "form": "dense", "L": 14, "n_max": 3, "chi": 256,
         "precision": 2, "graph": 0},
        # The headline's physics and local sizes (d = 5, chi_max = 1024, particle-number blocks) on 24
        # sites, FP64-accurate on the tensor cores.
        {"name": "step_L24_d5_chi1024_u1_exact", "kind": "step", "form": "u1", "L": 24, "n_max": 4, "chi": 1024,
         "precision": 2, "graph": 0},
        # A parameter scan: six simulations of the 48-simulation batch's kind stepped together.
        {"name": "batch6_d4_u1_exact", "kind": "batch", "n": 6, "L": 16, "n_max": 3, "chi": 128, "precision": 2},
        # Densities and currents of a large state, the only thing a monitoring program asks of it.
        {"name": "measure_L20_d4_chi384", "kind": "measure", "form": "dense", "L": 20, "n_max": 3, "chi": 384,
         "precision": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["correlator", "zgemm", "zgemm", "quench", "quench", "step", "step", "batch", "measure"])
    if kind == "correlator":
        return {"kind": kind, "chl": _log_int(rng, 1, 64), "chm": _log_int(rng, 2, 64), "chr": _log_int(rng, 1, 64),
                "d": rng.randint(2, 8)}
    if kind == "zgemm":
        precision = rng.choice([0, 1, 2])
        k = _log_int(rng, 16, 1500)
        return {"kind": kind, "precision": precision, "opB": rng.choice([0, 1]), "M": _log_int(rng, 32, 4096),
                "N": _log_int(rng, 16, 1024), "K": k if precision == 0 else min(k, 1024)}
    if kind == "quench":
        form = rng.choice(["dense", "u1", "supersite"])
        n_max = rng.randint(1, 3 if form == "supersite" else 4)
        return {"kind": kind, "form": form, "L": rng.randint(6, 14 if form == "dense" else 20 if form == "supersite" else 41),
                "n_max": n_max, "chi": rng.randint(8, 32 if form == "supersite" else 64), "steps": rng.randint(1, 2),
                "dt": round(rng.uniform(0.005, 0.05), 4), "precision": rng.choice([0, 2]),
                "w_cut": rng.choice([0.0, 1e-12, 1e-10])}
    if kind == "step":
        form = rng.choice(["dense", "u1"])
        if form == "dense":
            return {"kind": kind, "form": form, "L": rng.randint(8, 14), "n_max": rng.randint(2, 4),
                    "chi": _log_int(rng, 24, 160), "precision": rng.choice([0, 2]), "graph": rng.choice([0, 1])}
        chi = _log_int(rng, 48, 768)
        return {"kind": kind, "form": form, "L": rng.randint(10, 24), "n_max": rng.randint(2, 4), "chi": chi,
                "precision": rng.choice([0, 2]) if chi < 200 else 2, "graph": 0}
    if kind == "batch":
        return {"kind": kind, "n": rng.randint(2, 6), "L": rng.randint(10, 16), "n_max": rng.randint(2, 3),
                "chi": _log_int(rng, 24, 128), "precision": rng.choice([0, 2])}
    return {"kind": kind, "form": rng.choice(["dense", "u1"]), "L": rng.randint(10, 20), "n_max": rng.randint(2, 4),
            "chi": _log_int(rng, 32, 384), "precision": rng.choice([0, 2])}


# ---- inputs -------------------------------------------------------------------------


def _rng(seed, salt):
    return np.random.Generator(np.random.PCG64([int(seed), salt]))


def _physics(seed, salt=0):
    """U, J_NNN and K in the ranges of the 48-simulation batch."""
    r = _rng(seed, 100 + salt)
    return float(r.uniform(2.0, 6.0)), float(r.uniform(0.0, 0.15)), float(r.uniform(0.0, 0.01))


def _args(case, seed, salt=0):
    U, jn, K = _physics(seed, salt)
    return dict(L=case["L"], n_max=case["n_max"], chi_max=case["chi"], U=U, J=1.0, Jnnn=jn, K=K,
                jc=0.5 * (case["L"] + 1), dt=case.get("dt", 0.005))


def _occupation(L):
    """The charge-density wave |1, 0, 1, 0, ...>."""
    return (np.arange(L) + 1) % 2


def _dense_state(L, d, chi_max, seed):
    """A saturated right-canonical state with a geometric spectrum p_i ~ exp(-8 i / chi)."""
    r = _rng(seed, 1)
    chi = [min(chi_max, d ** min(k, L - k, 16)) for k in range(L + 1)]
    B = []
    for k in range(L):
        a, b = chi[k], chi[k + 1]
        x = r.standard_normal((d * b, a)) + 1j * r.standard_normal((d * b, a))
        B.append(np.ascontiguousarray(np.linalg.qr(x)[0].conj().T).reshape(a, d, b))
    lam = []
    for n in chi:
        p = np.exp(-8.0 * np.arange(n) / n)
        lam.append(np.sqrt(p / p.sum()))
    return B, lam


def _cplx(r, shape):
    return torch.from_numpy(r.standard_normal(shape) + 1j * r.standard_normal(shape)).cuda()


def _correlator_inputs(case, seed):
    r = _rng(seed, 2)
    chl, chm, chr_, d = case["chl"], case["chm"], case["chr"], case["d"]
    Bl, Br = _cplx(r, (chl, d, chm)) / math.sqrt(d * chm), _cplx(r, (chm, d, chr_)) / math.sqrt(d * chr_)
    lam = torch.from_numpy(r.uniform(0.1, 1.0, chl)).cuda()
    return Bl, lam / lam.norm(), Br


def _zgemm_inputs(case, seed):
    r = _rng(seed, 3)
    b = (case["N"], case["K"]) if case["opB"] else (case["K"], case["N"])
    # rows fall off like the rows lam (.) C of theta' do
    rows = torch.exp(torch.linspace(0.0, -6.0, case["M"], dtype=torch.float64, device="cuda"))
    return _cplx(r, (case["M"], case["K"])) * rows[:, None], _cplx(r, b)


def _handle(case, seed, salt=0):
    form, opts = case.get("form", "u1"), dict(precision=case["precision"])
    if "w_cut" in case:
        opts["w_cut"] = case["w_cut"]
    if form == "supersite":
        return SuperSiteTEBD(**_args(case, seed, salt), **opts)
    return TEBD(**_args(case, seed, salt), **opts, u1=True if form == "u1" else None)


def _saturated(case, seed, salt=0):
    g = _handle(case, seed, salt)
    L, d = case["L"], case["n_max"] + 1
    if case.get("form", "u1") == "u1":
        B, lam, q = workloads.synthetic_state_u1(L, d, case["chi"], L // 2, seed=seed + 1000 * salt)
        g.set_state(B, lam)
        g.set_charges(q)
    else:
        g.set_state(*_dense_state(L, d, case["chi"], seed))
        if case.get("graph"):
            g.set_option("graph", 1)
    return g


def prepare(case, seed):
    kind = case["kind"]
    if kind == "correlator":
        return {"case": case, "in": _correlator_inputs(case, seed)}
    if kind == "zgemm":
        return {"case": case, "in": _zgemm_inputs(case, seed)}
    if kind == "quench":
        return {"case": case, "g": _handle(case, seed), "occ": _occupation(case["L"])}
    if kind == "batch":
        sims = [_saturated(dict(case, L=max(8, case["L"] - i), chi=max(8, case["chi"] >> (i % 2))), seed, i)
                for i in range(case["n"])]
        return {"case": case, "sims": sims}
    return {"case": case, "g": _saturated(case, seed)}


# ---- one pass -----------------------------------------------------------------------


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _table(rows, width, fill):
    """Rows of different lengths in one array, as a program that records a run keeps them."""
    out = np.full((len(rows), width), fill)
    for k, x in enumerate(rows):
        out[k, :len(x)] = x
    return out


def _read(g, case, blocked=False):
    n, cur = g.measure()
    lam = [np.sort(g.get_lambda(k))[::-1] for k in range(g.L + 1)]
    out = {"n": n, "cur": cur, "lam": _table(lam, case["chi"], 0.0), "chi": g.bond_dims()}
    if blocked:
        out["q"] = _table([g.get_charges(k) for k in range(g.L + 1)], case["chi"], -1)
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "correlator":
        Bl, lam, Br = state["in"]
        out = torch.empty(1, dtype=torch.complex128, device="cuda")
        st = load().tebd_bond_correlator_noalloc(
            _ptr(Bl), _ptr(lam), _ptr(Br), case["chl"], case["chm"], case["chr"], case["d"], _ptr(out),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st:
            raise RuntimeError(f"tebd_bond_correlator_noalloc: {st}")
        return out
    if kind == "zgemm":
        A, B = state["in"]
        out = torch.empty(case["M"], case["N"], dtype=torch.complex128, device="cuda")
        st = load().tebd_zgemm(case["precision"], case["opB"], case["M"], case["N"], case["K"], 1.0, _ptr(A),
                               A.shape[1], _ptr(B), B.shape[1], _ptr(out), case["N"],
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st:
            raise RuntimeError(f"tebd_zgemm: {st}")
        return out
    if kind == "batch":
        batch_step(state["sims"], 1)
        return [_read(g, case, True) for g in state["sims"]]
    g = state["g"]
    if kind == "measure":
        n, cur = g.measure()
        return {"n": n, "cur": cur}
    if kind == "quench":
        g.init_product(state["occ"])
        g.step(case["steps"])
    else:
        g.step(1)
    return _read(g, case, case["form"] == "u1")


# ---- what a pass cannot do without ------------------------------------------------------


def _bonds(case):
    """Bond dimensions of the case's states: saturated, or (a quench's few steps) at most those."""
    ss = case.get("form") == "supersite"
    L, d = ((case["L"] + 1) // 2, (case["n_max"] + 1) ** 2) if ss else (case["L"], case["n_max"] + 1)
    return L, d, [min(case["chi"], d ** min(k, L - k, 16)) for k in range(L + 1)]


def _svd_flops(m, n, k):
    """Real operations of a truncated SVD of a complex m x n matrix: the triangular-reduction count of
    the smaller side plus the k kept vectors of each side."""
    s, b = min(m, n), max(m, n)
    return 4.0 * s * s * b + 16.0 / 3.0 * s ** 3 + 8.0 * k * s * (s + b)


def _step_work(case):
    L, d, chi = _bonds(case)
    flops = nbytes = 0.0
    if case.get("form") == "supersite":
        for first in (0, 1, 0):
            for i in range(first, L - 1, 2):
                a, b, c = chi[i], chi[i + 1], chi[i + 2]
                flops += 8.0 * a * d * d * c * b + 8.0 * a * c * d ** 4 + _svd_flops(a * d, d * c, b) + 8.0 * a * d * b * d * c
                nbytes += 32.0 * (a * d * b + b * d * c)
        return flops, nbytes
    for first in (0, 1, 2, 1, 0):
        for i in range(first, L - 2, 3):
            a, b, c, e = chi[i:i + 4]
            flops += 8.0 * a * d * d * c * b + 8.0 * a * d ** 3 * e * c + 8.0 * a * e * d ** 6
            flops += _svd_flops(a * d, d * d * e, b) + 8.0 * a * d * b * d * d * e
            flops += _svd_flops(b * d, d * e, c) + 8.0 * b * d * c * d * e
            nbytes += 32.0 * (a * d * b + b * d * c + c * d * e)
    if case.get("form", "u1") == "u1":  # what the charge blocks leave of it (counted: 1/110 to 1/245, 1/6.5 to 1/8.5)
        flops, nbytes = flops / 120.0, nbytes / 7.0
    return flops, nbytes


def work(case):
    kind = case["kind"]
    if kind == "correlator":
        a, m, c, d = case["chl"], case["chm"], case["chr"], case["d"]
        return {"bytes": 16.0 * d * m * (a + c) + 8.0 * a + 16.0, "flops": 8.0 * m * m * d * (a + c) + 8.0 * m * m}
    if kind == "zgemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 16.0 * (M * K + K * N + M * N), "flops": 8.0 * M * N * K}
    if kind == "measure":
        L, d, chi = _bonds(case)
        return {"bytes": sum(16.0 * chi[k] * d * chi[k + 1] for k in range(L)),
                "flops": sum(8.0 * d * chi[k + 1] ** 2 * (chi[k] + chi[k + 2]) for k in range(L - 1))}
    if kind == "batch":
        parts = [_step_work(dict(case, L=max(8, case["L"] - i), chi=max(8, case["chi"] >> (i % 2)))) for i in range(case["n"])]
        return {"bytes": sum(p[1] for p in parts), "flops": sum(p[0] for p in parts)}
    flops, nbytes = _step_work(case)
    if kind == "quench":  # its bonds grow from 1: a small part of the saturated step's work
        flops, nbytes = 0.1 * flops * case["steps"], 0.1 * nbytes * case["steps"]
    return {"bytes": nbytes, "flops": flops}


# ---- plain 64-bit values -----------------------------------------------------------------


def _local_ops(d):
    b = np.diag(np.sqrt(np.arange(1.0, d)), 1)
    return b, np.diag(np.arange(float(d)))


def _embed(ops, d, n):
    """Product of one-site operators {position: matrix} on n sites."""
    m = np.eye(1)
    for j in range(n):
        m = np.kron(m, ops.get(j, np.eye(d)))
    return m


def _window(sites, d, onsite, bond, nnn, a):
    """Bose-Hubbard terms on consecutive sites (1-based list), each with its share."""
    b, num = _local_ops(d)
    n = len(sites)
    h = np.zeros((d ** n, d ** n))
    for i, j in enumerate(sites):
        loc = 0.5 * a["U"] * num @ (num - np.eye(d)) + 0.5 * a["K"] * (j - a["jc"]) ** 2 * num
        h += _embed({i: loc}, d, n) * onsite(j)
        for dist, amp, share in ((1, a["J"], bond), (2, a["Jnnn"], nnn)):
            if i + dist < n:
                hop = _embed({i: b.T, i + dist: b}, d, n)
                h -= amp * share(j) * (hop + hop.T)
    return h


def _expm(h, tau):
    w, v = np.linalg.eigh(h)
    return (v * np.exp(-1j * tau * w)) @ v.T


def _cut(M, chi_max, w_cut, eps=1e-12):
    _, s, V = np.linalg.svd(M, full_matrices=False)
    p = s * s / np.sum(s * s)
    tail = np.append(np.cumsum(p[::-1])[::-1][1:], 0.0)
    k = max(1, min(chi_max, int(np.argmax(tail <= w_cut)) + 1, int(np.count_nonzero(p > eps))))
    norm = math.sqrt(np.sum(s[:k] ** 2))
    return s[:k] / norm, V[:k], norm


def _evolve(case, a, B, lam, steps):
    """Plain TEBD: `steps` second-order steps in B form, three-site gates or super sites."""
    ss, d, chi_max, w_cut, dt = case.get("form") == "supersite", case["n_max"] + 1, case["chi"], case.get("w_cut", 0.0), a["dt"]
    L, gates = len(B), {}

    def gate(i, tau):
        if (i, tau) not in gates:
            if ss:  # super bond (i, i+1): its own hops whole, what lies inside a super site shared
                share = lambda k: 1.0 if L == 2 else 1.0 / ((k > 0) + (k < L - 1))  # noqa: E731
                sup = lambda j: (j - 1) // 2  # noqa: E731
                h = _window([2 * i + 1, 2 * i + 2, 2 * i + 3, 2 * i + 4], d, lambda j: share(sup(j)),
                            lambda j: share(sup(j)) if j % 2 else 1.0, lambda j: 1.0, a)
            else:
                cover = lambda lo, hi: 1.0 / sum(1 for t in range(1, L - 1) if t <= lo and hi <= t + 2)  # noqa: E731
                h = _window([i + 1, i + 2, i + 3], d, lambda j: cover(j, j), lambda j: cover(j, j + 1), lambda j: 1.0, a)
            gates[i, tau] = _expm(h, tau)
        return gates[i, tau]

    def two(i, tau):
        x = np.tensordot(B[i], B[i + 1], (2, 0))
        l, p, _, r = x.shape
        C = np.einsum("ps,asb->apb", gate(i, tau), x.reshape(l, p * p, r)).reshape(l * p, p * r)
        lam[i + 1], V, n = _cut(np.repeat(lam[i], p)[:, None] * C, chi_max, w_cut)
        B[i], B[i + 1] = (C @ V.conj().T).reshape(l, p, -1) / n, V.reshape(-1, p, r)

    def three(i, tau):
        x = np.tensordot(np.tensordot(B[i], B[i + 1], (2, 0)), B[i + 2], (3, 0))
        l, r = x.shape[0], x.shape[-1]
        C = np.einsum("ps,asb->apb", gate(i, tau), x.reshape(l, d ** 3, r)).reshape(l * d, d * d * r)
        s, V, n = _cut(np.repeat(lam[i], d)[:, None] * C, chi_max, w_cut)
        B[i], lam[i + 1] = (C @ V.conj().T).reshape(l, d, -1) / n, s
        R = V.reshape(-1, d * r)
        lam[i + 2], V2, n2 = _cut(np.repeat(s, d)[:, None] * R, chi_max, w_cut)
        B[i + 1], B[i + 2] = (R @ V2.conj().T).reshape(len(s), d, -1) / n2, V2.reshape(-1, d, r)

    layers = ((0, 0.5), (1, 1.0), (0, 0.5)) if ss else ((0, 0.5), (1, 0.5), (2, 1.0), (1, 0.5), (0, 0.5))
    for _ in range(steps):
        for first, f in layers:
            for i in range(first, L - (1 if ss else 2), 2 if ss else 3):
                (two if ss else three)(i, f * dt)


def _observe(case, B, lam):
    """Densities and currents (J = 1) from the canonical form."""
    d, ss = case["n_max"] + 1, case.get("form") == "supersite"
    b, num = _local_ops(d)
    e = np.eye(d)
    n, cur = [], []
    for k, Bk in enumerate(B):
        t = lam[k][:, None, None] * Bk
        rho = np.einsum("asc,atc->st", t, t.conj())  # <O> = sum O[t, s] rho[s, t]
        if ss:
            n += [np.einsum("ts,st->", np.kron(num, e), rho).real, np.einsum("ts,st->", np.kron(e, num), rho).real]
            cur.append(2.0 * np.einsum("ts,st->", np.kron(b.T, b), rho).imag)
        else:
            n.append(np.einsum("ts,st->", num, rho).real)
        if k + 1 < len(B):
            up, down = (np.kron(e, b.T), np.kron(b, e)) if ss else (b.T, b)
            x = np.tensordot(t, B[k + 1], (2, 0))
            y = np.einsum("us,vt,astb->auvb", up, down, x, optimize=True)
            cur.append(2.0 * np.vdot(x, y).imag)
    return {"n": np.array(n), "cur": np.array(cur)}


def _cost(case, steps):
    """Rough seconds of `steps` plain steps on a few host cores."""
    L, d, chi = _bonds(case)
    f = 0.0
    for k in range(L - 1):
        m, n = sorted((chi[k] * d, d * (1 if case.get("form") == "supersite" else d) * chi[min(L, k + 3)]))
        f += 60.0 * m * m * n
    return (1.2 if case.get("form") == "supersite" else 3.5) * f * steps / 2e10


def exact(case, seed):
    kind = case["kind"]
    if kind == "correlator":
        Bl, lam, Br = _correlator_inputs(case, seed)
        b = torch.from_numpy(_local_ops(case["d"])[0]).cuda().to(torch.complex128)
        x = torch.einsum("a,asm,mtb->astb", lam.to(torch.complex128), Bl, Br)
        y = torch.einsum("su,tv,auvb->astb", b.T, b, x)
        return (x.conj() * y).sum().reshape(1)
    if kind == "zgemm":
        A, B = _zgemm_inputs(case, seed)
        return A @ (B.conj().T if case["opB"] else B)
    if kind == "batch" or (kind != "measure" and _cost(case, case.get("steps", 1)) > (60.0 if kind == "quench" else 12.0)):
        return None
    L, d, _ = _bonds(case)
    if kind == "measure":
        if case["form"] == "u1":
            B, lam, _ = workloads.synthetic_state_u1(L, d, case["chi"], L // 2, seed=seed)
        else:
            B, lam = _dense_state(L, d, case["chi"], seed)
        return _observe(case, B, lam)
    if kind == "quench":
        occ = _occupation(case["L"])
        if case["form"] == "supersite":
            p = np.append(occ, 0) if case["L"] % 2 else occ
            occ = p[::2] * (case["n_max"] + 1) + p[1::2]
        B = [np.eye(d, dtype=complex)[o].reshape(1, d, 1) for o in occ]
        lam, steps = [np.ones(1) for _ in range(L + 1)], case["steps"]
    elif case["form"] == "u1":
        B, lam, _ = workloads.synthetic_state_u1(L, d, case["chi"], L // 2, seed=seed)
        steps = 1
    else:
        B, lam = _dense_state(L, d, case["chi"], seed)
        steps = 1
    _evolve(case, _args(case, seed), B, lam, steps)
    out = dict(_observe(case, B, lam), lam=_table([np.sort(x)[::-1] for x in lam], case["chi"], 0.0),
               chi=None)
    if case["form"] == "u1":
        out["q"] = None
    return out
