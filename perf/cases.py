"""What the library is timed on: beta-steps, growth, single applies and QR gauges.

A user of this framework evolves rho_h(beta) of a Hubbard cluster, ladder or
cylinder: beta-step after beta-step (`Rho.step`), the observables after each
(`Rho.measure`), a checkpoint now and then (`Rho.save`), after a short 2-TDVP
growth (`Rho.grow`); many small instances go out as one `Batch`.  The kernel-
level calls (`heff_apply_terms_host`, `qr_device`) serve programs that bring their own
sweep.  Sizes are those of the workloads module, the tests and the benchmark.

The evolved states of the larger cases are synthetic: U(1)xU(1) sector tables
shaped like those of an evolved state (about 20 sectors per bond, Gaussian in
the charges, the largest with 17 % of the states) and right-canonical tensors
with bond weights falling over two decades, written as a checkpoint and
loaded, because growing them takes minutes.
"""
from __future__ import annotations

import math
import os
import struct
import tempfile

import numpy as np
import torch

from paper_2212_11973_gb300 import tantrg as tt
from paper_2212_11973_gb300 import workloads as wl

DTAU, KRYLOV, BETA = 0.05, 8, 0.5
EXACT = 3  # tt_precision of the exact-accumulation split (the benchmark's mode)

# local basis |0>, |up>, |dn>, |up dn> as (particle number, 2 Sz); pair charges
LOCAL = [(0, 0), (1, 1), (1, -1), (2, 0)]
PAIRS: dict = {}
for _a in range(4):
    for _b in range(4):
        PAIRS.setdefault((LOCAL[_a][0] - LOCAL[_b][0], LOCAL[_a][1] - LOCAL[_b][1]), []).append((_a, _b))
PAIRS = dict(sorted(PAIRS.items()))


def listed():
    """The cases, by what they stand for in use."""
    return [
        # the 4-site parity cluster: every beta-step is launches and latency
        dict(name="step-cluster-2x2-D64-fp64", kind="step", Lx=2, Wy=2, periodic=False, U=4.0, mu=0.0, D=64, prec=0),
        # a 16-site ladder with a checkpoint after the step, as a long run keeps them
        dict(name="step-ladder-2x8-D96-fp64-save", kind="save", Lx=8, Wy=2, periodic=False, U=4.0, mu=-0.3, D=96,
             prec=0),
        # CL4x8 at 1/8 doping in FP64 throughout: the small cylinder's own configuration
        dict(name="step-CL4x8-D256-fp64", kind="step", Lx=8, Wy=4, periodic=True, U=8.0, mu=-2.48, D=256, prec=0),
        # the same cylinder with mixed precision (split-BF16 x6) at its larger D
        dict(name="step-CL4x8-D512-bf16x6", kind="step", Lx=8, Wy=4, periodic=True, U=8.0, mu=-2.48, D=512, prec=2),
        # the benchmark's mode at a middling, ragged D
        dict(name="step-CL4x8-D300-exact", kind="step", Lx=8, Wy=4, periodic=True, U=8.0, mu=-2.48, D=300, prec=EXACT),
        # the headline: width-6 cylinder at D = 1024 on the exact split (3 columns of its 12: the time grows with Lx)
        dict(name="step-CL6x3-D1024-exact", kind="step", Lx=3, Wy=6, periodic=True, U=8.0, mu=-2.48, D=1024,
             prec=EXACT),
        # independent ladders stepped together as one graph
        dict(name="batch-ladders-2x8-n6-bf16x6", kind="batch", n=6, prec=2),
        # a state made from nothing: the MPO, rho_h(beta0), one 2-TDVP growth step, the observables
        dict(name="grow-ladder-2x4-D32-fp64", kind="grow", Lx=4, Wy=2, periodic=False, U=4.0, D=32, prec=0),
        # one H_eff apply on the caller's own host tensors (a program with its own sweep)
        dict(name="apply-W6-D1024-exact", kind="apply", D=1024, Wy=6, prec=EXACT),
        dict(name="apply-W4-D130-fp64", kind="apply", D=130, Wy=4, prec=0),
        # the gauge factorisation of one sector matrix: the tallest of the tests, and an ordinary sector
        dict(name="qr-2100x200-fp64", kind="qr", m=2100, n=200),
        dict(name="qr-333x37-fp64", kind="qr", m=333, n=37),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "save", "batch", "grow", "apply", "qr"])
    if kind in ("step", "save"):
        prec = 0 if kind == "save" else rng.choice([0, 2, EXACT])
        shape = rng.choice(["cluster", "ladder", "CL4", "CL6"])
        if kind == "save" or shape in ("cluster", "ladder"):
            Lx, Wy, per = (2, 2, False) if shape == "cluster" else (rng.randint(4, 8), 2, False)
            hi = 250
        elif shape == "CL4":
            Lx, Wy, per, hi = rng.randint(3, 8), 4, True, 256 if prec == 0 else 512
        else:
            Lx, Wy, per, hi = rng.randint(2, 3), 6, True, 256 if prec == 0 else 1000
        return dict(kind=kind, Lx=Lx, Wy=Wy, periodic=per, U=round(rng.uniform(2.0, 10.0), 3),
                    mu=round(rng.uniform(-2.5, 0.0), 3), D=_log(rng, 24, hi), prec=prec)
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(2, 6), prec=rng.choice([0, 2, EXACT]))
    if kind == "grow":
        return dict(kind="grow", Lx=rng.randint(2, 4), Wy=2, periodic=False, U=round(rng.uniform(2.0, 10.0), 3),
                    D=rng.randint(16, 32), prec=0)
    if kind == "apply":
        return dict(kind="apply", D=_log(rng, 24, 1024), Wy=rng.choice([2, 4, 6]), prec=rng.choice([0, EXACT]))
    n = _log(rng, 8, 200)
    return dict(kind="qr", m=n + _log(rng, 1, 1900), n=n)


# ---- synthetic states ------------------------------------------------------

def sector_dims(D):
    """{charge: dimension} of a bulk bond: Gaussian in (n, 2 Sz) with the largest
    sector at 17 % of D, tails below 1/44 of it truncated (21 sectors)."""
    w = {q: math.exp(-(q[0] ** 2 + q[1] ** 2) / 3.7) for q in wl.SECTOR_CHARGES}
    w = {q: v for q, v in w.items() if v >= 1.0 / 44}
    s = sum(w.values())
    return {q: d for q, v in w.items() if (d := int(v / s * D + 0.5)) > 0}


def chain_sectors(N, D):
    """Sector tables of bonds 0..N: the bulk table wherever the rows and columns
    of the neighbouring blocks can hold it."""
    tab = [{(0, 0): 1}] + [sector_dims(D) for _ in range(N - 1)] + [{(0, 0): 1}]
    while True:
        changed = False
        for k in list(range(1, N)) + list(range(N - 1, 0, -1)):
            new = {}
            for q, d in tab[k].items():
                left = sum(len(s) * tab[k - 1].get((q[0] - p[0], q[1] - p[1]), 0) for p, s in PAIRS.items())
                right = sum(len(s) * tab[k + 1].get((q[0] + p[0], q[1] + p[1]), 0) for p, s in PAIRS.items())
                if (c := min(d, left, right)) > 0:
                    new[q] = c
            changed |= new != tab[k]
            tab[k] = new
        if not changed:
            return [sorted(t.items()) for t in tab]


def _blocks(L, R):
    """Blocks (l, pair charge, r) of a site tensor in layout order: by r, l, p."""
    li = {q: i for i, (q, _) in enumerate(L)}
    out = []
    for r, (rq, dr) in enumerate(R):
        for l, (lq, dl) in enumerate(L):
            p = (rq[0] - lq[0], rq[1] - lq[1])
            if p in PAIRS:
                out.append((l, p, r, dl, len(PAIRS[p]), dr))
    assert len(li) == len(L)
    return out


def random_state(N, D, seed):
    """Right-canonical tensors (site 0 the centre, norm 1) of chain_sectors(N, D)
    as flat FP64 arrays in the library's block layout, and the tables."""
    tab = chain_sectors(N, D)
    g = torch.Generator(device="cuda").manual_seed(1000003 * N + 7919 * D + seed)
    sites = []
    for j in range(N):
        L, R = tab[j], tab[j + 1]
        blk = _blocks(L, R)
        val = [None] * len(blk)
        for l in range(len(L)):
            mine = [i for i, b in enumerate(blk) if b[0] == l]
            parts = []
            for i in mine:
                _, _, _, dl, m, dr = blk[i]
                x = torch.randn((dl, m, dr), generator=g, device="cuda", dtype=torch.float64)
                x *= 10.0 ** (-2.0 * torch.arange(dr, device="cuda", dtype=torch.float64) / max(dr, 1))
                parts.append(x.reshape(dl, m * dr))
            M = torch.cat(parts, 1)
            if j > 0:  # orthonormal rows: Cholesky of the Gram matrix, three times
                M = M / M.norm(dim=1, keepdim=True)
                for _ in range(3):
                    C = torch.linalg.cholesky(M @ M.T)
                    M = torch.linalg.solve_triangular(C, M, upper=False)
            o = 0
            for i in mine:
                n = blk[i][4] * blk[i][5]
                val[i] = M[:, o:o + n].reshape(-1)
                o += n
        a = torch.cat(val)
        sites.append(a / a.norm() if j == 0 else a)
    return tab, sites


def write_checkpoint(path, tab, sites):
    """The library's checkpoint format (tt_rho_save)."""
    with open(path, "wb") as f:
        f.write(b"TTRHO001" + struct.pack("<iddd", len(sites), BETA, 0.0, 0.0))
        for t in tab:
            f.write(struct.pack("<i", len(t)))
            for (n, s), d in t:
                f.write(struct.pack("<iii", n, s, d))
        for a in sites:
            f.write(struct.pack("<q", a.numel()))
            a.cpu().numpy().tofile(f)


def read_sites(path):
    """All site tensors of a checkpoint, one after the other."""
    with open(path, "rb") as f:
        raw = f.read()
    (N,) = struct.unpack_from("<i", raw, 8)
    o, out = 36, []
    for _ in range(N + 1):
        (n,) = struct.unpack_from("<i", raw, o)
        o += 4 + 12 * n
    for _ in range(N):
        (n,) = struct.unpack_from("<q", raw, o)
        out.append(np.frombuffer(raw, np.float64, n, o + 8))
        o += 8 + 8 * n
    return np.concatenate(out)


def _tmp():
    fd, path = tempfile.mkstemp(suffix=".ttck", dir="/dev/shm" if os.path.isdir("/dev/shm") else None)
    os.close(fd)
    return path


class _File:
    """A scratch file that goes with its state."""

    def __init__(self):
        self.path = _tmp()

    def __del__(self):
        try:
            os.unlink(self.path)
        except OSError:
            pass


# ---- preparation ---------------------------------------------------------------

def apply_model(case):
    """Bulk site of the Hubbard MPO on a width-Wy cylinder in automaton form
    (channels start, done, and per operator type the Wy open hops; the oldest
    closes here, a new one opens, the others pass with the parity), and the
    sector tables of the two bonds."""
    Wy, U, mu = case["Wy"], 8.0, -2.48
    F = np.diag([1.0, -1.0, -1.0, 1.0])
    cu, cd = np.zeros((4, 4)), np.zeros((4, 4))
    cu[0, 1] = cu[2, 3] = 1.0
    cd[0, 2], cd[1, 3] = 1.0, -1.0
    nu, nd = np.diag([0.0, 1.0, 0.0, 1.0]), np.diag([0.0, 0.0, 1.0, 1.0])
    opened, closed = [cu.T @ F, cd.T @ F, F @ cu, F @ cd], [cu, cd, cu.T, cd.T]
    onsite = U * (nu - 0.5 * np.eye(4)) @ (nd - 0.5 * np.eye(4)) - mu * (nu + nd)
    chan = [(0, 0), (0, 0)] + [q for q in ((1, 1), (1, -1), (-1, -1), (-1, 1)) for _ in range(Wy)]
    W = [(0, 0, np.eye(4)), (1, 1, np.eye(4)), (0, 1, onsite)]
    for o in range(4):
        at = 2 + o * Wy
        W += [(0, at + Wy - 1, opened[o]), (at, 1, -closed[o])] + [(at + i, at + i - 1, F) for i in range(1, Wy)]
    terms = [(wl, wr, s, t, float(op[s, t])) for wl, wr, op in W for s in range(4) for t in range(4) if op[s, t]]
    tables = [[(n, s, d) for (n, s), d in sorted(sector_dims(D).items())] for D in (case["D"], max(16, case["D"] - 3))]
    return chan, terms, tables[0], tables[1]


def apply_inputs(case, seed):
    chan, _, SL, SR = apply_model(case)
    nx, nl, nr = tt.layout_sizes_terms(chan, chan, SL, SR)
    return [wl.random_vector(n, 4 * seed + i) for i, n in enumerate((nl, nr, nx))]


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.Stream()
    if kind == "qr":
        g = torch.Generator(device="cuda").manual_seed(seed)
        A = torch.randn((case["m"], case["n"]), generator=g, device="cuda", dtype=torch.float64)
        return dict(case=case, ctx=tt.Context(), A=A)
    if kind == "apply":
        return dict(case=case, ctx=tt.Context(), model=apply_model(case), v=apply_inputs(case, seed))
    rng = np.random.default_rng(seed)
    with torch.cuda.stream(stream):
        ctx = tt.Context(stream=stream)
        if kind == "batch":
            ws = wl.batch_ladders(case["n"], wl.BATCH_SEED + seed)
            b = tt.Batch(ctx, ws, ws[0].beta0, tt.run_opts(0, KRYLOV, case["prec"]))
            b.pad()
            # past the zero-weight start, whose rank-deficient sectors take the
            # Householder fallback: what a run to beta = 8 does from then on
            b.step(DTAU, 4)
            return dict(case=case, ctx=ctx, batch=b, stream=stream)
        if kind == "grow":
            mu = float(rng.uniform(-2.0, 0.0))
            return dict(case=case, ctx=ctx, mu=mu, stream=stream)
        mpo = tt.Mpo(ctx, case["Lx"], case["Wy"], case["periodic"], t=1.0, U=case["U"], mu=case["mu"], form=1)
        f = _File()
        write_checkpoint(f.path, *random_state(case["Lx"] * case["Wy"], case["D"], seed))
        rho = tt.Rho.load(ctx, mpo, f.path, tt.run_opts(case["D"], KRYLOV, case["prec"]))
        stream.synchronize()
    return dict(case=case, ctx=ctx, mpo=mpo, rho=rho, stream=stream, file=f)


# ---- one pass ----------------------------------------------------------------------

OBS = ("energy_per_site", "density", "double_occ", "free_energy_per_site", "lnZ")


def _obs(o):
    return {k: o[k] for k in OBS}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "qr":
        Q, R = tt.qr_device(state["ctx"], state["A"])
        return {"Q": Q, "R": R}
    if kind == "apply":
        chan, terms, SL, SR = state["model"]
        return tt.heff_apply_terms_host(state["ctx"], chan, chan, terms, case["prec"], SL, SR, *state["v"])
    if kind == "batch":
        state["batch"].step(DTAU, 1)
        return [_obs(o) for o in state["batch"].measure()]
    if kind == "grow":
        ctx = state["ctx"]
        mpo = tt.Mpo(ctx, case["Lx"], case["Wy"], case["periodic"], t=1.0, U=case["U"], mu=state["mu"], form=1)
        rho = tt.Rho(ctx, mpo, 0.01, tt.run_opts(case["D"], KRYLOV, case["prec"]))
        rho.grow(DTAU, 0.05)
        out = _obs(rho.measure())
        rho.close()
        mpo.close()
        return out
    state["rho"].step(DTAU, 1)
    out = _obs(state["rho"].measure())
    if kind == "save":
        state["rho"].save(state["file"].path)
        out["tensors"] = read_sites(state["file"].path)
    return out


# ---- what a pass cannot do without -------------------------------------------------

def _channels(Wy):
    """Channel charges of a bulk MPO bond: start, done and 4 open hops per row."""
    return [(0, 0), (0, 0)] + [(a, b) for a in (1, -1) for b in (1, -1)] * Wy


def _apply_flops(L, R, chan):
    dl, dr = dict(L), dict(R)
    f = 0.0
    for (_, _, r, a, m, b), (l, p) in ((x, (x[0], x[1])) for x in _blocks(L, R)):
        lq, rq = L[l][0], R[r][0]
        rows = sum(dl.get((lq[0] + c[0], lq[1] + c[1]), 0) for c in chan)
        cols = sum(dr.get((rq[0] - c[0], rq[1] - c[1]), 0) for c in chan)
        f += 2.0 * a * m * b * (rows + cols)
    return f


def _chain_work(case):
    """One beta-step: per half sweep and site K applies, the environment update
    (an apply's worth of GEMMs), the QR; per bond K bond applies and the absorb.
    Bytes: every site tensor read and written once."""
    N = case["Lx"] * case["Wy"]
    tab, chan = chain_sectors(N, case["D"]), _channels(case["Wy"])
    flops = nbytes = 0.0
    for j in range(N):
        L, R = tab[j], tab[j + 1]
        size = sum(b[3] * b[4] * b[5] for b in _blocks(L, R))
        flops += 2 * (KRYLOV + 1) * _apply_flops(L, R, chan)
        nbytes += 16.0 * size
        if j + 1 < N:
            d = dict(R)
            rows = {r: 0 for r in range(len(R))}
            for b in _blocks(L, R):
                rows[b[2]] += b[3] * b[4]
            flops += 2 * sum(4.0 * rows[r] * d[R[r][0]] ** 2 for r in rows)
            for q, dq in R:
                others = sum(d.get((q[0] + c[0], q[1] + c[1]), 0) for c in chan)
                flops += 2 * KRYLOV * 4.0 * dq * dq * others
            flops += 2 * sum(2.0 * rows[r] * d[R[r][0]] ** 2 for r in rows)
    return {"bytes": nbytes, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "qr":
        m, n = case["m"], case["n"]
        return {"bytes": 8.0 * (2 * m * n + n * n), "flops": 4.0 * m * n * n - 4.0 / 3.0 * n ** 3}
    if kind == "apply":
        chan, _, SL, SR = apply_model(case)
        L, R = [((n, s), d) for n, s, d in SL], [((n, s), d) for n, s, d in SR]
        env = sum(d * dict(T).get((q[0] + c[0], q[1] + c[1]), 0) for T in (L, R) for q, d in T for c in chan)
        size = sum(b[3] * b[4] * b[5] for b in _blocks(L, R))
        return {"bytes": 8.0 * (2 * size + env), "flops": _apply_flops(L, R, chan)}
    if kind == "batch":
        out = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["n"]):
            w = _chain_work(dict(Lx=8, Wy=2, D=(64, 96, 128)[i % 3]))
            out = {k: out[k] + w[k] for k in out}
        return out
    return _chain_work(case)


# ---- the same in 64 bits, without the library ---------------------------------------

def _qr_exact(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn((case["m"], case["n"]), generator=g, device="cuda", dtype=torch.float64).cpu().numpy()
    Q, R = np.linalg.qr(A)
    s = np.where(np.diag(R) < 0, -1.0, 1.0)
    return {"Q": Q * s, "R": s[:, None] * R}


def _apply_exact(case, seed):
    """y = L W x R on dense FP64 tensors, read back in the block layout."""
    chan, terms, SL, SR = apply_model(case)
    Lv, Rv, xv = apply_inputs(case, seed)
    dev = torch.device("cuda")

    def offsets(S):
        return np.concatenate([[0], np.cumsum([d for _, _, d in S])])

    def env(v, S):
        v, off, o = torch.from_numpy(v).to(dev), offsets(S), 0
        at = {(n, s): i for i, (n, s, _) in enumerate(S)}
        E = torch.zeros((len(chan), off[-1], off[-1]), dtype=torch.float64, device=dev)
        for b, (n, s, d) in enumerate(S):
            for w, c in enumerate(chan):
                a = at.get((n + c[0], s + c[1]))
                if a is not None:
                    k = S[a][2] * d
                    E[w, off[a]:off[a + 1], off[b]:off[b + 1]] = v[o:o + k].reshape(-1, d)
                    o += k
        return E

    ol, orr = offsets(SL), offsets(SR)
    blk = _blocks([((n, s), d) for n, s, d in SL], [((n, s), d) for n, s, d in SR])
    x = torch.zeros((ol[-1], 4, 4, orr[-1]), dtype=torch.float64, device=dev)
    xt, o = torch.from_numpy(xv).to(dev), 0
    for l, p, r, dl, m, dr in blk:
        b = xt[o:o + dl * m * dr].reshape(dl, m, dr)
        o += dl * m * dr
        for k, (s, t) in enumerate(PAIRS[p]):
            x[ol[l]:ol[l + 1], s, t, orr[r]:orr[r + 1]] = b[:, k]
    L, R = env(Lv, SL), env(Rv, SR)
    y = torch.zeros_like(x)
    by_wr: dict = {}
    for t in terms:
        by_wr.setdefault(t[1], []).append(t)
    T1 = torch.einsum("wab,bstc->wastc", L, x)
    for wr, ts in by_wr.items():
        T2 = torch.zeros_like(x)
        for wl_, _, s, t, v in ts:
            T2[:, s] += v * T1[wl_][:, t]
        y += torch.einsum("astb,cb->astc", T2, R[wr])
    out = [y[ol[l]:ol[l + 1], [s for s, _ in PAIRS[p]], [t for _, t in PAIRS[p]], orr[r]:orr[r + 1]].reshape(-1)
           for l, p, r, _, _, _ in blk]
    return torch.cat(out).cpu().numpy()


def _cluster_hamiltonian(case):
    """H of the open 2x2 cluster on 4^4 states, sites in snake order
    (0,0) (0,1) (1,1) (1,0), modes (site, up) < (site, dn)."""
    I2, Z = np.eye(2), np.diag([1.0, -1.0])
    a = np.array([[0.0, 1.0], [0.0, 0.0]])

    def mode(k):  # annihilation operator of mode k of 8 (bit order: site major, up then dn)
        m = np.eye(1)
        for i in range(8):
            m = np.kron(m, Z if i < k else a if i == k else I2)
        return m

    c = [mode(k) for k in range(8)]
    H = np.zeros((256, 256))
    for i, j in ((0, 1), (1, 2), (2, 3), (0, 3)):
        for s in (0, 1):
            h = c[2 * i + s].T @ c[2 * j + s]
            H -= h + h.T
    n = [x.T @ x for x in c]
    one = np.eye(256)
    for i in range(4):
        H += case["U"] * (n[2 * i] - 0.5 * one) @ (n[2 * i + 1] - 0.5 * one) - case["mu"] * (n[2 * i] + n[2 * i + 1])
    # site basis |0>, |up>, |dn>, |up dn>: bits (up, dn) in kron order give 0, dn, up, updn
    perm = [0, 2, 1, 3]
    idx = [((perm[p] * 4 + perm[q]) * 4 + perm[r]) * 4 + perm[s] for p in range(4) for q in range(4) for r in range(4)
           for s in range(4)]
    dens = sum(n) / 4.0
    docc = sum(n[2 * i] @ n[2 * i + 1] for i in range(4)) / 4.0
    return [x[np.ix_(idx, idx)] for x in (H, dens, docc)]


def _cluster_step_exact(case, seed):
    """One symmetric 1-TDVP beta-step of the 4-site chain with dense projected
    Hamiltonians P^T (H x 1) P (P the tensors left and right of the centre)."""
    N = 4
    tab, sites = random_state(N, case["D"], seed)
    A = []
    for j in range(N):
        L, R = tab[j], tab[j + 1]
        ol = np.concatenate([[0], np.cumsum([d for _, d in L])])
        orr = np.concatenate([[0], np.cumsum([d for _, d in R])])
        X = np.zeros((ol[-1], 16, orr[-1]))
        v, o = sites[j].cpu().numpy(), 0
        for l, p, r, dl, m, dr in _blocks(L, R):
            b = v[o:o + dl * m * dr].reshape(dl, m, dr)
            o += dl * m * dr
            for k, (s, t) in enumerate(PAIRS[p]):
                X[ol[l]:ol[l + 1], 4 * s + t, orr[r]:orr[r + 1]] = b[:, k]
        A.append(X)
    H, dens, docc = _cluster_hamiltonian(case)

    def act(op, psi):  # op on the ket indices of psi[(s0 t0), (s1 t1), ...]
        x = psi.reshape([4, 4] * N).transpose(0, 2, 4, 6, 1, 3, 5, 7).reshape(256, 256)
        y = (op @ x).reshape([4] * 8)
        return y.transpose(0, 4, 1, 5, 2, 6, 3, 7).reshape(-1)

    def left(j):
        M = np.eye(1)
        for k in range(j):
            M = np.einsum("xa,apb->xpb", M, A[k]).reshape(-1, A[k].shape[2])
        return M

    def right(j):
        M = np.eye(1)
        for k in range(N - 1, j, -1):
            M = np.einsum("apb,bx->apx", A[k], M).reshape(A[k].shape[0], -1)
        return M

    def evolve(x, t, Lm, Rm, bond):
        """exp(t H_eff) x / norm, by Lanczos with full reorthogonalisation; ln of the norm."""
        shape = x.shape

        def heff(v):
            v = v.reshape(shape)
            if bond:
                full = Lm @ v @ Rm
                y = act(H, full.reshape(-1)).reshape(full.shape)
                return (Lm.T @ y @ Rm.T).reshape(-1)
            full = np.einsum("xa,apb,by->xpy", Lm, v, Rm, optimize=True)
            y = act(H, full.reshape(-1)).reshape(full.shape)
            return np.einsum("xa,xpy,by->apb", Lm, y, Rm, optimize=True).reshape(-1)

        nb = np.linalg.norm(x)
        Q, al, be = [x.reshape(-1) / nb], [], []
        for k in range(KRYLOV):
            w = heff(Q[k])
            al.append(Q[k] @ w)
            for _ in range(2):
                for q in Q:
                    w = w - (q @ w) * q
            b = np.linalg.norm(w)
            if k == KRYLOV - 1 or b <= 1e-13 * max(abs(np.array(al))):
                break
            be.append(b)
            Q.append(w / b)
        e, V = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
        c = V @ (np.exp(t * e) * V[0]) * nb
        y = sum(ci * q for ci, q in zip(c, Q))
        n = np.linalg.norm(y)
        return (y / n).reshape(shape), math.log(n)

    tau, logs = DTAU / 4, 0.0
    for j in range(N):
        A[j], s = evolve(A[j], -tau, left(j), right(j), False)
        logs += s
        if j < N - 1:
            a, p, b = A[j].shape
            q, S = np.linalg.qr(A[j].reshape(a * p, b))
            A[j] = q.reshape(a, p, -1)
            S, s = evolve(S, tau, left(j + 1), right(j), True)
            logs += s
            A[j + 1] = np.einsum("xa,apb->xpb", S, A[j + 1])
    for j in range(N - 1, -1, -1):
        A[j], s = evolve(A[j], -tau, left(j), right(j), False)
        logs += s
        if j > 0:
            a, p, b = A[j].shape
            q, S = np.linalg.qr(A[j].reshape(a, p * b).T)
            A[j] = q.T.reshape(-1, p, b)
            S, s = evolve(S.T, tau, left(j), right(j - 1), True)
            logs += s
            A[j - 1] = np.einsum("apb,bx->apx", A[j - 1], S)
    psi = (left(3) @ A[3].reshape(A[3].shape[0], -1)).reshape(-1)
    z = psi @ psi
    lnZ = 2 * logs + math.log(z)
    ev = [float(psi @ act(op, psi) / z) for op in (H, dens, docc)]
    return {"energy_per_site": ev[0] / N, "density": ev[1], "double_occ": ev[2],
            "free_energy_per_site": -lnZ / ((BETA + DTAU) * N), "lnZ": lnZ}


def exact(case, seed):
    if case["kind"] == "qr":
        return _qr_exact(case, seed)
    if case["kind"] == "apply":
        return _apply_exact(case, seed)
    if case["kind"] in ("step", "save") and case["Lx"] * case["Wy"] == 4:
        out = _cluster_step_exact(case, seed)
        if case["kind"] == "save":
            out["tensors"] = None
        return out
    return None
