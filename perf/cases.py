"""Performance cases: the calls a user of the framework makes, over the sizes of
its configurations and tests.

Every state is a seeded random block-sparse MPS in the gauge fits leave behind
(sector dimensions in proportion to the number of configurations, random
right-orthonormal site tensors, unit norm) and every Hamiltonian a seeded synthetic integral set: h symmetric with
diagonal U[-2, -0.5] and off-diagonal N(0, 0.1/(1+|i-j|)^2), (ij|kl) = sum_g
L^g_ij L^g_kl with 16 symmetric factors L^g_ij ~ N(0, 0.3/(1+|i-j|)).

Results of mixed-precision contexts are read in the type the context computes
in: complex64 for split TF32, bfloat16 real/imaginary pairs for BF16.
Site tensors are returned wherever the gauge of the result is fixed (one-site
schedules: QR with a positive diagonal) and its sectors well conditioned; the
results of truncated SVDs and of whole time steps, whose site tensors carry an
arbitrary or ill-conditioned gauge, are read as a user reads them, by the
one-body density matrix, norm and energy.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1902_08489_gb300 as td

SITE = ((0, 0), (1, 1), (1, -1), (2, 0))
N_CHOL = 16
DT = 0.05


def listed():
    return [
        # the smallest call: the projection of one small state on another, taken
        # after every step of a correlation function
        dict(name="overlap_small", kind="overlap", L=8, n=7, sz=1, D=32, prec="fp64"),
        # <phi|H|psi>: one entry of the Krylov Hamiltonian matrix, the operation
        # a time step repeats most
        dict(name="expectation", kind="expectation", L=16, n=15, sz=1, D=256, prec="fp64"),
        # the backward pass: energy and its adjoint with respect to every site tensor
        dict(name="energy_gradient", kind="gradient", L=12, n=12, sz=0, D=128, prec="fp64"),
        # a local iterative solver at the centre site: 8 products with the one-site
        # effective Hamiltonian, environments kept
        dict(name="local_operator", kind="local", L=16, n=15, sz=1, D=256, prec="tf32x3", site=8,
             reps=8),
        # the final superposition of a Runge-Kutta step: five states fitted into one
        dict(name="sum_of_five", kind="sum", L=12, n=12, sz=0, D=128, prec="fp64", terms=5,
             one_site=1),
        # a state truncated to half its bond dimension by SVD
        dict(name="compress", kind="compress", L=16, n=15, sz=1, D=256, prec="fp64", D_out=128),
        # the headline operation: one fitted H|psi> on the split-TF32 tensor cores
        dict(name="apply_H", kind="apply", L=16, n=15, sz=1, D=256, prec="tf32x3", one_site=1),
        # the same in full precision, on a smaller and odd-sized system
        dict(name="apply_H_fp64", kind="apply", L=11, n=11, sz=1, D=117, prec="fp64", one_site=1),
        # a larger active space in BF16
        dict(name="apply_H_bf16", kind="apply", L=24, n=23, sz=1, D=128, prec="bf16", one_site=1),
        # the small full-precision trajectory: one Runge-Kutta step with the default
        # schedule of the library (two-site sweeps with truncated SVDs, then one-site)
        dict(name="rk4_two_site", kind="rk4", L=8, n=7, sz=1, D=64, prec="fp64", two_site=2,
             one_site=2),
        # an ensemble of independent systems advanced together on worker streams
        dict(name="batch_rk4", kind="batch", L=14, n=14, sz=0, D=128, prec="tf32x3", items=4,
             one_site=2),
        # the flagship time step at its size: orthogonal Krylov basis, full-precision
        # inner products beside split-TF32 fits
        dict(name="krylov_step", kind="krylov", L=16, n=15, sz=1, D=256, prec="tf32x3", m=4,
             two_site=0, one_site=2),
    ]


def draw(rng):
    kind = rng.choice(["overlap", "expectation", "gradient", "local", "sum", "compress", "apply",
                       "apply", "rk4", "batch", "krylov", "krylov"])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    L = rng.randint(6, 16)
    n = L - rng.choice([0, 0, 1])
    c = dict(kind=kind, L=L, n=n, sz=n % 2, D=log_int(16, 256), prec="fp64")
    if kind == "local":
        c.update(prec=rng.choice(["fp64", "tf32x3"]), site=rng.randrange(L),
                 reps=rng.choice([2, 4, 8]))
    elif kind == "sum":
        c.update(terms=rng.randint(2, 8), one_site=1)
    elif kind == "compress":
        c.update(D_out=max(4, int(c["D"] * rng.uniform(0.3, 0.8))))
    elif kind == "apply":
        c.update(prec=rng.choice(["fp64", "tf32x3", "bf16"]), one_site=1)
    elif kind == "rk4":
        c.update(L=min(L, 9), D=log_int(16, 72), two_site=rng.randint(1, 2), one_site=1)
        c.update(n=c["L"] - 1, sz=(c["L"] - 1) % 2)
    elif kind == "batch":
        c.update(L=min(L, 14), D=log_int(16, 128), prec=rng.choice(["fp64", "tf32x3"]),
                 items=rng.randint(2, 6), one_site=1)
        c.update(n=c["L"], sz=c["L"] % 2)
    elif kind == "krylov":
        c.update(m=rng.randint(3, 4), prec=rng.choice(["fp64", "tf32x3"]),
                 two_site=0, one_site=rng.randint(1, 2))
        if c["prec"] == "fp64":   # no dearer than the listed step
            c.update(D=min(c["D"], 160))
        if rng.random() < 0.5:   # the physical schedule, on a smaller system
            c.update(L=min(L, 10), D=log_int(16, 72), two_site=1, one_site=1)
            c.update(n=c["L"] - 1, sz=(c["L"] - 1) % 2)
    return c


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=None)
def _bond_dims(L, n, sz, D):
    """Per bond: {(N, 2Sz): dimension}, in charge order."""
    up, dn = (n + sz) // 2, (n - sz) // 2
    bonds = []
    for k in range(L + 1):
        most = {}
        for a in range(k + 1):
            for b in range(k + 1):
                if 0 <= up - a <= L - k and 0 <= dn - b <= L - k:
                    most[(a + b, a - b)] = min(math.comb(k, a) * math.comb(k, b),
                                               math.comb(L - k, up - a) * math.comb(L - k, dn - b))
        most = dict(sorted(most.items()))
        total = sum(most.values())
        if total > D:
            share = {q: D * m / total for q, m in most.items()}
            d = {q: min(most[q], int(share[q])) for q in most}
            for q in sorted(share, key=lambda q: (int(share[q]) - share[q], q)):
                if sum(d.values()) < D and d[q] < most[q]:
                    d[q] += 1
            most = d
        bonds.append(most)
    changed = True
    while changed:   # no sector larger than its neighbours can reach
        changed = False
        order = [(k, k - 1, -1) for k in range(1, L + 1)] + [(k, k + 1, 1) for k in range(L - 1, -1, -1)]
        for k, nb, sign in order:
            for q in bonds[k]:
                lim = sum(bonds[nb].get((q[0] + sign * s[0], q[1] + sign * s[1]), 0) for s in SITE)
                if bonds[k][q] > lim:
                    bonds[k][q] = lim
                    changed = True
    return [{q: d for q, d in b.items() if d > 0} for b in bonds]


def _state(c, rng):
    """(tensors, labels) of a random state of case c."""
    bonds = _bond_dims(c["L"], c["n"], c["sz"], c["D"])
    labels = [np.array([q for q, d in b.items() for _ in range(d)], dtype=np.int64).reshape(-1, 2)
              for b in bonds]
    off = []
    for b in bonds:
        o, at = {}, 0
        for q, d in b.items():
            o[q] = at
            at += d
        off.append(o)
    tensors = []
    for i in range(c["L"]):
        A = np.zeros((len(labels[i]), 4, len(labels[i + 1])), dtype=np.complex128)
        for q, d in bonds[i].items():
            cols = [(s, off[i + 1][p], bonds[i + 1][p]) for s, x in enumerate(SITE)
                    for p in [(q[0] + x[0], q[1] + x[1])] if p in bonds[i + 1]]
            n = sum(e for _, _, e in cols)
            Q = np.linalg.qr(rng.standard_normal((n, d)) + 1j * rng.standard_normal((n, d)))[0].T
            for s, at, e in cols:
                A[off[i][q]:off[i][q] + d, s, at:at + e] = Q[:, :e]
                Q = Q[:, e:]
        tensors.append(A)
    return tensors, labels


def _integrals(L, rng):
    """h (L x L) and the Cholesky factors (N_CHOL x L x L) of (ij|kl)."""
    i, j = np.triu_indices(L)
    dist = 1.0 + np.abs(i - j)
    h = np.zeros((L, L))
    h[i, j] = h[j, i] = np.where(i == j, rng.uniform(-2.0, -0.5, len(i)),
                                 rng.standard_normal(len(i)) * 0.1 / dist ** 2)
    chol = np.zeros((N_CHOL, L, L))
    chol[:, i, j] = rng.standard_normal((N_CHOL, len(i))) * 0.3 / dist
    chol[:, j, i] = chol[:, i, j]
    return h, chol


def _items(case):
    """The systems of a case: one, or the uneven instances of a batch."""
    if case["kind"] != "batch":
        return [case]
    out = []
    for k in range(case["items"]):
        L = max(6, case["L"] - 2 * (k % 4))
        out.append(dict(case, kind="rk4", two_site=0, L=L, n=L, sz=L % 2,
                        D=max(8, case["D"] >> (k % 3))))
    return out


def _inputs(case, seed):
    """Host inputs of every system of a case: (h, chol, [states])."""
    rng = np.random.default_rng([seed, case["L"], case["D"]])
    out = []
    for c in _items(case):
        h, chol = _integrals(c["L"], rng)
        count = {"overlap": 2, "expectation": 2, "sum": c.get("terms", 0)}.get(c["kind"], 1)
        out.append((h, chol, [_state(c, rng) for _ in range(count)]))
    return out


def _coefficients(terms):
    """Complex weights of a fitted sum, the first one dominant."""
    return [1.0] + [(0.5 + 0.1 * k) * (1j if k % 2 else -1.0) / 3.0 for k in range(1, terms)]


def prepare(case, seed):
    ctx = td.Context(case["prec"])
    ctx.set_schedule(case.get("two_site", 0), case.get("one_site", 1))
    mpos, states = [], []
    for c, (h, chol, st) in zip(_items(case), _inputs(case, seed)):
        if case["kind"] not in ("overlap", "sum", "compress"):
            eri = np.einsum("gij,gkl->ijkl", chol, chol, optimize=True)
            mpos.append(td.build_mpo(ctx, h, eri, n_elec=c["n"]))
        states += [td.mps_import(ctx, A, q) for A, q in st]
    state = dict(case=case, ctx=ctx, mpos=mpos, states=states)
    if case["kind"] == "local":
        state["op"] = td.local_hamiltonian(ctx, mpos[0], states[0], case["site"])
        state["work"] = [states[0].copy(), states[0].copy()]
    return state


# ------------------------------------------------------------------ one pass

def _read(case, x):
    """A result in the type its context computes in."""
    x = torch.from_numpy(x)
    if case["prec"] == "bf16":
        return torch.view_as_real(x).to(torch.bfloat16)
    return x if case["prec"] == "fp64" else x.to(torch.complex64)


def _observe(ctx, case, mpo, psi):
    """What a user records after a time step."""
    return dict(rdm=_read(case, td.one_rdm(ctx, psi)),
                norm=_read(case, np.array([td.overlap(ctx, psi, psi)])),
                energy=_read(case, np.array([td.expectation(ctx, mpo, psi, psi)])))


def run(state):
    case, ctx, mpos, states = state["case"], state["ctx"], state["mpos"], state["states"]
    kind, D = case["kind"], case["D"]
    if kind == "overlap":
        return np.complex128(td.overlap(ctx, states[0], states[1]))
    if kind == "expectation":
        return np.complex128(td.expectation(ctx, mpos[0], states[0], states[1]))
    if kind == "gradient":
        energy, grad, _ = td.energy_gradient(ctx, mpos[0], states[0])
        return [np.float64(energy)] + grad.export()[0]
    if kind == "local":
        x = states[0]
        for r in range(case["reps"]):
            y = state["work"][r % 2]
            state["op"].apply(x, y)
            x = y
        return _read(case, x.export()[0][case["site"]])
    if kind == "sum":
        out = td.mps_sum(ctx, _coefficients(case["terms"]), states, D, 0.0)
        return out.export()[0]
    if kind == "compress":
        psi = states[0].copy()
        lost = td.compress(ctx, psi, case["D_out"], 1e-12)
        return dict(lost=np.float64(lost), rdm=td.one_rdm(ctx, psi))
    if kind == "apply":
        out = td.apply_H(ctx, mpos[0], states[0], -1j * DT, D, 0.0)
        return [_read(case, t) for t in out.export()[0]]
    if kind == "rk4":
        psi = states[0].copy()
        td.rk4_step(ctx, mpos[0], psi, 0.01, D, 0.0)
        return _observe(ctx, case, mpos[0], psi)
    if kind == "batch":
        psis = [s.copy() for s in states]
        td.evolve_batch(ctx, mpos, psis, 0.01, 1, [c["D"] for c in _items(case)], method="rk4",
                        n_workers=4)
        return [_read(case, td.one_rdm(ctx, p)) for p in psis]
    psi = states[0].copy()
    td.krylov_step(ctx, mpos[0], psi, DT, case["m"], True, D, 1e-8)
    return _observe(ctx, case, mpos[0], psi)


# ------------------------------------------------------------------ algorithmic work

@functools.lru_cache(maxsize=None)
def _mpo_blocks(L):
    """Per bond {charge: channels}, per site {(s, s', g_out): non-zeros}, non-zeros."""
    h, chol = _integrals(L, np.random.default_rng(0))
    mpo = td.build_mpo(None, h, np.einsum("gij,gkl->ijkl", chol, chol, optimize=True))
    charge = {0: (0, 0)}
    bonds, tables, nnz = [{(0, 0): 1}], [], 0
    for i in range(L):
        win, wout, s, sp, _ = mpo.elements(i)
        nnz += len(win)
        nxt = {}
        table = {}
        site = np.array(SITE)
        qin = np.array([charge[w] for w in range(max(charge) + 1)])
        q = qin[win] + site[s] - site[sp]
        for w, (a, b) in zip(wout.tolist(), q.tolist()):
            nxt[w] = (a, b)
        key, count = np.unique(np.column_stack([s, sp, q]), axis=0, return_counts=True)
        for (x, y, a, b), m in zip(key.tolist(), count.tolist()):
            table[(x, y, (a, b))] = m
        size = {}
        for v in nxt.values():
            size[v] = size.get(v, 0) + 1
        charge = nxt
        bonds.append(size)
        tables.append(table)
    return bonds, tables, nnz


def _sub(a, b):
    return a[0] - b[0], a[1] - b[1]


def _add(a, b):
    return a[0] + b[0], a[1] + b[1]


@functools.lru_cache(maxsize=None)
def _site_flops(L, n, sz, D, operator):
    """Per site: real operations of one environment step (product with the
    ket, with the operator, with the bra), block-sparse, 8 per complex
    multiply-add."""
    bonds = _bond_dims(L, n, sz, D)
    if operator:
        mb, tables, _ = _mpo_blocks(L)
    else:
        mb = [{(0, 0): 1}] * (L + 1)
        tables = [{}] * L
    out = []
    for i in range(L):
        total = 0.0
        for qa, da in bonds[i].items():
            done = set()
            for g, W in mb[i].items():
                ka = _sub(qa, g)
                if ka not in bonds[i]:
                    continue
                for sp in range(4):
                    kb = _add(ka, SITE[sp])
                    e = bonds[i + 1].get(kb, 0)
                    if not e:
                        continue
                    total += 8.0 * da * W * bonds[i][ka] * e
                    for s in range(4):
                        f = bonds[i + 1].get(_add(qa, SITE[s]), 0)
                        go = _add(g, _sub(SITE[s], SITE[sp]))
                        m = tables[i].get((s, sp, go), 0) if operator else int(s == sp)
                        if not f or not m:
                            continue
                        total += 4.0 * m * da * e if operator else 0.0
                        if (s, go) not in done:
                            done.add((s, go))
                            total += 8.0 * f * da * mb[i + 1][go] * e
        out.append(total)
    return out


def _fit_flops(c, terms, operator):
    """A fit: environments from the right, then a local product and an
    environment update per site and direction of every sweep."""
    s = sum(_site_flops(c["L"], c["n"], c["sz"], c["D"], operator))
    return terms * s * (1.0 + 8.0 / 3.0 * (c.get("one_site", 1) + 2 * c.get("two_site", 0)))


def _entries(c):
    bonds = _bond_dims(c["L"], c["n"], c["sz"], c["D"])
    return sum(d * bonds[i + 1].get(_add(q, x), 0) for i in range(c["L"])
               for q, d in bonds[i].items() for x in SITE)


def work(case):
    flops = nbytes = 0.0
    for c in _items(case):
        key = (c["L"], c["n"], c["sz"], c["D"])
        kind, state = c["kind"], 16.0 * _entries(c)
        ham = 16.0 * _mpo_blocks(c["L"])[2] if kind not in ("overlap", "sum", "compress") else 0.0
        if kind == "overlap":
            flops += sum(_site_flops(*key, False))
            nbytes += 2 * state
        elif kind == "expectation":
            flops += sum(_site_flops(*key, True))
            nbytes += 2 * state + ham
        elif kind == "gradient":
            flops += sum(_site_flops(*key, True)) * 8.0 / 3.0
            nbytes += 2 * state + ham
        elif kind == "local":
            flops += c["reps"] * _site_flops(*key, True)[c["site"]]
            env = sum(d * b.get(_sub(q, g), 0) * w
                      for k in (0, 1)
                      for b in [_bond_dims(*key)[c["site"] + k]]
                      for g, w in _mpo_blocks(c["L"])[0][c["site"] + k].items()
                      for q, d in b.items())
            nbytes += 8.0 * env + ham / c["L"]
        elif kind == "sum":
            flops += _fit_flops(c, c["terms"], False)
            nbytes += (c["terms"] + 1) * state
        elif kind == "compress":
            bonds = _bond_dims(*key)
            for i in range(c["L"]):
                for q, d in bonds[i + 1].items():
                    rows = sum(bonds[i].get(_sub(q, x), 0) for x in SITE)
                    flops += 3 * 8.0 * rows * d * d
            nbytes += state * (1 + c["D_out"] / c["D"])
        elif kind == "apply":
            flops += _fit_flops(c, 1, True)
            nbytes += 2 * state + ham
        elif kind == "rk4":
            flops += _fit_flops(c, 4, True) + _fit_flops(c, 11, False)
            nbytes += 2 * state + ham
        else:
            m = c["m"]
            flops += _fit_flops(c, m - 1, True) + _fit_flops(c, m * (m + 1) // 2 + m - 1, False)
            flops += m * (m + 1) / 2 * (sum(_site_flops(*key, True)) + sum(_site_flops(*key, False)))
            nbytes += 2 * state + ham
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------ 64-bit values

def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda", torch.complex128)


def _vector(tensors):
    """The 4^L amplitudes of an MPS, site 0 slowest."""
    v = torch.ones(1, 1, dtype=torch.complex128, device="cuda")
    for A in tensors:
        v = (v @ A.reshape(A.shape[0], -1)).reshape(-1, A.shape[2])
    return v.reshape(-1)


# (from, to, sign) of the annihilators of |0>, |up>, |down>, |up down> = c+_up c+_down |0>
LOWER = (((1, 0, 1.0), (3, 2, 1.0)), ((2, 0, 1.0), (3, 1, -1.0)))


def _ladder(v, L, k, spin, raising):
    """c_(k spin) v, or its adjoint, with the Jordan-Wigner sign of sites before k."""
    v = v.reshape(4 ** k, 4, -1)
    sign = torch.ones(1, dtype=torch.complex128, device="cuda")
    for _ in range(k):
        sign = torch.kron(sign, torch.tensor([1, -1, -1, 1], dtype=torch.complex128, device="cuda"))
    out = torch.zeros_like(v)
    for a, b, x in LOWER[spin]:
        if raising:
            a, b = b, a
        out[:, b] += x * sign[:, None] * v[:, a]
    return out.reshape(-1)


def _one_body(v, L, M):
    """sum_ij,s M_ij c+_is c_js v for every matrix M of a list."""
    low = [torch.stack([_ladder(v, L, j, s, False) for j in range(L)]) for s in range(2)]
    outs = []
    for m in M:
        m = _dev(m)
        out = torch.zeros_like(v)
        for s in range(2):
            mixed = m @ low[s]
            for i in range(L):
                out += _ladder(mixed[i], L, i, s, True)
        outs.append(out)
    return outs


def _hamiltonian(v, h, chol):
    """H v = sum h' E v + 1/2 sum_g O_g O_g v, O_g = sum_ij L^g_ij E_ij."""
    L = h.shape[0]
    first = _one_body(v, L, [h - 0.5 * np.einsum("gij,gjk->ik", chol, chol)] + list(chol))
    out = first[0]
    for g in range(len(chol)):
        out = out + 0.5 * _one_body(first[1 + g], L, [chol[g]])[0]
    return out


def _qr(M):
    Q, R = torch.linalg.qr(M)
    d = torch.diagonal(R)
    ph = d / d.abs()
    return Q * ph[None, :], R * ph.conj()[:, None]


def _right_canonical(C):
    C = list(C)
    for i in range(len(C) - 1, 0, -1):
        a, _, b = C[i].shape
        Q, R = _qr(C[i].reshape(a, 4 * b).conj().T)
        C[i] = Q.conj().T.reshape(-1, 4, b)
        C[i - 1] = torch.tensordot(C[i - 1], R.conj().T, dims=1)
    return C


def _kept(s, D, eps):
    s = s.cpu().numpy()
    k = int(np.sum(s > 1e-12 * s[0]))
    tail = np.sum(s[k:] ** 2)
    total = np.sum(s ** 2)
    while k > 1 and tail + s[k - 1] ** 2 <= eps * total:
        k -= 1
        tail += s[k] ** 2
    k = min(k, D)
    return k, float(np.sum(s[k:] ** 2) / total)


def _right_bases(C):
    out = [None] * (len(C) + 1)
    out[len(C)] = torch.ones(1, 1, dtype=torch.complex128, device="cuda")
    for i in range(len(C) - 1, -1, -1):
        out[i] = torch.tensordot(C[i], out[i + 1], dims=1).reshape(C[i].shape[0], -1)
    return out


def _left_bases(C):
    out = [torch.ones(1, 1, dtype=torch.complex128, device="cuda")]
    for A in C:
        out.append((out[-1] @ A.reshape(A.shape[0], -1)).reshape(-1, A.shape[2]))
    return out


def _fit(T, guess, c, D, eps):
    """The variational fit of the vector T: two-site, then one-site sweeps, each
    local solution the projection of T on the current bases."""
    C = _right_canonical(guess)
    L = len(C)
    for two, count in ((True, c.get("two_site", 0)), (False, c.get("one_site", 1))):
        w = 2 if two else 1
        for _ in range(count):
            R = _right_bases(C)
            P = T.reshape(1, -1)
            for i in range(L - w + 1):
                a = P.shape[0]
                S = P.reshape(a * 4 ** w, -1) @ R[i + w].conj().T
                if two:
                    S = S.reshape(4 * a, -1)
                    U, s, V = torch.linalg.svd(S, full_matrices=False)
                    k, _ = _kept(s, D, eps)
                    C[i] = U[:, :k].reshape(a, 4, k)
                    C[i + 1] = (s[:k, None] * V[:k]).reshape(k, 4, -1)
                elif i == L - 1:
                    C[i] = S.reshape(a, 4, -1)
                    break
                else:
                    C[i] = _qr(S)[0].reshape(a, 4, -1)
                P = C[i].reshape(4 * a, -1).conj().T @ P.reshape(4 * a, -1)
            left = _left_bases(C)
            P = T.reshape(-1, 1)
            for i in range(L - w, -1, -1):
                b = P.shape[1]
                S = left[i].conj().T @ P.reshape(left[i].shape[0], -1)
                if two:
                    S = S.reshape(-1, 4 * b)
                    U, s, V = torch.linalg.svd(S, full_matrices=False)
                    k, _ = _kept(s, D, eps)
                    C[i] = (U[:, :k] * s[:k]).reshape(-1, 4, k)
                    C[i + 1] = V[:k].reshape(k, 4, b)
                    P = P.reshape(-1, 4 * b) @ C[i + 1].reshape(k, -1).conj().T
                elif i == 0:
                    C[i] = S.reshape(-1, 4, b)
                else:
                    Q = _qr(S.reshape(-1, 4 * b).conj().T)[0]
                    C[i] = Q.conj().T.reshape(-1, 4, b)
                    P = P.reshape(-1, 4 * b) @ Q
    return C


def _rdm_vector(v, L):
    low = torch.stack([_ladder(v, L, j, s, False) for s in range(2) for j in range(L)])
    low = low.reshape(2, L, -1)
    return sum(low[s].conj() @ low[s].T for s in range(2)).cpu().numpy()


def _rdm_tensors(C):
    """The one-body density matrix by transfer matrices (any length)."""
    L = len(C)
    R = [None] * L + [torch.ones(1, 1, dtype=torch.complex128, device="cuda")]
    for i in range(L - 1, -1, -1):
        X = torch.tensordot(C[i].conj(), R[i + 1], dims=1)
        R[i] = X.reshape(X.shape[0], -1) @ C[i].reshape(C[i].shape[0], -1).T
    par = torch.tensor([1, -1, -1, 1], dtype=torch.complex128, device="cuda")
    low = torch.zeros(2, 4, 4, dtype=torch.complex128, device="cuda")
    for s in range(2):
        for a, b, x in LOWER[s]:
            low[s, b, a] = x

    def step(E, op, A):   # sum conj(A)[x s p] op[s t] E[x y] A[y t q]
        X = torch.tensordot(E, A, dims=1)
        X = torch.einsum("st,cxtq->cxsq", op, X)
        return torch.einsum("xsp,cxsq->cpq", A.conj(), X)

    gam = np.zeros((L, L), dtype=np.complex128)
    one = torch.ones(1, 1, 1, dtype=torch.complex128, device="cuda")
    opened, eye = [None, None], torch.eye(4, dtype=torch.complex128, device="cuda")
    for j in range(L):
        for s in range(2):
            E = step(one, low[s].conj().T @ low[s], C[j])
            gam[j, j] += complex((E[0] * R[j + 1]).sum())
            if j:
                E = step(opened[s], low[s], C[j])
                gam[:j, j] += (E * R[j + 1][None]).sum((1, 2)).cpu().numpy()
            new = step(one, low[s].conj().T * par[None, :], C[j])
            old = step(opened[s], torch.diag(par), C[j]) if j else new[:0]
            opened[s] = torch.cat([old, new])
        one = step(one, eye, C[j])
    return gam + np.tril(gam.conj().T, -1)


def _exact_observe(C, h, chol):
    v = _vector(C)
    return dict(rdm=_rdm_vector(v, len(C)), norm=np.array([complex(torch.vdot(v, v))]),
                energy=np.array([complex(torch.vdot(v, _hamiltonian(v, h, chol)))]))


def _exact_rk4(c, psi, h, chol, dt):
    D = c["D"]
    v = _vector(psi)
    ks, at = [], psi
    for step in (0.5, 0.5, 1.0, None):
        k = _fit(-1j * dt * _hamiltonian(_vector(at), h, chol), at, c, D, 0.0)
        ks.append(_vector(k))
        if step:
            at = _fit(v + step * ks[-1], psi, c, D, 0.0)
    return _fit(v + ks[0] / 6 + ks[1] / 3 + ks[2] / 3 + ks[3] / 6, psi, c, D, 0.0)


def _exact_krylov(c, psi, h, chol, dt, eps):
    phi, vec, hv = [psi], [_vector(psi)], []
    for k in range(c["m"]):
        hv.append(_hamiltonian(vec[k], h, chol))
        if k == c["m"] - 1:
            break
        u = _fit(hv[k], phi[k], c, c["D"], eps)
        T = _vector(u)
        for x in vec:
            T = T - torch.vdot(x, hv[k]) / torch.vdot(x, x) * x
        w = _fit(T, u, c, c["D"], eps)
        w[0] = w[0] / torch.linalg.norm(w[0])
        phi.append(w)
        vec.append(_vector(w))
    N = np.array([[complex(torch.vdot(x, y)) for y in vec] for x in vec])
    H = np.array([[complex(torch.vdot(x, y)) for y in hv] for x in vec])
    H = np.triu(H) + np.triu(H, 1).conj().T
    lam, V = np.linalg.eigh(N)
    X = V[:, lam > 1e-12 * lam[-1]] / np.sqrt(lam[lam > 1e-12 * lam[-1]])
    e, U = np.linalg.eigh(X.conj().T @ H @ X)
    a = X @ (U @ (np.exp(-1j * dt * e) * (U.conj().T @ (X.conj().T @ N[:, 0]))))
    return _fit(sum(complex(a[k]) * vec[k] for k in range(c["m"])), psi, c, c["D"], eps)


def exact(case, seed):
    kind, L = case["kind"], case["L"]
    if kind not in ("overlap", "compress", "batch") and L > 12:
        return None   # 4^L amplitudes take too long
    if kind == "overlap":
        A, B = (s[0] for s in _inputs(case, seed)[0][2])
        E = _dev(np.ones((1, 1)))
        for x, y in zip(A, B):
            x, y = _dev(x), _dev(y)
            X = (E @ y.reshape(y.shape[0], -1)).reshape(-1, y.shape[2])
            E = x.reshape(-1, x.shape[2]).conj().T @ X
        return np.complex128(E[0, 0].item())
    inputs = _inputs(case, seed)
    if kind == "batch":
        return [_rdm_vector(_vector(_exact_rk4(c, [_dev(t) for t in st[0][0]], h, chol, 0.01)), c["L"])
                if c["L"] <= 10 else None for c, (h, chol, st) in zip(_items(case), inputs)]
    h, chol, st = inputs[0]
    psi = [[_dev(t) for t in s[0]] for s in st]
    if kind == "compress":
        C, lost = _right_canonical(psi[0]), 0.0
        for i in range(L - 1):
            a, _, b = C[i].shape
            U, s, V = torch.linalg.svd(C[i].reshape(4 * a, b), full_matrices=False)
            k, w = _kept(s, case["D_out"], 1e-12)
            lost += w
            C[i] = U[:, :k].reshape(a, 4, k)
            C[i + 1] = torch.tensordot(s[:k, None] * V[:k], C[i + 1], dims=1)
        return dict(lost=np.float64(lost), rdm=_rdm_tensors(C))
    if kind == "expectation":
        return np.complex128(torch.vdot(_vector(psi[0]), _hamiltonian(_vector(psi[1]), h, chol)).item())
    if kind == "gradient":
        v = _vector(psi[0])
        w = _hamiltonian(v, h, chol)
        n = torch.vdot(v, v).real
        e = torch.vdot(v, w).real / n
        T = (w - e * v) / n
        left, right = _left_bases(psi[0]), _right_bases(psi[0])
        out = [np.float64(e.item())]
        for i in range(L):
            G = left[i].conj().T @ T.reshape(left[i].shape[0], -1)
            G = G.reshape(-1, right[i + 1].shape[1]) @ right[i + 1].conj().T
            out.append(G.reshape(-1, 4, right[i + 1].shape[0]).cpu().numpy())
        return out
    if kind == "local":
        i, x = case["site"], psi[0][case["site"]]
        left, right = _left_bases(psi[0])[i], _right_bases(psi[0])[i + 1]
        for _ in range(case["reps"]):
            v = ((left @ x.reshape(x.shape[0], -1)).reshape(-1, x.shape[2]) @ right).reshape(-1)
            w = left.conj().T @ _hamiltonian(v, h, chol).reshape(left.shape[0], -1)
            x = (w.reshape(-1, right.shape[1]) @ right.conj().T).reshape(x.shape)
        return x.cpu().numpy()
    if kind == "sum":
        T = sum(k * _vector(p) for k, p in zip(_coefficients(case["terms"]), psi))
        C = _fit(T, psi[0], case, case["D"], 0.0)
        return [t.cpu().numpy() for t in C]
    if kind == "apply":
        C = _fit(-1j * DT * _hamiltonian(_vector(psi[0]), h, chol), psi[0], case, case["D"], 0.0)
        out = [t.cpu().numpy() for t in C]
        if case["prec"] == "bf16":
            out = [np.ascontiguousarray(t).view(np.float64).reshape(*t.shape, 2) for t in out]
        return out
    if kind == "rk4":
        return _exact_observe(_exact_rk4(case, psi[0], h, chol, 0.01), h, chol)
    return _exact_observe(_exact_krylov(case, psi[0], h, chol, DT, 1e-8), h, chol)
