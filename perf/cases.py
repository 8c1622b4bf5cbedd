"""The work that a user of the library has it do, as cases that can be timed and compared.

Sizes are those of the package's own workloads (`paper_2410_04204_gb300/inputs.py`), its tests
and its benchmark: the critical chain h_z = 1 with a weak longitudinal field (L = 24 with every
momentum sector, L = 40 S(k = 0, w), L = 60 overlap-ordered quench, L = 80 energy-ordered quench
with many variants), and complete small chains at any h_z.  A seed chooses the fields (h_x; on the
chains truncated by quasiparticle number only, whose sizes do not depend on it, also h_z), which
are what a user scans.  The longest workloads of the benchmark are cut by their energy cutoff so
that one pass stays below two seconds.

Kinds of cases:
  heff      contraction table, Pfaffians and the complex H_eff (tgba_compute_x, tgba_assemble_heff)
  spectrum  contraction table, Pfaffians and all eigenvalues for several h_x (tgba_eigvals)
  dsf       S(k = 0, w) and the lowest levels at a new h_x, X kept (tgba_dsf)
  dsf_k     S(k, w) at a finite momentum (tgba_dsf_k)
  quench    the quench from its eigenpairs: nested overlap-ordered truncations, Eq. 11 metric
  variants  the quench of many (h_x, cutoff) variants at once (Chebyshev propagation)
  corr      the quench's equal-time correlators (tgba_quench_correlators)
  train     one batch of the screening network's training: loss and gradient (FP32)
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2410_04204_gb300 import tgba


# ---------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: a first look at a short chain, where launches and latency are the cost
        dict(name="heff_L12_M4", kind="heff", L=12, mq=4, e_cut=-1.0, sectors="0"),
        # H_eff of every momentum sector of the L = 24 chain (to be handed to another solver)
        dict(name="heff_L24_sectors", kind="heff", L=24, mq=6, e_cut=11.925, sectors="all"),
        # one large sector with many quasiparticles: Pfaffians of every size up to 20
        dict(name="heff_L80_M10", kind="heff", L=80, mq=10, e_cut=5.5, sectors="0"),
        # exact spectrum of a complete short chain: one small matrix, as in a convergence check
        dict(name="spectrum_L12_full", kind="spectrum", L=12, mq=12, e_cut=-1.0, sectors="0", fields=1),
        # the benchmark's step: every sector, two fields
        dict(name="spectrum_L24_sectors", kind="spectrum", L=24, mq=6, e_cut=11.925, sectors="all", fields=2),
        # all levels of one sector of a longer chain: a single mid-sized matrix
        dict(name="spectrum_L40_k0", kind="spectrum", L=40, mq=6, e_cut=8.5, sectors="0", fields=1),
        # dynamic structure factor at k = 0, the L = 40 grid
        dict(name="dsf_L40_k0", kind="dsf", L=40, mq=6, e_cut=8.5, n_w=4096, w_max=10.0, eta=0.01),
        # dynamic structure factor at a finite momentum of the L = 24 chain
        dict(name="dsf_k_L24", kind="dsf_k", L=24, mq=6, e_cut=11.925, m=5, n_w=1024, w_max=8.0, eta=0.05),
        # the paper's quench with overlap-ordered nested truncations and their convergence metric
        dict(name="quench_L60_overlap", kind="quench", L=60, mq=6, e_cut=6.5, sizes="1000,1500,2000", order=1,
             t_max=480.0, n_t=4801),
        # a scan of fields and nested cutoffs on the L = 80 chain, propagated together
        dict(name="variants_L80", kind="variants", L=80, mq=10, e_cut=5.5, cuts="4.0,4.5,5.0,-1", fields=4,
             t_max=100.0, n_t=2000),
        # equal-time correlators after the quench, a light-cone plot
        dict(name="corr_L60", kind="corr", L=60, mq=4, e_cut=6.0, chi=101, order=1, j_max=8, t_max=20.0, n_t=201),
        # one batch of the screener's training, the batch size that tgba_screen_train uses
        dict(name="train_B4096", kind="train", batch=4096),
    ]


def draw(rng):
    kind = rng.choice(["heff", "heff", "spectrum", "spectrum", "dsf", "dsf_k", "quench", "variants", "corr", "train"])
    e = lambda lo, hi: round(rng.uniform(lo, hi), 4)  # the state count grows exponentially with the cutoff  # noqa: E731
    if kind in ("heff", "spectrum"):
        c = rng.choice([
            lambda: dict(L=rng.choice([8, 10, 12, 14]), mq=rng.choice([4, 6, 8, 10]), e_cut=-1.0, sectors=rng.choice(["0", "all"])),
            lambda: dict(L=24, mq=6, e_cut=e(8.0, 11.5), sectors="all"),
            lambda: dict(L=rng.choice([30, 32, 34]), mq=6, e_cut=e(6.5, 9.0), sectors="0,%d,%d" % (rng.randint(1, 7), rng.randint(8, 15))),
            lambda: dict(L=40, mq=6, e_cut=e(6.0, 8.5), sectors="0"),
            lambda: dict(L=60, mq=6, e_cut=e(4.5, 6.0), sectors="0"),
            lambda: dict(L=80, mq=10, e_cut=e(3.5, 5.5 if kind == "heff" else 4.4), sectors="0")])()
        if kind == "spectrum":
            c["fields"] = rng.choice([1, 2]) if c["sectors"] == "all" else rng.choice([1, 2, 3])
        return dict(kind=kind, **c)
    if kind == "dsf":
        L, lo, hi = rng.choice([(24, 8.0, 11.9), (40, 6.0, 8.4), (60, 4.5, 5.9)])
        return dict(kind=kind, L=L, mq=6, e_cut=e(lo, hi), n_w=rng.choice([257, 1000, 1024, 4096, 10001]), w_max=e(4.0, 10.0),
                    eta=rng.choice([0.01, 0.02, 0.05]))
    if kind == "dsf_k":
        L, lo, hi = rng.choice([(20, 10.0, 14.0), (24, 8.0, 11.9), (32, 7.0, 9.0)])
        return dict(kind=kind, L=L, mq=6, e_cut=e(lo, hi), m=rng.randint(1, L - 1), n_w=rng.choice([257, 1000, 1024, 4096]),
                    w_max=e(4.0, 10.0), eta=rng.choice([0.02, 0.05]))
    if kind == "quench":
        L, ec = rng.choice([(40, 8.5), (60, 6.0)])
        lo = rng.randint(50, 900)
        sizes = [lo] + [int(lo * f) for f in (1.5, 2.0)[: rng.randint(0, 2)]]
        return dict(kind=kind, L=L, mq=6, e_cut=ec, sizes=",".join(map(str, sizes)), order=1, t_max=e(10.0, 480.0),
                    n_t=rng.choice([201, 500, 1001, 4801]))
    if kind == "variants":
        top = e(4.0, 5.4)
        cuts = ["%.4f" % (top - d) for d in (1.0, 0.5)[rng.randint(0, 2):]] + ["-1"]
        return dict(kind=kind, L=80, mq=10, e_cut=top, cuts=",".join(cuts), fields=rng.randint(1, 4), t_max=e(10.0, 100.0),
                    n_t=rng.choice([101, 500, 1001, 2000]))
    if kind == "corr":
        L, ec = rng.choice([(24, 8.0), (40, 6.0), (60, 5.0)])
        return dict(kind=kind, L=L, mq=4, e_cut=ec, chi=rng.randint(11, 100), order=1, j_max=rng.randint(1, 8),
                    t_max=e(5.0, 40.0), n_t=rng.choice([33, 101, 201]))
    return dict(kind="train", batch=int(round(math.exp(rng.uniform(math.log(60), math.log(16000))))))


# ---------------------------------------------------------------------------------- inputs
H_Z0 = 0.5       # the quench starts from the ground states of the chain at this field


class Basis:
    """A basis handle that is given back with the object."""

    def __init__(self, case, sectors, h_z):
        self.h = tgba.tgba_build_basis(case["L"], h_z, sectors, case["mq"], case["e_cut"])

    def __del__(self):
        tgba.tgba_basis_free(self.h)


class Screener:
    def __init__(self, params):
        self.h = tgba.tgba_screen_create(256, params)

    def __del__(self):
        tgba.tgba_screen_free(self.h)


def _fields(case, seed):
    """The fields that the seed chooses: (h_z, list of h_x)."""
    g = np.random.default_rng([2410, int(seed)])
    h_z = float(g.uniform(0.6, 1.4)) if case["e_cut"] < 0 else 1.0     # an energy cutoff is made for h_z = 1
    n = int(case.get("fields", 1))
    return h_z, [float(x) for x in np.sort(g.uniform(0.025, 0.2, n))]


def _sector_list(case):
    kind = case["kind"]
    if kind in ("heff", "spectrum"):
        return list(range(case["L"])) if case["sectors"] == "all" else [int(x) for x in case["sectors"].split(",")]
    return [0, case["m"]] if kind == "dsf_k" else [0]


def _variants(case, hx):
    cuts = [float(x) for x in case["cuts"].split(",")]
    return [h for _ in cuts for h in hx], [c for c in cuts for _ in hx]


def _train_inputs(case, seed):
    g = np.random.default_rng([2411, int(seed)])
    B, L = case["batch"], 24
    x = np.zeros((B, 20), np.float32)
    for p, M in ((0, g.choice([2, 4, 6], B)), (8, g.choice([2, 4, 6], B))):
        k = np.sort(g.integers(-L // 2, L // 2, (B, 8)) * 2 + 1 - p // 8, axis=1) / L
        x[:, p:p + 8] = np.where(np.arange(8)[None, :] < M[:, None], k, 0.0)
        x[:, 16 + p // 8] = M / 8
    x[:, 18] = 24.0 / L
    x[:, 19] = 1.0
    # parameters in the library's flat order (W1, b1, W2, b2, w3, b3), He-normal as at the start of a training
    params = np.concatenate([g.standard_normal(256 * 20) * math.sqrt(2 / 20), g.standard_normal(256) * 0.01,
                             g.standard_normal(256 * 256) * math.sqrt(2 / 256), g.standard_normal(256) * 0.01,
                             g.standard_normal(256) * math.sqrt(2 / 256), [-3.0]]).astype(np.float32)
    return x, g.uniform(-6.0, -1.0, B).astype(np.float32), params


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t, params = _train_inputs(case, seed)
        s = Screener(params)
        n = tgba.tgba_screen_nparams(s.h)
        return dict(case=case, s=s, x=torch.from_numpy(x).cuda(), t=torch.from_numpy(t).cuda(),
                    grad=torch.empty(n, dtype=torch.float32, device="cuda"))
    h_z, hx = _fields(case, seed)
    b = Basis(case, _sector_list(case), h_z)
    st = dict(case=case, b=b, hx=hx)
    f64 = functools.partial(torch.empty, dtype=torch.float64, device="cuda")
    sizes = tgba.tgba_sector_sizes(b.h)
    n_states = sum(x + y for x, y in sizes)
    if kind == "heff":
        st["H"] = torch.empty(tgba.tgba_basis_totals(b.h)[2], dtype=torch.complex128, device="cuda")
    elif kind == "spectrum":
        st["ev"] = f64(len(hx) * n_states)
    else:
        tgba.tgba_compute_x(b.h)          # X is kept while the longitudinal field is scanned
        if kind in ("dsf", "dsf_k"):
            st["S"] = torch.empty(case["n_w"], dtype=torch.float32, device="cuda")
            st["n_ev"] = min(40, sum(sizes[-1]))
            st["ev"] = f64(st["n_ev"])
        elif kind == "quench":
            st["sizes"] = [int(x) for x in case["sizes"].split(",")]
            nv = len(st["sizes"])
            st.update(mx=f64(nv, case["n_t"]), norm=f64(nv), eps=f64(max(1, nv - 1)))
        elif kind == "variants":
            st["vhx"], st["vcut"] = _variants(case, hx)
            nv = len(st["vhx"])
            st.update(mx=f64(nv, case["n_t"]), norm=f64(nv))
        else:
            st.update(mx=f64(case["n_t"]), corr=f64(case["j_max"], case["n_t"]), norm=f64(1))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "train":
        loss = tgba.tgba_screen_grad(st["s"].h, st["x"], st["t"], st["grad"])
        return [st["grad"], loss]
    b, hx = st["b"].h, st["hx"]
    if kind == "heff":
        tgba.tgba_compute_x(b)
        tgba.tgba_assemble_heff(b, hx[0], st["H"])
        return [st["H"]]
    if kind == "spectrum":
        tgba.tgba_compute_x(b)
        tgba.tgba_eigvals(b, hx, st["ev"])
        return list(st["ev"].view(len(hx), -1))
    if kind == "dsf":
        tgba.tgba_dsf(b, 0, hx[0], 0.0, case["w_max"], case["n_w"], case["eta"], st["S"], st["ev"], st["n_ev"])
        return [st["S"], st["ev"]]
    if kind == "dsf_k":
        tgba.tgba_dsf_k(b, 1, 0, hx[0], 0.0, case["w_max"], case["n_w"], case["eta"], st["S"], st["ev"], st["n_ev"])
        return [st["S"], st["ev"]]
    if kind == "quench":
        nv = len(st["sizes"])
        eps = st["eps"] if nv > 1 else None
        tgba.tgba_quench_ordered(b, 0, H_Z0, hx * nv, st["sizes"], case["order"], case["t_max"], case["n_t"], st["mx"],
                                 st["norm"], eps)
        return [st["mx"], st["norm"]] + ([eps] if nv > 1 else [])
    if kind == "variants":
        tgba.tgba_quench(b, 0, H_Z0, st["vhx"], st["vcut"], case["t_max"], case["n_t"], st["mx"], st["norm"], method=2)
        return list(st["mx"]) + [st["norm"]]
    tgba.tgba_quench_correlators(b, 0, H_Z0, hx[0], case["chi"], case["order"], case["t_max"], case["n_t"], case["j_max"],
                                 st["mx"], st["corr"], st["norm"])
    return [st["mx"], st["corr"], st["norm"]]


# ------------------------------------------------------- the method in plain numpy and torch
# (C.f. Eq. 6-7, S1-S4, S6.)  Parity 0: NS, 1: R; mode labels n with k = pi n / L, ascending.
def _modes(L, par, h):
    n = [(-(L - 1) if par == 0 else -(L - 2)) + 2 * i for i in range(L)]
    eps, th, ex = [], [], []
    for q in n:
        if q == L:
            eps.append(2.0 * (h - 1.0)); th.append(0.0); ex.append(-eps[-1])
            continue
        k = math.pi * q / L
        c = math.cos(0.5 * k)
        eps.append(2.0 * math.sqrt((h - 1.0) * (h - 1.0) + 4.0 * h * c * c))
        th.append(0.0 if q == 0 else math.copysign(math.acos(min(1.0, max(-1.0, 2.0 * (h + math.cos(k)) / eps[-1]))), k))
        ex.append(eps[-1])
    e_vac, norm = 0.0, 1.0
    for q, e, t in zip(n, eps, th):
        e_vac += e if q != L else 0.0
        norm /= math.cos(0.5 * t) if 0 < q < L else 1.0
    e_vac = -0.5 * e_vac + (0.5 * eps[-1] if par else 0.0)
    return np.array(n), np.array(ex), np.array(th), e_vac, norm


@functools.lru_cache(maxsize=8)
def _parity_states(L, par, h, mq, e_cut):
    """All states below the cutoff, of every sector: [(sector m, E, modes [count][M])] per M."""
    n, ex, _, e_vac, _ = _modes(L, par, h)
    cut = _modes(L, 0, h)[3] + e_cut + 1e-9 if e_cut >= 0 else math.inf
    neg = float(np.minimum(0.0, ex).sum())
    md, E, out = np.zeros((1, 0), np.int16), np.zeros(1), []
    for M in range(mq + 1):
        if M % 2 == 0:
            s = np.sort(ex[md], axis=1)
            e = np.zeros(len(md))
            for q in range(M):
                e = e + s[:, q]
            e = e_vac + e
            keep = e <= cut
            out.append((n[md[keep]].sum(axis=1) % (2 * L) // 2, e[keep], md[keep]))
        last = md[:, -1] if M else np.full(len(md), -1)
        nmd, nE = [], []
        for i in range(L):
            k = (last < i) & (E + ex[i] + e_vac + neg <= cut + 1e-6)
            if k.any():
                nmd.append(np.concatenate([md[k], np.full((int(k.sum()), 1), i, np.int16)], axis=1))
                nE.append(E[k] + ex[i])
        if not nmd:
            break
        md, E = np.concatenate(nmd), np.concatenate(nE)
    return out


def _sector(case, h, m):
    """States of sector m in basis order, per parity: [(M, E, modes)] groups."""
    res = []
    for par in (0, 1):
        groups = []
        for sec, E, md in _parity_states(case["L"], par, h, case["mq"], case["e_cut"]):
            k = sec == m
            if k.any():
                e, q = E[k], md[k]
                o = np.lexsort(tuple(q[:, j] for j in reversed(range(q.shape[1]))) + (e,))
                groups.append((md.shape[1], e[o], q[o]))
        res.append(groups)
    return res


def _pf(A):
    """Pfaffian of one complex skew matrix."""
    A, n, v = A.copy(), len(A), 1.0 + 0.0j
    for k in range(0, n, 2):
        p = k + 1 + int(np.argmax(np.abs(A[k + 1:, k])))
        if p != k + 1:
            A[[k + 1, p]] = A[[p, k + 1]]
            A[:, [k + 1, p]] = A[:, [p, k + 1]]
            v = -v
        v *= A[k, k + 1]
        if k + 2 < n:
            t, r = A[k, k + 2:] / A[k, k + 1], A[k + 1, k + 2:]
            A[k + 2:, k + 2:] += np.outer(r, t) - np.outer(t, r)
    return v


@functools.lru_cache(maxsize=4)
def _table(L, h):
    """(C0, R): X_ab = C0 (-i)^{n/2} Pf(R[sel]) with sel = (NS mode i: row L - 1 - i, descending) ++
    (R mode i: row L + i, ascending); the Schur complement of both vacua and sigma^x_1."""
    (n0, _, t0, _, w0), (n1, _, t1, _, w1) = _modes(L, 0, h), _modes(L, 1, h)
    j = np.arange(1, L + 1)
    plane = lambda n, s: np.exp(1j * s * math.pi * n * j / L) / math.sqrt(L)  # noqa: E731
    dag = lambda n, t: (math.sin(t / 2) * plane(n, 1), 1j * math.cos(t / 2) * plane(n, 1))  # (U, V) of d_k^dag  # noqa: E731
    ann = lambda n, t: (-1j * math.cos(t / 2) * plane(n, -1), math.sin(t / 2) * plane(n, -1))  # of d_k  # noqa: E731
    e1, zero = (j == 1).astype(complex), np.zeros(L, complex)
    string = [(0, dag(n0[i], t0[i])) for i in range(L)]
    string += [(1, ann(n0[i], t0[i])) for i in reversed(range(L))]
    string += [(0, (e1, e1))]
    string += [(1, (plane(n1[i], 1), zero) if n1[i] == L else dag(n1[i], t1[i])) for i in range(L)]
    string += [(0, ann(n1[i], t1[i])) for i in reversed(range(L - 1))]
    U, V = (np.array([s[1][q] for s in string]) for q in (0, 1))
    A = np.triu(V @ U.T, 1)
    A = A - A.T
    E = np.array([s[0] for s in string], bool)
    F = ~E
    S = A[np.ix_(E, E)] + A[np.ix_(F, E)].T @ np.linalg.solve(A[np.ix_(F, F)], A[np.ix_(F, E)])
    k = math.pi * np.concatenate([n0[::-1], -n1]) / L
    R = (1j * np.exp(1j * (k[:, None] + k[None, :])) * S).real
    return w0 * w1 * _pf(A[np.ix_(F, F)]), R - np.diag(np.diag(R))


def _pf_batch(A):
    """Pfaffians of real skew matrices [batch][n][n] (destroyed)."""
    B, n, _ = A.shape
    v = torch.ones(B, dtype=A.dtype, device=A.device)
    rows = torch.arange(B, device=A.device)
    for k in range(0, n, 2):
        p = k + 1 + A[:, k, k + 1:].abs().argmax(dim=1)
        r = A[:, k + 1].clone()
        A[:, k + 1] = A[rows, p]
        A[rows, p] = r
        c = A[:, :, k + 1].clone()
        A[:, :, k + 1] = A[rows, :, p]
        A[rows, :, p] = c
        a = A[:, k, k + 1].clone()
        v = torch.where(p != k + 1, -v, v) * a
        if k + 2 < n:
            t = A[:, k, k + 2:] / torch.where(a == 0, torch.ones_like(a), a)[:, None]
            r = A[:, k + 1, k + 2:]
            o = r[:, :, None] * t[:, None, :]
            A[:, k + 2:, k + 2:] += o - o.transpose(1, 2)
    return v


def _x_real(L, h, ns, r):
    """P_ab over two group lists, on the GPU: X_ab = C0 (-i)^{(M_a + M_b)/2} P_ab."""
    R = torch.from_numpy(_table(L, h)[1]).cuda()
    P = torch.empty(sum(len(g[1]) for g in ns), sum(len(g[1]) for g in r), dtype=torch.float64, device="cuda")
    i0 = 0
    for Ma, _, qa in ns:
        sa = torch.from_numpy((L - 1 - qa[:, ::-1].astype(np.int64)).copy()).cuda()
        j0 = 0
        for Mb, _, qb in r:
            sb = torch.from_numpy(L + qb.astype(np.int64)).cuda()
            na, nb, n = len(sa), len(sb), Ma + Mb
            step = max(1, int(2.5e8 / (max(1, n * n) * nb)))
            for i in range(0, na if n else 0, step):
                c = min(step, na - i)
                sel = torch.cat([sa[i:i + c, None, :].expand(c, nb, Ma), sb[None].expand(c, nb, Mb)], 2).reshape(c * nb, n)
                P[i0 + i:i0 + i + c, j0:j0 + nb] = _pf_batch(R[sel[:, :, None], sel[:, None, :]]).view(c, nb)
            if n == 0:
                P[i0:i0 + na, j0:j0 + nb] = 1.0
            j0 += nb
        i0 += len(sa)
    return P


def _energies(groups):
    return np.concatenate([g[1] for g in groups]) if groups else np.zeros(0)


def _count(groups):
    return sum(len(g[1]) for g in groups)


def _h_real(L, c0, h_x, E, P):
    """H_eff in the real gauge: diag(E) with the off-diagonal block -L h_x |C0| P."""
    H = torch.diag(torch.from_numpy(E).cuda())
    a = P.shape[0]
    H[:a, a:] = -L * h_x * abs(c0) * P
    H[a:, :a] = H[:a, a:].T
    return H


def _lorentz(case, w, dE):
    om = torch.linspace(0.0, 1.0, case["n_w"], dtype=torch.float64, device="cuda") * case["w_max"]
    S = torch.empty_like(om)
    for i in range(0, len(om), 512):
        S[i:i + 512] = (2.0 * case["eta"] / ((om[i:i + 512, None] - dE) ** 2 + case["eta"] ** 2)) @ w
    return S


def _overlaps(L, h, sec):
    """c~0 = conj(gauge) <phi|Phi0> (Eq. S6) of all states: complex, NS then R."""
    z, c0 = _table(L, H_Z0)[0], _table(L, h)[0]
    out = []
    for par in (0, 1):
        n, _, th, _, _ = _modes(L, par, h)
        d = th - _modes(L, par, H_Z0)[2]
        base = np.prod(np.cos(0.5 * d[(n > 0) & (n < L)])) * math.sqrt(0.5)
        for M, _, q in sec[par]:
            nq = n[q]
            ok = np.all(nq == -nq[:, ::-1], axis=1) & np.all((nq != 0) & (nq != L), axis=1)
            v = base * np.where(ok, np.prod(np.tan(0.5 * d[q[:, M // 2:]]), axis=1), 0.0)
            out.append((v * (-1.0) ** (M // 2)).astype(complex) if par == 0 else v * (np.conj(z) / abs(z)) * (c0 / abs(c0)))
    return np.concatenate(out)


def _evolve(L, h, h_x, E, P, c, t):
    """(<sigma^x>(t), ||c||^2, B(t)) from the eigenpairs of the kept states (NS then R)."""
    c0 = _table(L, h)[0]
    ev, U = torch.linalg.eigh(_h_real(L, c0, h_x, E, P))
    a, kn = U.T.to(torch.complex128) @ torch.from_numpy(c).cuda(), P.shape[0]
    t = torch.from_numpy(t).cuda()
    ph = torch.exp(-1j * ev[:, None] * t[None, :]) * a[:, None]
    B = torch.complex(U @ ph.real, U @ ph.imag)
    norm = float(np.vdot(c, c).real)
    X = abs(c0) * P
    Br = B[kn:]
    XB = torch.complex(X @ Br.real, X @ Br.imag)
    return 2.0 * (B[:kn].conj() * XB).real.sum(0) / norm, norm, B


def _rank(case, h, sec, c):
    """Order of the sector's states by |<phi|Phi0>| (largest first), ties by energy and labels."""
    E = np.concatenate([_energies(sec[0]), _energies(sec[1])])
    e0 = _modes(case["L"], 0, h)[3]
    labels = [(par, M, tuple(q)) for par in (0, 1) for M, _, md in sec[par] for q in md.tolist()]
    a = [-int(round(x * 1e10)) for x in np.abs(c)]
    return sorted(range(len(E)), key=lambda i: (a[i], int(round((E[i] - e0) * 1e9))) + labels[i]), E


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    L = case["L"]
    h, hx = _fields(case, seed)
    c0 = _table(L, h)[0]
    secs = [_sector(case, h, m) for m in _sector_list(case)]
    E = [np.concatenate([_energies(s[0]), _energies(s[1])]) for s in secs]
    if kind == "heff":
        out = []
        for s, e in zip(secs, E):
            P = _x_real(L, h, *s)
            ph = [np.concatenate([np.full(len(g[1]), (-1j) ** (g[0] // 2)) for g in p]) if p else np.zeros(0, complex) for p in s]
            X = -L * hx[0] * c0 * torch.from_numpy(ph[0]).cuda()[:, None] * torch.from_numpy(ph[1]).cuda()[None, :] * P
            H = torch.diag(torch.from_numpy(e).cuda().to(torch.complex128))
            a = X.shape[0]
            H[:a, a:] = X
            H[a:, :a] = X.conj().T
            out.append(H.T.reshape(-1))              # column-major
        return [torch.cat(out)]
    if kind == "spectrum":
        if sum(len(e) ** 3 for e in E) > 2.5e11:
            return None
        ev = torch.cat([torch.linalg.eigvalsh(_h_real(L, c0, hx[0], e, _x_real(L, h, *s))) for s, e in zip(secs, E)])
        return [ev] + [None] * (len(hx) - 1)         # one of the fields: the others take as long again
    if kind in ("dsf", "dsf_k"):
        P = _x_real(L, h, *secs[0])
        ev, U = torch.linalg.eigh(_h_real(L, c0, hx[0], E[0], P))
        u0, e0, a = U[:, 0], ev[0], P.shape[0]
        v = abs(c0) * torch.cat([P @ u0[a:], P.T @ u0[:a]])
        if kind == "dsf_k":
            del U
            (ns0, r0), (nsk, rk) = secs
            ev, U = torch.linalg.eigh(_h_real(L, c0, hx[0], E[1], _x_real(L, h, nsk, rk)))
            v = abs(c0) * torch.cat([_x_real(L, h, nsk, r0) @ u0[a:], _x_real(L, h, ns0, rk).T @ u0[:a]])
        return [_lorentz(case, L * (U.T @ v) ** 2, ev - e0), ev[:min(40, len(ev))]]
    sec, E = secs[0], E[0]
    c = _overlaps(L, h, sec)
    t = case["t_max"] * np.arange(case["n_t"]) / max(1, case["n_t"] - 1)
    n_ns = _count(sec[0])
    if kind == "variants":
        out, norms = [], []
        P, e_ns = _x_real(L, h, *sec), _modes(L, 0, h)[3]
        for f, cut in zip(*_variants(case, hx)):
            keep = np.flatnonzero(E <= (e_ns + cut) + 1e-9) if cut >= 0 else np.arange(len(E))
            kn, kr = keep[keep < n_ns], keep[keep >= n_ns] - n_ns
            norms.append(float(np.vdot(c[keep], c[keep]).real))
            small = len(keep) <= 3200 and len([x for x in out if x is not None]) < 4
            out.append(_evolve(L, h, f, E[keep], P[kn][:, kr], c[keep], t)[0] if small else None)
        return out + [torch.tensor(norms, dtype=torch.float64)]
    rank, _ = _rank(case, h, sec, c)
    sizes = [int(x) for x in case["sizes"].split(",")] if kind == "quench" else [case["chi"]]
    mx, norms, eps, prev = [], [], [], None
    P = _x_real(L, h, *sec)
    for chi in sizes:
        kn = [q for q in rank[:chi] if q < n_ns]
        kr = [q for q in rank[:chi] if q >= n_ns]
        m, nrm, B = _evolve(L, h, hx[0], E[kn + kr], P[kn][:, [q - n_ns for q in kr]], c[kn + kr], t)
        mx.append(m)
        norms.append(nrm)
        full = dict(zip(kn + kr, range(len(kn) + len(kr))))
        if prev is not None:
            sub = [full[q] for q in prev[0]]
            rest = torch.ones(len(full), dtype=torch.bool, device="cuda")
            rest[sub] = False
            d = (B[sub] - prev[1]).abs().square().sum(0) + B[rest].abs().square().sum(0)
            eps.append(float(d.sqrt().max()))
        prev = (kn + kr, B)
    if kind == "corr":
        return [mx[0], None, torch.tensor(norms, dtype=torch.float64)]
    return [torch.stack(mx), torch.tensor(norms, dtype=torch.float64)] + ([torch.tensor(eps, dtype=torch.float64)] if eps else [])


def _exact_train(case, seed):
    x, t, params = _train_inputs(case, seed)
    theta = torch.from_numpy(params).double().requires_grad_()
    W1, b1, W2, b2, w3, b3 = torch.split(theta, [256 * 20, 256, 256 * 256, 256, 256, 1])
    x, t = torch.from_numpy(x).double(), torch.from_numpy(t).double()
    y = torch.relu(torch.relu(x @ W1.view(256, 20).T + b1) @ W2.view(256, 256).T + b2) @ w3 + b3
    loss = ((y - t) ** 2).mean()
    loss.backward()
    return [theta.grad, float(loss)]


# ---------------------------------------------------------------------------------- least work
def _f(n):
    """Flops of one real Pfaffian by Parlett-Reid elimination."""
    return sum(2 * m * (m - 1) + m for m in range(n - 2, 0, -2))


def _pf_flops(ns, r):
    return sum(len(a[1]) * len(b[1]) * _f(a[0] + b[0]) for a, b in itertools.product(ns, r))


def work(case):
    """Inputs read once, outputs written once, and the flops of the dense method (Pfaffians by
    elimination, 4 n^3 / 3 for the spectrum of an n x n matrix, products of the propagation)."""
    kind = case["kind"]
    if kind == "train":
        B = case["batch"]
        n = 256 * 20 + 256 + 256 * 256 + 256 + 256 + 1
        return {"bytes": 4.0 * (B * 21 + 2 * n), "flops": 6.0 * B * n}
    L, nf = case["L"], int(case.get("fields", 1))
    h = _fields(case, 0)[0]
    secs = [_sector(case, h, m) for m in _sector_list(case)]
    cnt = [(_count(s[0]), _count(s[1])) for s in secs]
    n = [a + b for a, b in cnt]
    state = 9.0 + 3 * case["mq"]                    # energy, M, mode indices and table rows of a state
    x_bytes = 8.0 * sum(a * b for a, b in cnt)
    pf = float(sum(_pf_flops(*s) for s in secs))
    if kind == "heff":
        return {"bytes": state * sum(n) + 16.0 * sum(x * x for x in n), "flops": pf}
    if kind == "spectrum":
        return {"bytes": state * sum(n) + 8.0 * nf * sum(n), "flops": pf + nf * sum(4.0 * x ** 3 / 3.0 for x in n)}
    if kind == "dsf":
        return {"bytes": x_bytes + 8.0 * n[0] + 4.0 * case["n_w"], "flops": 4.0 * n[0] ** 3 / 3 + 5.0 * n[0] * case["n_w"]}
    if kind == "dsf_k":
        return {"bytes": x_bytes + 8.0 * sum(n) + 4.0 * case["n_w"],
                "flops": sum(4.0 * x ** 3 / 3 for x in n) + 5.0 * n[1] * case["n_w"]}
    if kind == "variants":
        R, K = 0.55 * case["e_cut"], 0
        K = R * case["t_max"] + 30
        e0 = _modes(L, 0, h)[3]
        fl = 0.0
        for cut in [float(x) for x in case["cuts"].split(",")]:
            k = [int((_energies(p) <= (e0 + cut if cut >= 0 else math.inf) + 1e-9).sum()) for p in secs[0]]
            fl += 8.0 * K * k[0] * k[1] * nf
        return {"bytes": x_bytes + 8.0 * nf * len(case["cuts"].split(",")) * case["n_t"], "flops": fl}
    if kind == "quench":
        sizes = [int(x) for x in case["sizes"].split(",")]
        return {"bytes": 8.0 * (max(sizes) ** 2 / 4 + len(sizes) * case["n_t"]),
                "flops": sum(4.0 * x ** 3 / 3 + 6.0 * x * x * case["n_t"] for x in sizes)}
    chi = case["chi"]
    size = 4 + 2 * case["j_max"]
    return {"bytes": 8.0 * (chi * chi / 4 + (1 + case["j_max"]) * case["n_t"]),
            "flops": 4.0 * chi ** 3 / 3 + case["j_max"] * chi * chi * (2.0 * _f(size) + 4.0 * case["n_t"])}
