"""Workloads of the variational-embedding solver that its speed and accuracy are followed on.

Every case is one call sequence a program makes through paper_2106_02682_gb300.ve:

  sweep      resume a translation-invariant instance from a checkpoint in host memory, advance it,
             take the new checkpoint: ve_set_state, ve_iterate, ve_get_state (long solves, warm
             starts and certification runs are strings of these).
  batch      the same for several instances advanced together (parameter scans, the training
             solves of the learned warm start): ve_batch_iterate.
  general    the same for the solver without translation invariance (disordered spin chains) and
             for spinless fermions: ve_general_iterate.
  bound      the certificate of a state a solve has reached: ve_bound.
  circulant  the X step alone on device memory, as a library call: ve_circulant_project.

Checkpoints are taken from the handle after `start` sweeps from the cold start, so the sweeps of a
pass are those of the middle of a solve.  A case's field, anisotropy or disorder comes from the
seed.  In the mixed precision the sweeps before convergence are float32 arithmetic; a program keeps
such a checkpoint as float32, so those passes return the state in float32.
"""
import math

import numpy as np
import torch

from paper_2106_02682_gb300 import ve

PREC = {"fp64": ve.VE_PREC_FP64, "mixed": ve.VE_PREC_MIXED, "df64": ve.VE_PREC_DF64}
MU, NU, EPS = 10.0, 10.0, 2.0   # the defaults of ve_default_options, which every case takes


# ---- the cases -----------------------------------------------------------------------------------

def _sweep(model, lx, ly, cx, cy, precision, start, sweeps, name=None):
    c = dict(kind="sweep", model=model, lx=lx, ly=ly, cx=cx, cy=cy, precision=precision,
             start=start, sweeps=sweeps)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest solve a user runs (and the first one anybody tries): 16 spins, one a cluster
        _sweep("tfim", 16, 0, 1, 1, "fp64", 40, 50, "chain16_D4_fp64"),
        # the 100-spin, 2-spin-cluster instance of the paper's tables, plain float64
        _sweep("tfim", 100, 0, 2, 1, "fp64", 40, 20, "chain100_D16_fp64"),
        # the long chain of the headline benchmark (4096 wavevectors), plain float64
        _sweep("tfim", 8192, 0, 2, 1, "fp64", 40, 20, "chain8192_D16_fp64"),
        # the same chain in the mixed precision, as a solve to a given tolerance runs it first
        _sweep("tfim", 8192, 0, 2, 1, "mixed", 40, 40, "chain8192_D16_mixed"),
        # a two-dimensional lattice in 2 x 1 clusters, double-float: what mixed solves finish in
        _sweep("tfim", 64, 64, 2, 1, "df64", 40, 20, "square64_D16_df64"),
        # 3-spin clusters on an XXZ chain (64 x 64 marginals), a ragged cluster count, float64
        _sweep("xxz", 510, 0, 3, 1, "fp64", 10, 6, "chain510_D64_fp64"),
        # the tightest relaxation: 4-spin clusters (256 x 256 marginals), 4096 spins, mixed
        _sweep("tfim", 4096, 0, 4, 1, "mixed", 10, 8, "chain4096_D256_mixed"),
        # a scan of small instances of several lengths, fields and cluster sizes in one batch
        dict(kind="batch", count=16, length=256, precision="mixed", start=40, sweeps=40,
             name="batch16_mixed"),
        # a disordered chain with all-to-all couplings: 8128 pairs, X of 512 x 512
        dict(kind="general", model="tfim", spins=128, cluster=1, start=6, sweeps=4,
             name="disordered128_X512"),
        # the paper's long-range fermion ring: 45 pairs of 16 x 16, X of 160 x 160
        dict(kind="general", model="fermion", spins=20, cluster=2, start=20, sweeps=20,
             name="fermions20_X160"),
        # the certificate of the long chain, taken every hundred sweeps of a certification run
        dict(kind="bound", model="tfim", lx=8192, ly=0, cx=2, cy=1, start=40, name="bound8192_D16"),
        # the X step as a library call on a ragged two-dimensional lattice, from a cold start
        dict(kind="circulant", M0=30, M1=45, D=16, precision="fp64", name="xstep30x45_D16_fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _clusters(n):
    """The cluster count nearest n that a one-dimensional lattice may have: up to 64, or n1 * n2 with
    both factors up to 64."""
    ok = lambda k: 2 <= k <= 64 or (64 < k <= 4096 and any(k % a == 0 and k // a <= 64 for a in range(2, 65)))  # noqa: E731
    return next(k for d in range(4096) for k in (n - d, n + d) if ok(k))


def draw(rng):
    kind = rng.choices(["sweep", "batch", "general", "bound", "circulant"], [10, 1, 3, 1, 1])[0]
    model = rng.choice(["tfim", "xxz"])
    if kind == "sweep":
        L = rng.choice([1, 2, 2, 2, 3, 4])
        if L == 4:
            n = _clusters(_log(rng, 24, 400))
            if rng.random() < 0.3:
                a = rng.randint(4, 16)
                return _sweep("tfim", 2 * a, 2 * rng.randint(4, 16), 2, 2, "mixed", 10, rng.randint(6, 12))
            return _sweep(model, 4 * n, 0, 4, 1, "mixed", 10, rng.randint(6, 12))
        precision = rng.choice(["fp64", "fp64", "mixed", "df64"])
        if L == 3:
            return _sweep(model, 3 * _clusters(_log(rng, 16, 160)), 0, 3, 1, precision, 10, rng.randint(4, 8))
        sweeps = rng.randint(15, 50)
        if rng.random() < 0.3:
            a, b = rng.randint(4, 64), rng.randint(4, 64)
            return _sweep(model, a * L, b, L, 1, precision, 40, sweeps)
        return _sweep(model, L * _clusters(_log(rng, 12, 4096)), 0, L, 1, precision, 40, sweeps)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 32), length=_log(rng, 64, 512),
                    precision=rng.choice(["mixed", "fp64"]), start=40, sweeps=rng.randint(10, 40))
    if kind == "general":
        if rng.random() < 0.4:
            n = 2 * rng.randint(4, 12)
            return dict(kind="general", model="fermion", spins=n, cluster=2, start=20, sweeps=rng.randint(10, 20))
        L = rng.choice([1, 2])
        n = _log(rng, 16, 128) if L == 1 else 2 * _log(rng, 6, 32)
        return dict(kind="general", model=model, spins=n, cluster=L, start=6, sweeps=rng.randint(3, 8))
    if kind == "bound":
        L = rng.choice([1, 2])
        return dict(kind="bound", model=model, lx=L * _clusters(_log(rng, 24, 4096)), ly=0, cx=L, cy=1, start=40)
    return dict(kind="circulant", M0=rng.randint(4, 64), M1=rng.randint(4, 64), D=rng.choice([4, 16, 16]),
                precision=rng.choice(["fp64", "df64"]))


# ---- inputs --------------------------------------------------------------------------------------

def _rng(seed):
    return np.random.default_rng([20210604, int(seed)])


def _field(model, rng):
    """h of the transverse-field Ising model, or Delta of the XXZ model."""
    return float(rng.uniform(0.2, 2.0) if model == "tfim" else rng.uniform(0.0, 1.5))


def _shape(case):
    lattice = (case["lx"], case["ly"]) if case["ly"] else (case["lx"],)
    cluster = (case["cx"], case["cy"]) if case["ly"] else (case["cx"],)
    return lattice, cluster


def _ham(model, x, dim):
    return ve.ve_ham_tfim(dim, 1.0, x) if model == "tfim" else ve.ve_ham_xxz(dim, 1.0, x)


def _instances(case, seed):
    """Chains of the batch: half Ising, half XXZ, lengths around case["length"], 2- and (every
    fourth) 3-spin clusters."""
    rng = _rng(seed)
    out = []
    for i in range(case["count"]):
        model = "tfim" if i % 2 == 0 else "xxz"
        L = 3 if i % 4 == 3 else 2
        n = _clusters(max(4, (case["length"] * (3 + i % 5)) // (5 * L * (4 if L == 3 else 1))))
        out.append((model, _field(model, rng), n * L, L))
    return out


def _disordered(spins, model, rng):
    """Open chain with random fields and couplings xi / r^2 between all spins."""
    h = rng.uniform(0.5, 1.5, size=spins)
    s, t = np.triu_indices(spins, 1)
    J = rng.uniform(0.5, 1.5, size=len(s)) / (t - s).astype(np.float64) ** 2
    x, z = np.array([[0.0, 1.0], [1.0, 0.0]]), np.diag([1.0, -1.0])
    zz = np.kron(z, z)
    if model == "tfim":
        on, ops = -h[:, None, None] * x, -J[:, None, None] * zz
    else:
        delta = rng.uniform(0.0, 1.5, size=spins)
        flip = np.zeros((4, 4))
        flip[1, 2] = flip[2, 1] = 2.0  # xx + yy
        on, ops = -0.1 * h[:, None, None] * z, J[:, None, None] * (flip + delta[s][:, None, None] * zz)
    return dict(nspins=spins, onsite=on, bond_sites=np.stack([s, t], 1).astype(np.int32), bond_ops=ops)


def _fermions(sites, rng):
    """Ring with hopping -1 and the long-range repulsion 2 U / d(i, j)."""
    U = float(rng.uniform(0.5, 1.5))
    hops = [(i, j, -1.0) for i, j in sorted({tuple(sorted((i, (i + 1) % sites))) for i in range(sites)})]
    pairs = [(i, j, 2.0 * U / min(j - i, sites - j + i)) for i in range(sites) for j in range(i + 1, sites)]
    return dict(nsites=sites, hops=hops, pairs=pairs)


class _Handle:
    """A solver handle that goes with the state that holds it."""

    def __init__(self, h, destroy):
        self.h, self._destroy = h, destroy

    def __del__(self):
        if self.h:
            self._destroy(self.h)
            self.h = None


def _host(n, dtype=torch.float64):
    """Page-locked host memory, as a program keeps for its checkpoints."""
    return torch.empty(n, dtype=dtype, pin_memory=torch.cuda.is_available())


def _buffers(s, size, get, h, precision):
    n = size(h) // 8
    s["saved"], s["out"] = _host(n), _host(n)
    get(h, s["saved"].numpy())
    if precision == "mixed":
        s["out32"] = torch.empty(n, dtype=torch.float32).zero_()


def prepare(case, seed):
    kind, s = case["kind"], dict(case=case)
    if kind in ("sweep", "bound"):
        lattice, cluster = _shape(case)
        x = _field(case["model"], _rng(seed))
        opt = ve.ve_default_options(precision=PREC[case.get("precision", "fp64")])
        h = ve.ve_create(lattice, cluster, _ham(case["model"], x, len(lattice)), opt)
        s["handle"] = _Handle(h, ve.ve_destroy)
        ve.ve_iterate(h, case["start"])
        if kind == "sweep":
            _buffers(s, ve.ve_state_size, ve.ve_get_state, h, case["precision"])
    elif kind == "batch":
        inst = [((n,), (L,), _ham(model, x, 1)) for model, x, n, L in _instances(case, seed)]
        b = ve.ve_create_batch(inst, ve.ve_default_options(precision=PREC[case["precision"]]))
        s["handle"] = _Handle(b, ve.ve_batch_destroy)
        ve.ve_batch_iterate(b, case["start"])
        s["parts"] = []
        for i in range(case["count"]):
            part = dict(h=ve.ve_batch_handle(b, i))
            _buffers(part, ve.ve_state_size, ve.ve_get_state, part["h"], case["precision"])
            s["parts"].append(part)
    elif kind == "general":
        rng = _rng(seed)
        if case["model"] == "fermion":
            h = ve.ve_general_create_fermions(_fermions(case["spins"], rng), case["cluster"])
        else:
            h = ve.ve_general_create(_disordered(case["spins"], case["model"], rng), case["cluster"])
        s["handle"] = _Handle(h, ve.ve_general_destroy)
        ve.ve_general_iterate(h, case["start"])
        _buffers(s, ve.ve_general_state_size, ve.ve_general_get_state, h, "fp64")
    else:
        M, D = (case["M0"], case["M1"]), case["D"]
        s["x"] = torch.from_numpy(_first_row(M, D, _rng(seed))).cuda()
        s["y"] = torch.empty_like(s["x"])
        s["ws"] = torch.empty(ve.ve_circulant_workspace_size(M, D), dtype=torch.uint8, device="cuda")
    return s


def _first_row(M, D, rng):
    """A first block row with X_{0,-delta} = X_{0,delta}^T whose block-circulant matrix has
    eigenvalues of both signs."""
    N = M[0] * M[1]
    X = rng.normal(size=(M[0], M[1], D, D)) / np.sqrt(N)
    neg = np.roll(X[::-1, ::-1], (1, 1), (0, 1))  # X_{0,-delta}
    X = 0.5 * (X + np.swapaxes(neg, 2, 3)).reshape(N, D, D)
    X[0] += 0.1 * np.eye(D)
    return X


# ---- one pass ------------------------------------------------------------------------------------

def _saved(s, get, h):
    get(h, s["out"].numpy())
    return s["out32"].copy_(s["out"]) if "out32" in s else s["out"]


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "sweep":
        h = s["handle"].h
        ve.ve_set_state(h, s["saved"].numpy())
        _, st = ve.ve_iterate(h, case["sweeps"])
        return {"energy": st.energy_per_spin, "state": _saved(s, ve.ve_get_state, h)}
    if kind == "bound":
        c = ve.ve_bound(s["handle"].h)
        return {"bound": c.bound_per_spin, "raw": c.raw_bound, "primal": c.primal_per_spin}
    if kind == "batch":
        for p in s["parts"]:
            ve.ve_set_state(p["h"], p["saved"].numpy())
        _, sts = ve.ve_batch_iterate(s["handle"].h, case["sweeps"])
        return {"energy": np.array([st.energy_per_spin for st in sts]).astype(np.float32),
                "states": [_saved(p, ve.ve_get_state, p["h"]) for p in s["parts"]]}
    if kind == "general":
        h = s["handle"].h
        ve.ve_general_set_state(h, s["saved"].numpy())
        _, st = ve.ve_general_iterate(h, case["sweeps"])
        return {"energy": st.energy_per_spin, "state": _saved(s, ve.ve_general_get_state, h)}
    ve.ve_circulant_project(s["x"].data_ptr(), s["y"].data_ptr(), (case["M0"], case["M1"]), case["D"],
                            s["ws"].data_ptr(), s["ws"].numel(), PREC[case["precision"]],
                            torch.cuda.current_stream().cuda_stream)
    return s["y"]


# ---- what a pass cannot do without ---------------------------------------------------------------

def _eig(n, cplx):
    """Flops of one projection: tridiagonalise, back-transform, rebuild (13/3 n^3; complex x 4)."""
    return 13.0 / 3.0 * n ** 3 * (4 if cplx else 1)


def _ti_work(N, L, sweeps):
    D = 4 ** L
    m = 2 ** L
    state = 8.0 * (m * m + 2 * (N - 1) * (D * D + m * m) + N * D * D)
    fft = 2 * 5.0 * N * math.log2(N) * D * D / 2
    # opposite offsets and opposite wavevectors share one projection
    return state, sweeps * (N / 2 * (_eig(D, False) + 60 * D * D) + (N / 2 + 1) * _eig(D, True) + fft)


def work(case):
    kind = case["kind"]
    if kind in ("sweep", "bound"):
        lattice, cluster = _shape(case)
        L = int(np.prod(cluster))
        N = int(np.prod(lattice)) // L
        state, flops = _ti_work(N, L, case.get("sweeps", 1))
        if kind == "sweep":
            return {"bytes": 2 * state, "flops": flops}
        D = 4 ** L  # eigenvalues alone: the tridiagonalisation
        return {"bytes": state / 3, "flops": (N - 1) * 4 / 3 * D ** 3 + (N / 2 + 1) * 16 / 3 * D ** 3}
    if kind == "batch":
        w = [_ti_work(n // L, L, case["sweeps"]) for _, _, n, L in _instances(case, 0)]
        return {"bytes": 2 * sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    if kind == "general":
        L, n = case["cluster"], case["spins"]
        N, D, m = n // L, 4 ** L, 2 ** L
        K = N * (N - 1) / 2
        state = 8.0 * (N * m * m + 2 * K * (D * D + m * m) + (N * D) ** 2)
        return {"bytes": 2 * state,
                "flops": case["sweeps"] * (K * (_eig(D, False) + 60 * D * D) + _eig(N * D, False))}
    N, D = case["M0"] * case["M1"], case["D"]
    return {"bytes": 16.0 * N * D * D,
            "flops": (N / 2 + 1) * _eig(D, True) + 2 * 5.0 * N * math.log2(N) * D * D / 2}


# ---- the same in plain 64-bit arithmetic (Algorithms 5 and 6 of arXiv:2106.02682) ----------------

def _psd(C):
    w, V = torch.linalg.eigh(0.5 * (C + C.mH))
    return (V * w.clamp_min(0.0).unsqueeze(-2)) @ V.mH


def _A1(r, m):
    return torch.einsum("...abcb->...ac", r.reshape(r.shape[:-2] + (m,) * 4))


def _A2(r, m):
    return torch.einsum("...abad->...bd", r.reshape(r.shape[:-2] + (m,) * 4))


def _up1(y):
    m = y.shape[-1]
    e = torch.eye(m, dtype=y.dtype, device=y.device)
    return torch.einsum("...ac,bd->...abcd", y, e).reshape(y.shape[:-2] + (m * m, m * m))


def _up2(y):
    m = y.shape[-1]
    e = torch.eye(m, dtype=y.dtype, device=y.device)
    return torch.einsum("ac,...bd->...abcd", e, y).reshape(y.shape[:-2] + (m * m, m * m))


def _G(r, m):
    return torch.einsum("...adbc->...abcd", r.reshape(r.shape[:-2] + (m,) * 4)).reshape(r.shape)


def _eff(H, X, m):
    S = torch.einsum("...prsq->...pqrs", X.reshape(X.shape[:-2] + (m,) * 4)).reshape(X.shape)
    return H - S - S.mT


def _solve(y, m):
    """(mu + nu A1* A1 + nu A2* A2)^-1 y."""
    D, a = m * m, NU * m
    P1, P2 = _up1(_A1(y, m)) / m, _up2(_A2(y, m)) / m
    Q = torch.einsum("...ii->...", y)[..., None, None] * torch.eye(D, dtype=y.dtype, device=y.device) / D
    return (y - P1 - P2 + Q) / MU + (P1 + P2 - 2 * Q) / (MU + a) + Q / (MU + 2 * a)


def _H00(X, m):
    return torch.einsum("...abad->...bd", X.reshape(X.shape[:-2] + (m,) * 4))


def _G00(r):
    m = r.shape[-1]
    e = torch.eye(m, dtype=r.dtype, device=r.device)
    return torch.einsum("ac,...db->...abcd", e, r).reshape(r.shape[:-2] + (m * m, m * m))


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _embed(op, sites, n):
    """`op` on the listed spins of n."""
    k = len(sites)
    rest = [q for q in range(n) if q not in sites]
    full = np.kron(op, np.eye(2 ** (n - k))).reshape([2] * (2 * n))
    order = list(sites) + rest
    inv = [order.index(q) for q in range(n)]
    return full.transpose(inv + [n + q for q in inv]).reshape(2 ** n, 2 ** n)


def _ti_blocks(model, x, lattice, cluster):
    px, pz = np.array([[0.0, 1.0], [1.0, 0.0]]), np.diag([1.0, -1.0])
    if model == "tfim":
        on, bond = -x * px, -np.kron(pz, pz)
    else:
        flip = np.zeros((4, 4))
        flip[1, 2] = flip[2, 1] = 2.0
        on, bond = np.zeros((2, 2)), flip + x * np.kron(pz, pz)
    dim = len(lattice)
    M = tuple(a // b for a, b in zip(lattice, cluster))
    L = int(np.prod(cluster))
    m, N = 2 ** L, int(np.prod(M))
    H0, Hp = np.zeros((m, m)), np.zeros((N, m * m, m * m))
    at = lambda s: int(np.ravel_multi_index([s[p] % cluster[p] for p in range(dim)], cluster))  # noqa: E731
    of = lambda s: int(np.ravel_multi_index([s[p] // cluster[p] for p in range(dim)], M))  # noqa: E731
    for s in np.ndindex(*cluster):
        H0 += _embed(on, [at(s)], L)
        for p in range(dim):
            for step in (1, -1):
                t = tuple((s[q] + step * (q == p)) % lattice[q] for q in range(dim))
                if of(t) == 0:
                    H0 += _embed(bond, [at(s), at(t)], L) if step == 1 else 0.0
                else:  # the bond operators are symmetric under exchange of their two spins
                    Hp[of(t)] += _embed(bond, [at(s), L + at(t)], 2 * L)
    return M, L, m, H0, Hp


def _sweep_exact(model, x, lattice, cluster, sweeps, bound=False):
    M, L, m, H0, Hp = _ti_blocks(model, x, lattice, cluster)
    N, D, d = int(np.prod(M)), m * m, _dev()
    H0, Hp = torch.from_numpy(H0).to(d), torch.from_numpy(Hp[1:]).to(d)
    P, f = N - 1, dict(dtype=torch.float64, device=d)
    rho0, rt = torch.eye(m, **f) / m, torch.eye(D, **f).repeat(P, 1, 1) / D
    lam, l1, l2 = torch.zeros(P, D, D, **f), torch.zeros(P, m, m, **f), torch.zeros(P, m, m, **f)
    X = torch.zeros(N, D, D, **f)
    X[0] = torch.eye(D, **f)
    axes, energy = tuple(range(len(M))), None
    half = _half(M)
    for _ in range(sweeps):
        rhs = MU * rt + _up1(NU * rho0 - l1) + _up2(NU * rho0 - l2) + lam - _eff(Hp, X[1:], m)
        rho = _solve(rhs, m)
        rt = _psd(rho - lam / MU)
        a1, a2 = _A1(rho, m), _A2(rho, m)
        r = ((NU * a1 + l1).sum(0) - (H0 - _H00(X[0], m))) / (NU * P)
        rho0 = r + (1 - r.trace()) / m * torch.eye(m, **f)
        lam, l1, l2 = lam + MU * (rt - rho), l1 + NU * (a1 - rho0), l2 + NU * (a2 - rho0)
        X = X - EPS * torch.cat([_G00(rho0)[None], _G(rho, m)])
        F = torch.fft.fftn(X.reshape(M + (D, D)), dim=axes).reshape(N, D, D)
        Y = torch.empty_like(F)
        k, mk = half
        p = _psd(F[k])
        Y[mk] = p.conj()
        Y[k] = p
        X = torch.fft.ifftn(Y.reshape(M + (D, D)), dim=axes).real.reshape(N, D, D).contiguous()
        energy = ((H0 @ rho0).trace() + 0.5 * (Hp * rho.mT).sum()) / L
    if not bound:
        return energy, torch.cat([t.reshape(-1) for t in (rho0, rt, lam, l1, l2, X)])
    idx = np.arange(N).reshape(M)
    neg = np.roll(idx[tuple(slice(None, None, -1) for _ in M)], [1] * len(M), axes).reshape(-1)
    K = _eff(Hp, X[1:], m) + _up1(l1) + _up2(l1[torch.from_numpy(neg[1:] - 1).to(d)])
    K0 = H0 - _H00(X[0], m) - l1.sum(0)
    cc = np.stack(np.unravel_index(np.arange(N), M), 1)
    # c(delta): the ordered pairs a < a + delta
    count = np.zeros(N)
    for a in range(N):
        count += np.ravel_multi_index(tuple(((cc[a] + cc) % np.array(M)).T), M) > a
    pairs = torch.linalg.eigvalsh(0.5 * (K + K.mT))[:, 0]
    raw = N * torch.linalg.eigvalsh(0.5 * (K0 + K0.mT))[0] + (torch.from_numpy(count[1:]).to(d) * pairs).sum()
    F = torch.fft.fftn(X.reshape(M + (D, D)), dim=axes).reshape(N, D, D)[half[0]]
    low = torch.linalg.eigvalsh(0.5 * (F + F.mH)).min()
    return raw, (raw - N * m * torch.clamp(-low, min=0.0)) / (N * L), energy


def _half(M):
    """One of each pair of opposite wavevectors, and the other."""
    idx = np.arange(int(np.prod(M))).reshape(M)
    neg = np.roll(idx[tuple(slice(None, None, -1) for _ in M)], [1] * len(M), tuple(range(len(M)))).reshape(-1)
    k = np.nonzero(np.arange(len(neg)) <= neg)[0]
    return torch.from_numpy(k).to(_dev()), torch.from_numpy(neg[k]).to(_dev())


def _ladder(n):
    """Annihilation operators of n sites (Jordan-Wigner), basis (empty, occupied) per site."""
    a, z = np.array([[0.0, 1.0], [0.0, 0.0]]), np.diag([1.0, -1.0])
    out = []
    for i in range(n):
        op = np.eye(1)
        for j in range(n):
            op = np.kron(op, z if j < i else a if j == i else np.eye(2))
        out.append(op)
    return out


def _general_blocks(case, seed):
    """H_i, H_ij and the signs of the off-diagonal blocks of G."""
    L = case["cluster"]
    N, m = case["spins"] // L, 2 ** L
    pi, pj = np.triu_indices(N, 1)
    slot = {(i, j): k for k, (i, j) in enumerate(zip(pi, pj))}
    Hi, Hij = np.zeros((N, m, m)), np.zeros((len(pi), m * m, m * m))
    rng = _rng(seed)
    if case["model"] == "fermion":
        t = _fermions(case["spins"], rng)
        a1, a2 = _ladder(L), _ladder(2 * L)
        terms = [(i, j, v, True) for i, j, v in t["hops"]] + [(i, j, v, False) for i, j, v in t["pairs"]]
        for i, j, v, hop in terms:
            ci, cj = i // L, j // L
            a, n = (a1, L) if ci == cj else (a2, 2 * L)
            x, y = a[i % L], a[j % L if ci == cj else L + j % L]
            e = 0.5 * np.eye(2 ** n)
            op = v * (x.T @ y + y.T @ x) if hop else v * (x.T @ x - e) @ (y.T @ y - e)
            (Hi[ci] if ci == cj else Hij[slot[(ci, cj)]])[...] += op
        p = np.array([bin(s).count("1") % 2 for s in range(m)])
        pa, pc, pd = np.meshgrid(p, p, p, indexing="ij")
        sign = np.broadcast_to(((-1.0) ** (pa * (pc + pd)))[:, None], (m, m, m, m)).reshape(m * m, m * m)
        return Hi, Hij, pi, pj, sign.copy()
    t = _disordered(case["spins"], case["model"], rng)
    for s in range(case["spins"]):
        Hi[s // L] += _embed(t["onsite"][s], [s % L], L)
    for (s, u), op in zip(t["bond_sites"], t["bond_ops"]):
        s, u = int(s), int(u)
        if s // L == u // L:
            Hi[s // L] += _embed(op, [s % L, u % L], L)
        else:
            Hij[slot[(s // L, u // L)]] += _embed(op, [s % L, L + u % L], 2 * L)
    return Hi, Hij, pi, pj, np.ones((m * m, m * m))


def _general_exact(case, seed):
    Hi, Hij, pi, pj, sign = _general_blocks(case, seed)
    d, L = _dev(), case["cluster"]
    N, m = Hi.shape[0], Hi.shape[1]
    D, K = m * m, len(pi)
    Hi, Hij, sign = (torch.from_numpy(v).to(d) for v in (Hi, Hij, sign))
    pi, pj = torch.from_numpy(pi).to(d), torch.from_numpy(pj).to(d)
    f = dict(dtype=torch.float64, device=d)
    ri, rt = torch.eye(m, **f).repeat(N, 1, 1) / m, torch.eye(D, **f).repeat(K, 1, 1) / D
    lam, l1, l2 = torch.zeros(K, D, D, **f), torch.zeros(K, m, m, **f), torch.zeros(K, m, m, **f)
    X, diag, energy = torch.eye(N * D, **f), torch.arange(N, device=d), None
    for _ in range(case["start"] + case["sweeps"]):
        X4 = X.reshape(N, D, N, D)
        Hp = _eff(Hij, sign * X4[pi, :, pj, :], m)
        rhs = MU * rt + _up1(NU * ri[pi] - l1) + _up2(NU * ri[pj] - l2) + lam - Hp
        rho = _solve(rhs, m)
        rt = _psd(rho - lam / MU)
        a1, a2 = _A1(rho, m), _A2(rho, m)
        acc = _H00(X4[diag, :, diag, :], m) - Hi
        acc = acc.index_add(0, pi, NU * a1 + l1).index_add(0, pj, NU * a2 + l2) / (NU * (N - 1))
        z = (1.0 - torch.einsum("nii->n", acc)) / m
        ri = acc + z[:, None, None] * torch.eye(m, **f)
        lam, l1, l2 = lam + MU * (rt - rho), l1 + NU * (a1 - ri[pi]), l2 + NU * (a2 - ri[pj])
        g = sign * _G(rho, m)
        G = torch.zeros(N, D, N, D, **f)
        G[pi, :, pj, :] = g
        G[pj, :, pi, :] = g.mT
        G[diag, :, diag, :] = _G00(ri)
        X = _psd(X - EPS * G.reshape(N * D, N * D))
        energy = ((Hi * ri.mT).sum() + (Hij * rho.mT).sum()) / (N * L)
    return energy, torch.cat([t.reshape(-1) for t in (ri, rt, lam, l1, l2, X)])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sweep", "bound"):
        lattice, cluster = _shape(case)
        if np.prod(cluster) > 3:
            return None  # hundreds of 256 x 256 eigenproblems a sweep
        x = _field(case["model"], _rng(seed))
        if kind == "bound":
            raw, bound, primal = _sweep_exact(case["model"], x, lattice, cluster, case["start"], True)
            return {"bound": float(bound), "raw": float(raw), "primal": float(primal)}
        e, state = _sweep_exact(case["model"], x, lattice, cluster, case["start"] + case["sweeps"])
        return {"energy": float(e), "state": state.cpu()}
    if kind == "batch":
        got = [_sweep_exact(model, x, (n,), (L,), case["start"] + case["sweeps"]) if L == 2 else (None, None)
               for model, x, n, L in _instances(case, seed)]
        return {"energy": None, "states": [None if v is None else v.cpu() for _, v in got]}
    if kind == "general":
        e, state = _general_exact(case, seed)
        return {"energy": float(e), "state": state.cpu()}
    M, D = (case["M0"], case["M1"]), case["D"]
    X = torch.from_numpy(_first_row(M, D, _rng(seed))).to(_dev()).reshape(M + (D, D))
    F = torch.fft.fftn(X, dim=(0, 1))
    Y = torch.fft.ifftn(_psd(F.reshape(-1, D, D)).reshape(M + (D, D)), dim=(0, 1)).real
    return Y.reshape(M[0] * M[1], D, D).cpu()
