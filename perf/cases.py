"""Performance cases of the Wilson-loop library: what its users have it compute.

Each case is one call of a public entry point (plain, nested and spin-resolved Wilson
loops, single planes and stacks, and the plaquette flux) on a tight-binding model given
as a hopping list: two- and four-band models on small and long grids, spinful
many-orbital models of Wannier type, and disordered or defective supercells; in both
precisions the entry points offer.  Models and sizes are those of the repository's
configurations, tests and benchmark.  Every seed gives another model (couplings,
disorder, hoppings) and another plane origin; a small generic on-site term keeps the
phases away from the symmetric values 0 and pi, where their sign would be rounding.
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2312_13051_gb300 import _lib
from paper_2312_13051_gb300 import inputs as I

FP64, MIXED = "fp64", "mixed"


def _case(name, kind, model, size, N, Nt, precision, Ns=1, drop=0):
    c = dict(kind=kind, model=model, size=size, N=N, Nt=Nt, Ns=Ns, drop=drop, precision=precision)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a two-band Chern insulator in a parameter scan (one loop per ky)
        _case("eq4_24x24_fp64", "loop", "eq4", 1, 24, 24, FP64),
        # the benchmark's headline: nested loop of a quadrupole insulator
        _case("bbh_60x60_nested_mixed", "nested", "bbh", 1, 60, 60, MIXED),
        # spin-Chern number of the four-band spin-Hall model, default precision
        _case("spin_hall_51x51_spin_fp64", "spin", "spin_hall", 1, 51, 51, FP64),
        # a long scan of one direction: thousands of independent loops in one call
        _case("bbh_60x3840_mixed", "loop", "bbh", 1, 60, 3840, MIXED),
        # nested loop against k_z of a three-dimensional higher-order insulator
        _case("choti_32x32x16_nested_fp64", "nested", "choti", 1, 32, 32, FP64, Ns=16),
        # six coupled quadrupole layers (n = 24, p = 12): nested loop, odd grid
        _case("layers6_31x31_nested_mixed", "nested", "layers", 6, 31, 31, MIXED),
        # n = 32, p = 8: the largest model solved in shared memory, spin-resolved
        _case("orbital16_21x21_spin_fp64", "spin", "manyband", 16, 21, 21, FP64),
        # a vacancy in a topological insulator (n = 124, p = 62), spin-resolved
        _case("vacancy6_16x16_spin_fp64", "spin", "vacancy", 6, 16, 16, FP64),
        # many-orbital model in FP64, one orbital removed (n = 127, p = 32)
        _case("orbital64_17x17_fp64", "loop", "manyband", 64, 17, 17, FP64, drop=1),
        # the many-band configuration (n = 256, p = 64) on a ragged grid
        _case("orbital128_31x27_mixed", "loop", "manyband", 128, 31, 27, MIXED),
        # disordered supercell at half filling (n = 400, p = 200)
        _case("disordered10_16x16_mixed", "loop", "disordered", 10, 16, 16, MIXED),
        # spin-Chern number of a disordered quadrupolar supercell by plaquettes (n = 324)
        _case("quadrupolar9_6x6_flux_mixed", "flux", "quadrupolar", 9, 6, 6, MIXED),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: model family, its size, the grid and the precision."""
    while True:
        precision = rng.choice((FP64, MIXED))
        fam = rng.choice(("few", "few", "orbital", "orbital", "supercell"))
        Ns = 1
        drop = 0
        if fam == "few":
            model, kind = rng.choice((("eq4", "loop"), ("bbh", "nested"), ("bbh", "loop"),
                                      ("spin_hall", "spin"), ("choti", "nested"), ("choti", "loop")))
            size = 1
            N = rng.randint(12, 80)
            Nt = rng.randint(12, 60) if kind == "nested" else _log(rng, 12, 3000)
            Ns = rng.randint(2, 16) if model == "choti" and Nt <= 60 else 1
        elif fam == "orbital":
            model, kind = rng.choice((("manyband", "loop"), ("manyband", "spin"), ("layers", "nested")))
            size = _log(rng, 2, 20) if model == "layers" else _log(rng, 8, 128)
            drop = rng.choice((0, 1)) if kind == "loop" else 0
            N, Nt = rng.randint(11, 41), rng.randint(5, 41)
        else:
            model, kind = rng.choice((("disordered", "loop"), ("disordered", "spin"),
                                      ("vacancy", "loop"), ("vacancy", "spin"), ("quadrupolar", "flux")))
            size = rng.randint(4, 10)
            if kind == "flux":
                size, N, Nt = min(size, 9), rng.randint(5, 8), rng.randint(5, 8)
            else:
                N, Nt = rng.randint(10, 18), rng.randint(5, 18)
        c = _case(None, kind, model, size, N, Nt, precision, Ns=Ns, drop=drop)
        n, p, _ = _sizes(c)
        K = N * Nt * Ns
        # cost of the solves, FP64 arithmetic counted four times; at most the largest listed
        # case (n = 256, 31 x 27, mixed)
        cost = K * n ** 3 * (4.0 if precision == FP64 else 1.0) * (1.5 if kind in ("spin", "flux") else 1.0)
        if cost <= 0.8 * 31 * 27 * 256.0 ** 3 and p >= 1:
            return c


def _sizes(c):
    """(orbitals n, occupied bands p, nested sector m) of a case."""
    L = c["size"]
    if c["model"] == "eq4":
        return 2, 1, 1
    if c["model"] in ("bbh", "spin_hall", "choti"):
        return 4, 2, 1
    if c["model"] == "layers":
        return 4 * L, 2 * L, L
    if c["model"] == "manyband":
        return 2 * L - c["drop"], 2 * (L // 4), L // 4
    cells = L * L - (len(I.vacancy_cells(L, 1.0)) if c["model"] == "vacancy" else 0)
    return 4 * cells, 2 * cells, cells


def _generic(model, rng, eps=0.05):
    """The model with a random Hermitian on-site term of size eps."""
    n = model.n
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    T = eps * 0.5 * (A + A.conj().T)
    ii, jj = np.nonzero(np.ones((n, n)))
    return I.HoppingList(n=n, R=np.concatenate([model.R, np.zeros((n * n, 3), np.int32)]),
                         i=np.concatenate([model.i, ii]), j=np.concatenate([model.j, jj]),
                         t=np.concatenate([model.t, T[ii, jj]]), dim=model.dim, name=model.name)


def _inputs(c, seed):
    """(model, plane or stack, spin operator or None), from the seed alone."""
    rng = np.random.default_rng([20231213, int(seed)])
    L, name = c["size"], c["model"]
    u = rng.uniform
    if name == "eq4":
        model = _generic(I.chern_eq4(u(1.0, 1.5)), rng)
    elif name == "bbh":
        model = _generic(I.bbh(u(0.4, 0.6), u(0.4, 0.6)), rng)
    elif name == "spin_hall":
        model = _generic(I.spin_hall(u(0.8, 1.2)), rng)
    elif name == "choti":
        model = _generic(I.choti_eq9(u(0.8, 1.2), u(-1.7, -1.3)), rng)
    elif name == "layers":  # coupled by the on-site term
        model = I.direct_sum([I.bbh(u(0.4, 0.6), u(0.4, 0.6)) for _ in range(L)])
        model = _generic(model, rng, eps=0.2 / math.sqrt(model.n))
    elif name == "manyband":
        model = I.manyband(L, seed=int(rng.integers(2 ** 31)))
        if c["drop"]:
            model = I.remove_orbitals(model, [model.n - 1])
    elif name == "disordered":
        model = I.supercell(I.spin_hall(u(0.8, 1.2)), L, W=u(0.5, 1.5), seed=int(rng.integers(2 ** 31)))
    elif name == "vacancy":
        model = I.vacancy_supercell(I.bhz_eq7(u(1.3, 1.5)), L, 1.0, W=u(0.1, 0.3),
                                    seed=int(rng.integers(2 ** 31)))
    else:
        model = I.supercell(I.quadrupolar_eq10(), L, W=u(0.5, 1.0), seed=int(rng.integers(2 ** 31)),
                            onsite=I.EQ10_SPIN)
    origin = tuple(u(0.0, 1.0) if d < model.dim else 0.0 for d in range(3))
    plane = I.Plane(c["N"], c["Nt"], origin=origin)
    if c["Ns"] > 1:
        plane = I.PlaneStack(plane, (0, 0, 1), c["Ns"])
    S = None
    if c["kind"] in ("spin", "flux"):
        cell = {"spin_hall": I.SPIN_HALL_SZ, "disordered": I.SPIN_HALL_SZ, "quadrupolar": I.EQ10_SPIN,
                "vacancy": np.diag([1.0, -1.0, -1.0, 1.0]).astype(np.complex128)}.get(name)
        S = I.manyband_sz(L) if cell is None else np.kron(np.eye(model.n // 4), cell)
    return model, plane, S


def prepare(case, seed):
    model, plane, S = _inputs(case, seed)
    n, p, m = _sizes(case)
    # a context keeps the plan of its last hopping list: a program that works with a dense
    # many-orbital model (10^5 hoppings and more) keeps a context for it, while a scan over
    # couplings or disorder realisations passes a new list to the same one in every call
    ctx = _lib.Context(torch.cuda.current_device()) if case["model"] == "manyband" else _lib.context()
    return dict(case=case, model=model, plane=plane, S=S, p=p, m=m, ctx=ctx)


def run(state):
    c = state["case"]
    # check=False: a scan reads the sticky status once at its end
    kw = dict(precision=c["precision"], ctx=state["ctx"], check=False)
    if c["kind"] == "loop":
        return _lib.wilson_loop(state["model"], state["plane"], state["p"], **kw)
    if c["kind"] == "nested":
        return _lib.nested_wilson_loop(state["model"], state["plane"], state["p"], m=state["m"], **kw)
    if c["kind"] == "spin":
        return _lib.spin_resolved_wilson_loop(state["model"], state["plane"], state["p"], state["S"], -1, **kw)
    return _lib.plaquette_flux(state["model"], state["plane"], state["p"], state["S"], -1, **kw)


def work(case):
    """Bytes: the hopping list and the outputs once.  Flops (real, FP64-grade): Bloch sums,
    Hermitian eigensolves with p vectors, spin split, overlaps, loop products, eigenphases."""
    n, p, m = _sizes(case)
    N, Nt, kind = case["N"], case["Nt"] * case["Ns"], case["kind"]
    K = N * Nt
    nnz = {"eq4": 16, "bbh": 40, "spin_hall": 56, "choti": 84}.get(case["model"])
    if nnz is None:
        nnz = {"manyband": 13 * n * n, "layers": n * n + 10 * n}.get(case["model"], 11 * n)
    per_k = 8 * nnz + 16 / 3 * n ** 3 + 8 * n * n * p
    pe = p
    if kind in ("spin", "flux"):
        pe = p // 2
        per_k += 8 * n * p * p + 8 * n * p * pe + 16 / 3 * p ** 3 + 8 * p * p * pe
    per_k += (2 if kind == "flux" else 1) * 8 * n * pe * pe
    flops = K * per_k
    if kind == "flux":
        flops += K * 2 * 8 / 3 * pe ** 3
        out = K + 1 + 2 * Nt
    else:
        flops += Nt * ((N - 1) * 8 * pe ** 3 + 10 * pe ** 3)
        out = Nt * pe + Nt
        if kind == "spin":
            out += K * p + Nt
        if kind == "nested":
            flops += K * (8 * p * p * m + 8 * n * p * m + 8 * n * m * m + 8 * m ** 3)
            out += N * case["Ns"] * m + Nt
    return {"bytes": 36.0 * nnz + 8.0 * out, "flops": float(flops)}


# --------------------------------------------------------------------------
# The same results in plain numpy / torch FP64 on the host
# --------------------------------------------------------------------------

def _pool(fn, items):
    def one(x):
        torch.set_num_threads(1)
        return fn(x)
    with ThreadPoolExecutor(16) as ex:
        return list(ex.map(one, items))


def _row_states(T, Rs, f, p):
    """Eigenvalues and the p lowest eigenvectors of H(f) for the k-points of a row block."""
    ph = np.exp(2j * np.pi * (f @ Rs.T))
    n = T.shape[1]
    H = (ph @ T.reshape(len(Rs), n * n)).reshape(len(f), n, n)
    if n <= 32:
        E, V = np.linalg.eigh(H)
    else:
        E, V = (x.numpy() for x in torch.linalg.eigh(torch.from_numpy(H)))
    return E, np.ascontiguousarray(V[:, :, :p])


def _angles(W):
    if W.shape[-1] <= 4:
        lam = np.linalg.eigvals(W)
    else:
        lam = np.stack(_pool(lambda w: torch.linalg.eigvals(torch.from_numpy(w)).numpy(), list(W)))
    return lam


def _wrap_gap(a, b):
    d = np.abs(a[:, :, None] - b[:, None, :])
    return np.min(np.minimum(d, 2 * np.pi - d), axis=(1, 2))


def exact(case, seed):
    model, plane, S = _inputs(case, seed)
    n, p, m = _sizes(case)
    base = plane.plane if case["Ns"] > 1 else plane
    N, Ntp, Ns, kind = case["N"], case["Nt"], case["Ns"], case["kind"]
    Nt = Ntp * Ns
    if N * Nt * n ** 3 > 3e10:
        return None
    Rs, inv = np.unique(model.R, axis=0, return_inverse=True)
    T = np.zeros((len(Rs), n, n), np.complex128)
    np.add.at(T, (inv.reshape(-1), model.i, model.j), model.t)
    Rs = Rs.astype(np.float64)
    j = np.arange(N)[:, None] / N
    rows = []
    for i in range(Nt):
        o = np.array(base.origin) + (i % Ntp) / Ntp * np.array(base.trans_dir)
        if Ns > 1:
            o = o + (i // Ntp) / Ns * np.array(plane.sweep_dir, float)
        rows.append(o[None, :] + j * np.array(base.loop_dir, float)[None, :])
    block = max(1, 4096 // N) if n <= 32 else 1
    chunks = [np.concatenate(rows[a:a + block]) for a in range(0, Nt, block)]
    parts = _pool(lambda f: _row_states(T, Rs, f, p), chunks)
    E = np.concatenate([x[0] for x in parts]).reshape(Nt, N, n)
    U = np.concatenate([x[1] for x in parts]).reshape(Nt, N, n, p)
    gap = (E[:, :, p] - E[:, :, p - 1]).min(axis=1)
    dag = lambda x: x.conj().swapaxes(-1, -2)  # noqa: E731
    out_pso = pgap = None
    if S is not None:
        s = np.diag(S).real  # every spin operator here is diagonal
        mu, V = np.linalg.eigh(dag(U) @ (s[:, None] * U))
        out_pso, pgap = mu, np.abs(mu).min(axis=(1, 2))
        U = U @ V[..., : p // 2]
    lead = (Ns, Ntp) if Ns > 1 else (Nt,)
    if kind == "flux":
        def link(A, B):
            d = np.linalg.slogdet(dag(A) @ B)[0]
            return d / np.abs(d)
        Lx = link(np.roll(U, -1, axis=1), U)
        Ly = link(np.roll(U, -1, axis=0), U)
        fl = np.angle(Ly * np.roll(Lx, -1, axis=0) * np.conj(np.roll(Ly, -1, axis=1)) * np.conj(Lx))
        return fl, np.array(fl.sum() / (2 * np.pi)), gap, pgap
    M = dag(np.roll(U, -1, axis=1)) @ U
    W = M[:, 0]
    for q in range(1, N):
        W = M[:, q] @ W
    if kind != "nested":
        th = np.sort(np.angle(_angles(W)), axis=-1)
        th = th.reshape(lead + th.shape[-1:])
        if kind == "spin":
            return th, out_pso, pgap.reshape(lead), gap.reshape(lead)
        return th, gap.reshape(lead)
    lam, Z = np.linalg.eig(W)
    th = np.angle(lam)
    ordr = np.argsort(np.mod(th + np.pi, 2 * np.pi), axis=1)
    ths = np.take_along_axis(th, ordr, axis=1)
    wg = _wrap_gap(ths[:, :m], ths[:, m:])
    nu = np.take_along_axis(Z, ordr[:, None, :m], axis=2)
    w = np.empty((N, Nt, n, m), np.complex128)
    for q in range(N):
        nu = np.linalg.qr(nu)[0]
        w[q] = U[:, q] @ nu
        nu = M[:, q] @ nu
    w = w.reshape(N, Ns, Ntp, n, m)
    A = dag(np.roll(w, -1, axis=2)) @ w
    Q = A[:, :, 0]
    for q in range(1, Ntp):
        Q = A[:, :, q] @ Q
    nest = np.sort(np.angle(np.linalg.eigvals(Q)), axis=-1).swapaxes(0, 1)
    nest = nest if Ns > 1 else nest[0]
    th = np.sort(th, axis=1)
    return th.reshape(lead + (p,)), nest, wg.reshape(lead), gap.reshape(lead)
