"""The cases by which this framework's speed is measured.

A case is a plain dict.  ``prepare`` makes what a user's program holds before the call (the
Hamiltonian, the trial and the AFQMC state on its stream), ``run`` is one pass through the public
entry points (a block of steps and the reading of what it gave), ``exact`` the same pass in plain
float64 PyTorch, written from the method's equations and sharing no code with the package.

Kinds
  walk   a phaseless walk: a block of steps, its energy records, the walkers and weights
         (closed shell, or two spin blocks when Ndn > 0; float64 or a mixed precision)
  noci   a walk with a multi-determinant trial of non-orthogonal determinants
  bp     a back-propagation window: the walk that records it and the density it gives
  group  uneven systems advanced together by one graph launch per block
  serve  whole requests through the continuous-batching server: set-up, walk, energies
  mcd    the modified Cholesky decomposition that makes the vectors L

Hamiltonians are the synthetic ones of this repository's workloads: h1 with the diagonal
linspace(-2, 2, M) and off-diagonal N(0, 0.05), Cholesky vectors with entries N(0, a exp(-g/M)) and
a such that sum_g |L_g|_F^2 is the value at M = 12, 48 vectors, a = 0.5; they are drawn on the GPU
here, because they are made many times.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1711_02242_gb300 as pkg
from paper_1711_02242_gb300.serve import Request, Server

DEV = "cuda:0"
PRECISION = {"fp64": pkg.AFQMC_FP64, "tf32": pkg.AFQMC_MIXED_TF32, "bf16": pkg.AFQMC_MIXED_BF16}


def _walk(name, prec, M, N, G, W, steps, energy, qr=5, comb=0, graph=1, Ndn=0):
    c = {"kind": "walk", "precision": prec, "M": M, "N": N, "nchol": G, "walkers": W,
         "steps": steps, "energy_period": energy, "qr_period": qr, "pc_period": comb,
         "graph": graph, "Ndn": Ndn}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the benchmark's default: 300 orbitals, 1800 vectors, 512 walkers, an energy every 10 steps
        _walk("walk-bf16-300", "bf16", 300, 25, 1800, 512, 10, 10),
        # the middle size, 1024 walkers: a production run of a medium molecule
        _walk("walk-bf16-100", "bf16", 100, 10, 500, 1024, 10, 10),
        # the smallest served run: every kernel is short, launches and latency count
        _walk("walk-bf16-20", "bf16", 20, 2, 100, 128, 20, 20),
        # the higher mixed precision on a ragged shape (nothing a multiple of a tile)
        _walk("walk-tf32-217", "tf32", 217, 17, 1003, 301, 10, 10),
        # the parity run in the default precision: 12 orbitals, 32 walkers, an energy every step,
        # the comb every 10, kernels launched one by one (the parameters' defaults)
        _walk("walk-fp64-12", "fp64", 12, 3, 48, 32, 10, 1, comb=10, graph=0),
        # the middle size in the default precision
        _walk("walk-fp64-100", "fp64", 100, 10, 500, 1024, 5, 5),
        # an open-shell molecule: two spin blocks, float64 only
        _walk("walk-fp64-spin-150", "fp64", 150, 13, 700, 150, 5, 5, Ndn=10),
        # a multi-determinant trial: four rotated determinants at the middle size
        {"name": "noci-bf16-100", "kind": "noci", "precision": "bf16", "M": 100, "N": 10,
         "nchol": 500, "walkers": 256, "ndet": 4, "steps": 5, "qr_period": 5},
        # ground-state densities: a window of 10 steps and its backward sweep
        {"name": "bp-bf16-100", "kind": "bp", "precision": "bf16", "M": 100, "N": 10,
         "nchol": 500, "walkers": 512, "steps": 10, "qr_period": 5},
        # several molecules of a batch at once: sizes of the batched workload
        {"name": "group-bf16", "kind": "group", "precision": "bf16", "systems": 6, "Mmin": 40,
         "Mmax": 200, "Wmin": 64, "Wmax": 1024, "shape_seed": 3000, "steps": 10},
        # requests to the server, from the arrays a client sends to the energies it gets back
        {"name": "serve-bf16", "kind": "serve", "precision": "bf16", "systems": 3, "Mmin": 20,
         "Mmax": 180, "Wmin": 128, "Wmax": 1024, "shape_seed": 4000, "steps": 50},
        # the decomposition before the walk: 5050 orbital pairs, about 500 vectors
        {"name": "mcd-pairs-100", "kind": "mcd", "M": 100, "nchol": 500, "delta": 1e-8},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: the kinds in about the proportion of the list, sizes over their whole range.
    Walkers are drawn so that a pass does no more than the largest listed one of its kind."""
    kind = rng.choice(["mixed"] * 8 + ["fp64"] * 5 + ["noci", "noci", "bp", "group", "serve", "mcd"])
    if kind in ("mixed", "fp64"):
        spin = kind == "fp64" and rng.random() < 0.35
        prec = "fp64" if kind == "fp64" else rng.choice(["bf16", "bf16", "tf32"])
        M = _log_int(rng, 20, 300 if kind == "mixed" else 180)
        N = rng.randint(2, max(2, M // 8))
        Ndn = rng.randint(1, N) if spin else 0
        G = rng.randint(3 * M, 6 * M)
        steps, most = (10, 2e12) if kind == "mixed" else (5, 1e11)
        c = _walk(None, prec, M, N, G, 1, steps, steps, comb=rng.choice([0, 0, 5]) if prec == "fp64" else 0,
                  graph=rng.choice([0, 1]), Ndn=Ndn)
        c["walkers"] = _log_int(rng, 32, int(min(2048, max(33, most / work(c)["flops"]))))
        return c
    if kind == "noci":
        M = _log_int(rng, 40, 120)
        c = {"kind": "noci", "precision": rng.choice(["bf16", "bf16", "fp64"]), "M": M,
             "N": rng.randint(5, max(5, M // 8)), "nchol": rng.randint(3 * M, 5 * M), "walkers": 1,
             "ndet": rng.randint(2, 5), "steps": 5, "qr_period": 5}
        most = 5e10 if c["precision"] == "bf16" else 1.5e10
        c["walkers"] = _log_int(rng, 32, int(min(512, max(33, most / work(c)["flops"]))))
        return c
    if kind == "bp":
        M = _log_int(rng, 30, 120)
        return {"kind": "bp", "precision": "bf16", "M": M, "N": rng.randint(2, max(2, M // 8)),
                "nchol": rng.randint(3 * M, 5 * M), "walkers": _log_int(rng, 64, 512),
                "steps": rng.randint(4, 10), "qr_period": 5}
    if kind in ("group", "serve"):
        lo, hi = (40, 200) if kind == "group" else (20, 180)
        wlo, whi = (64, 1024) if kind == "group" else (128, 1024)
        return {"kind": kind, "precision": "bf16", "systems": rng.randint(2, 6 if kind == "group" else 3),
                "Mmin": lo, "Mmax": hi, "Wmin": wlo, "Wmax": whi, "shape_seed": rng.randint(1, 10 ** 6),
                "steps": 10 if kind == "group" else 50}
    M = _log_int(rng, 30, 100)
    return {"kind": "mcd", "M": M, "nchol": rng.randint(3 * M, 5 * M), "delta": 1e-8}


# ------------------------------------------------------------------ inputs --
def _systems(case):
    """Shapes (M, N, nchol, walkers) of a batch or of a stream of requests."""
    r = np.random.Generator(np.random.PCG64(case["shape_seed"]))
    out = []
    for _ in range(case["systems"]):
        if case["kind"] == "group":
            M = int(r.choice(np.arange(case["Mmin"], case["Mmax"] + 1, 20)))
            N = M // 8
            W = int(r.choice(np.arange(case["Wmin"], case["Wmax"] + 1, 64)))
        else:
            M = int(r.integers(case["Mmin"], case["Mmax"] + 1))
            N = int(r.integers(2, max(2, M // 8) + 1))
            W = int(r.integers(case["Wmin"], case["Wmax"] + 1))
        out.append((M, N, 5 * M, W))
    return out


def _generator(seed, stream=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _amplitude(M, G):
    def spread(m, n, d):
        return m * m * sum(math.exp(-2.0 * k / d) for k in range(n))

    return 0.5 * math.sqrt(spread(12, 48, 12.0) / spread(M, G, float(M)))


def _hamiltonian(M, G, gen):
    """(h1 [M][M], L [G][M][M]) on the GPU, float64."""
    h1 = torch.triu(0.05 * torch.randn(M, M, generator=gen, device=DEV, dtype=torch.float64), 1)
    h1 = h1 + h1.T + torch.diag(torch.linspace(-2.0, 2.0, M, device=DEV, dtype=torch.float64))
    L = torch.randn(G, M, M, generator=gen, device=DEV, dtype=torch.float64).triu_()
    L *= (_amplitude(M, G) * torch.exp(-torch.arange(G, device=DEV, dtype=torch.float64) / M))[:, None, None]
    L += torch.triu(L, 1).transpose(1, 2)
    return h1, L


def _scf(h1, L, N, iterations=12):
    """Occupied orbitals [M][N] of a few damped Roothaan iterations (an RHF trial's quality is
    the user's affair; the library takes any orthonormal columns)."""
    G, M, _ = L.shape
    Lf = L.reshape(G, M * M)
    C = torch.linalg.eigh(h1)[1][:, :N]
    D = C @ C.T
    for _ in range(iterations):
        J = 2.0 * ((Lf @ D.reshape(-1)) @ Lf).reshape(M, M)
        LC = torch.matmul(L, C).permute(1, 0, 2).reshape(M, G * N)
        C = torch.linalg.eigh(h1 + J - LC @ LC.T)[1][:, :N]
        D = 0.5 * D + 0.5 * (C @ C.T)
    return C


def _inputs(case, seed):
    """Everything that ``prepare`` and ``exact`` both start from, on the GPU."""
    gen = _generator(seed)
    M, N = case["M"], case["N"]
    h1, L = _hamiltonian(M, case["nchol"], gen)
    up = _scf(h1, L, N)
    inp = {"h1": h1, "L": L, "up": up}
    if case.get("Ndn"):
        # spin-down orbitals of their own: the spin-up ones mixed slightly with the virtual space
        mix = up[:, :case["Ndn"]] + 0.02 * torch.randn(M, case["Ndn"], generator=gen, device=DEV, dtype=torch.float64)
        inp["dn"] = torch.linalg.qr(mix)[0]
    if case["kind"] == "noci":
        def rotated():
            d = up + 0.03 * torch.randn(M, N, generator=gen, device=DEV, dtype=torch.float64)
            return torch.linalg.qr(d)[0]

        nd = case["ndet"]
        inp["coef"] = np.array([1.0] + [0.3 / nd] * (nd - 1), np.complex128)
        inp["ups"] = [up] + [rotated() for _ in range(nd - 1)]
        inp["dns"] = [up] + [rotated() for _ in range(nd - 1)]
    return inp


def _params(case, seed, **kw):
    return pkg.default_params(case["M"], case["N"], case["nchol"], case["walkers"], seed=int(seed) + 1,
                              precision=PRECISION[case["precision"]], qr_period=case["qr_period"], **kw)


def _np(t):
    return t.cpu().numpy()


class _Population:
    """Device buffers into which a program reads a state's walkers and weights."""

    def __init__(self, run):
        self.run, n = run, run.p.nwalkers
        self.index = torch.arange(n, dtype=torch.int32, device=DEV)
        self.nm = run.ncols * run.p.M
        self.rows = torch.empty((n, 4 * self.nm + 2), dtype=torch.float64, device=DEV)
        self.weights = torch.empty(n, dtype=torch.float64, device=DEV)

    def read(self):
        lib, s = pkg.lib(), self.run.s
        for rc in (lib.afqmc_export_weights(s, ctypes.c_void_p(self.weights.data_ptr())),
                   lib.afqmc_pack_walkers(s, ctypes.c_void_p(self.index.data_ptr()), self.run.p.nwalkers,
                                          ctypes.c_void_p(self.rows.data_ptr()))):
            if rc != 0:
                raise RuntimeError(lib.afqmc_last_error().decode())
        k = 2 * self.nm
        return {"phi": self.rows[:, :k], "theta": self.rows[:, k:2 * k], "logov": self.rows[:, 2 * k:],
                "weights": self.weights}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mcd":
        _, L = _hamiltonian(case["M"], case["nchol"], _generator(seed))
        return {"case": case, "V": _pair_matrix(L)}
    if kind in ("group", "serve"):
        sysd = []
        for k, (M, N, G, W) in enumerate(_systems(case)):
            h1, L = _hamiltonian(M, G, _generator(seed, 1 + k))
            sysd.append((_np(h1), _np(L), _np(_scf(h1, L, N)), W))
        if kind == "serve":
            server = Server(1, precision=PRECISION[case["precision"]], chunk_steps=10, device=DEV)
            reqs = _requests(sysd, case, seed)
            need = sum(server.footprint(r) + 256 for r in reqs)
            return {"case": case, "seed": seed, "systems": sysd,
                    "server": Server(need + 4096, precision=PRECISION[case["precision"]], chunk_steps=10, device=DEV)}
        runs = []
        for k, (h1, L, C, W) in enumerate(sysd):
            c = {"M": h1.shape[0], "N": C.shape[1], "nchol": L.shape[0], "walkers": W, "qr_period": 5,
                 "precision": case["precision"]}
            p = _params(c, seed + 100 * k, energy_period=case["steps"], use_graph=1, max_records=1)
            runs.append(pkg.AfqmcRun(h1, L, C, p, device=DEV))
        return {"case": case, "group": pkg.AfqmcGroup(runs), "runs": runs, "pops": [_Population(r) for r in runs]}
    inp = _inputs(case, seed)
    h1, L = _np(inp["h1"]), _np(inp["L"])
    if kind == "noci":
        p = _params(case, seed, energy_period=0, ndet=case["ndet"], use_graph=1)
        trial = (inp["coef"], _np(torch.stack(inp["ups"])), _np(torch.stack(inp["dns"])))
        return {"case": case, "run": pkg.AfqmcRun(h1, L, trial, p, device=DEV)}
    if kind == "bp":
        p = _params(case, seed, energy_period=0, bp_steps=case["steps"])
        run = pkg.AfqmcRun(h1, L, _np(inp["up"]), p, device=DEV, stream=torch.cuda.Stream())
        return {"case": case, "run": run, "pop": _Population(run)}
    p = _params(case, seed, energy_period=case["energy_period"], pc_period=case["pc_period"],
                use_graph=case["graph"], Ndn=case["Ndn"], max_records=case["steps"] // case["energy_period"])
    trial = (_np(inp["up"]), _np(inp["dn"])) if case["Ndn"] else _np(inp["up"])
    run = pkg.AfqmcRun(h1, L, trial, p, device=DEV)
    return {"case": case, "run": run, "pop": _Population(run)}


def _requests(sysd, case, seed):
    return [Request(k, 0.0, h1, L, C, W, case["steps"], int(seed) + 1 + 100 * k, energy_period=case["steps"] // 2)
            for k, (h1, L, C, W) in enumerate(sysd)]


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case.get("steps")
    if kind == "mcd":
        L, piv, resid = pkg.afqmc_modified_cholesky_pairs(state["V"], case["M"], case["delta"], case["nchol"] + 16)
        return {"L": L, "pivots": piv}
    if kind == "serve":
        done = state["server"].run(_requests(state["systems"], case, state["seed"]), realtime=False)
        return {str(r.rid): r.energies for r in done}
    if kind == "group":
        state["group"].propagate(steps)
        state["group"].synchronize()
        return [dict(p.read(), log=r.energy_log()) for r, p in zip(state["runs"], state["pops"])]
    r = state["run"]
    if kind == "noci":
        r.propagate(steps)
        return {"eloc": r.local_energies(), "weights": r.weights()}
    if kind == "bp":
        r.bp_begin()
        r.propagate(steps)
        rho, phl, wf, wsum, n = r.bp_end()
        return dict(state["pop"].read(), rho=rho, rho_phl=phl, sum_wf=np.array([wf]), sum_w=np.array([wsum]))
    r.propagate(steps)
    return dict(state["pop"].read(), log=r.energy_log())


# -------------------------------------------------- work and tolerances -----
def _walk_flops(M, N, G, steps, energies, sweeps, ndet=1):
    """Per walker: force bias, V, the half steps, the series (order 6), overlap and Theta; the
    local energies; Gram-Schmidt."""
    pair = 2.0 * ndet if ndet > 1 else 1.0
    step = (4 * G * N * M * pair + 2 * G * M * (M + 1) + 8 * M * M * N + 48 * M * M * N
            + (8 * N ** 3 + 8 * max(0, M - N) * N * N) * pair)
    return steps * step + energies * (4 * G * N * N * M) * pair + sweeps * 8 * M * N * N


def work(case):
    kind = case["kind"]
    if kind == "mcd":
        P, G = case["M"] * (case["M"] + 1) // 2, case["nchol"]
        return {"bytes": 8.0 * (P * G * 2 + case["M"] ** 2 * G), "flops": float(P) * G * G}
    size = {"fp64": 8, "tf32": 4, "bf16": 2}[case["precision"]]
    if kind in ("group", "serve"):
        b = f = 0.0
        for M, N, G, W in _systems(case):
            n = case["steps"]
            f += W * _walk_flops(M, N, G, n, 1 if kind == "group" else 2, n // 5)
            b += n * (size * G * M * (M + 1) / 2 + 64.0 * W * N * M) + 32.0 * W * N * M
            b += 8.0 * G * M * M if kind == "serve" else 0.0
        return {"bytes": b, "flops": f}
    M, G, W, n = case["M"], case["nchol"], case["walkers"], case["steps"]
    N = case["N"] + case.get("Ndn", 0)
    nd = case.get("ndet", 1)
    sweeps = n // case["qr_period"]
    energies = {"noci": 1, "bp": n}.get(kind) or n // case["energy_period"]
    f = W * _walk_flops(M, N, G, n, energies, sweeps, nd)
    # the vectors once per step, every walker's orbitals read and written once per step, the rows
    # that are read out at the end
    b = n * (size * G * M * (M + 1) / 2.0 + 64.0 * W * N * M) + 32.0 * W * N * M
    if kind == "bp":
        f += n * W * (2 * G * M * (M + 1) + 56 * M * M * N)
        b += n * (size * G * M * (M + 1) / 2.0 + 2.0 * size * W * G)
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    """About four times the errors against float64 of listed and drawn cases.  float64: up to
    2e-13 of an output's norm (K up to a few thousand terms a sum, several steps, inverses of
    well-conditioned overlaps; a walk whose walkers wander further from the trial shows a few times
    that).  Mixed: BF16 operands up to 4.5e-3, TF32 up to 1.1e-3 (the operands' rounding, 2^-9 and
    2^-11, through a block of steps)."""
    if case["kind"] == "mcd":
        return {"rel": 2e-12, "max": 1e-9}
    if case["precision"] == "fp64":
        return {"rel": 2e-12, "max": 1e-9}
    return {"rel": 0.02, "max": 0.5} if case["precision"] == "bf16" else {"rel": 0.005, "max": 0.1}


# ------------------------------------------------ float64 in plain PyTorch --
_MASK = 0xFFFFFFFF


def _philox(c, key):
    """Philox4x32-10 words for counters c (four int64 tensors of 32-bit words)."""
    k0, k1 = key & _MASK, (key >> 32) & _MASK

    def mul(a, b):
        hi = (a * (b >> 16) + ((a * (b & 0xFFFF)) >> 16)) >> 16
        return hi & _MASK, (a * b) & _MASK

    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
    return c


def _uniform(hi, lo):
    return (((hi >> 5) * 67108864 + (lo >> 6)).double() + 0.5) * 2.0 ** -53


def _fields(seed, step, W, G):
    k = torch.arange((G + 1) // 2, device=DEV)[None, :].expand(W, -1)
    w = torch.arange(W, device=DEV)[:, None].expand_as(k)
    x = _philox((k, w, torch.full_like(k, step), torch.zeros_like(k)), seed)
    rad = torch.sqrt(-2.0 * torch.log(_uniform(x[0], x[1])))
    ang = 2.0 * math.pi * _uniform(x[2], x[3])
    return torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], -1).reshape(W, -1)[:, :G]


def _wrap(a):
    w = torch.remainder(a + math.pi, 2.0 * math.pi) - math.pi
    return torch.where(w == -math.pi, torch.full_like(w, math.pi), w)


def _cmul(phi, A):
    """A Phi for real A [M][M] and complex Phi [W][M][N]."""
    return torch.complex(torch.matmul(A, phi.real), torch.matmul(A, phi.imag))


class _Exact:
    """The phaseless walk, every quantity in float64."""

    def __init__(self, h1, L, dets, coef, sf, W, seed, dt=0.005, order=6):
        # dets[d] = the spin blocks' trial orbitals; a walker's columns are split over them when
        # there are two blocks of their own (sf = 1 and one determinant), else shared by both spins
        self.h1, self.L, self.W, self.seed, self.dt, self.order = h1, L, W, seed, dt, order
        self.G, self.M, _ = L.shape
        self.dets, self.coef, self.sf = dets, coef, sf
        self.split = len(dets) == 1 and len(dets[0]) == 2
        P = sum(V @ V.T for V in dets[0]) * (2.0 if len(dets[0]) == 1 else 1.0)
        self.c = torch.mv(L.reshape(self.G, -1), P.reshape(-1))
        Lr = L.permute(1, 0, 2).reshape(self.M, -1)
        v0 = h1 - 0.5 * (Lr @ Lr.T) + torch.tensordot(self.c, L, 1)
        self.H0p = -0.5 * float(self.c.square().sum())
        ev, U = torch.linalg.eigh(-0.5 * dt * v0)
        self.Bh = (U * torch.exp(ev)) @ U.T
        i, j = torch.triu_indices(self.M, self.M, device=DEV)
        self.Lp = L[:, i, j]
        self.unpack = torch.zeros(self.M, self.M, dtype=torch.long, device=DEV)
        self.unpack[i, j] = torch.arange(i.numel(), device=DEV)
        self.unpack[j, i] = self.unpack[i, j].clone()
        start = torch.cat(dets[0], 1) if self.split else dets[0][0]
        one = start.to(torch.complex128)[None]
        self.E_T = float(self.energies(self.overlap(one)).real[0])
        self.phi = one.expand(W, -1, -1).clone()
        self.state = self.overlap(self.phi)
        self.w = torch.ones(W, dtype=torch.float64, device=DEV)
        self.step, self.log, self.bp = 0, [], None

    def columns(self, s):
        if not self.split:
            return slice(None)
        n = self.dets[0][0].shape[1]
        return slice(0, n) if s == 0 else slice(n, None)

    def overlap(self, phi):
        """log <T|phi>, and per determinant its share of the overlap and Theta of each block."""
        logs, thetas = [], []
        for blocks in self.dets:
            la = ph = 0.0
            th = []
            for s, V in enumerate(blocks):
                f = phi[:, :, self.columns(s)]
                S = _cmul(f, V.T)
                sign, ab = torch.linalg.slogdet(S)
                mult = 2.0 if len(blocks) == 1 else 1.0
                la, ph = la + mult * ab, ph + mult * torch.angle(sign)
                th.append(torch.linalg.solve(S, f, left=False))
            logs.append(torch.complex(la, ph))
            thetas.append(th)
        lo = torch.stack(logs, 1) + torch.log(torch.as_tensor(self.coef, device=DEV).conj())[None, :]
        ref = lo.real.max(1, keepdim=True).values
        terms = torch.exp(lo - ref)
        tot = terms.sum(1)
        logov = torch.log(tot) + ref[:, 0]
        return torch.complex(logov.real, _wrap(logov.imag)), terms / tot[:, None], thetas

    def traces(self, V, th):
        """Tr(V^T L_g Theta) per walker and vector."""
        Lh = torch.matmul(V.T, self.L).reshape(self.G, -1)
        t = th.transpose(1, 2).reshape(th.shape[0], -1)
        return torch.complex(t.real @ Lh.T, t.imag @ Lh.T)

    def force(self, st):
        t = 0.0
        for d, blocks in enumerate(self.dets):
            mult = 2.0 if len(blocks) == 1 else 1.0
            t = t + st[1][:, d:d + 1] * mult * sum(self.traces(V, th) for V, th in zip(blocks, st[2][d]))
        return t

    def energies(self, st):
        e = 0.0
        for d, blocks in enumerate(self.dets):
            mult = 2.0 if len(blocks) == 1 else 1.0
            e1 = ex = tr = 0.0
            for V, th in zip(blocks, st[2][d]):
                n = V.shape[1]
                hh = (V.T @ self.h1).reshape(-1)
                t = th.transpose(1, 2).reshape(th.shape[0], -1)
                e1 = e1 + mult * torch.complex(t.real @ hh, t.imag @ hh)
                tr = tr + mult * self.traces(V, th)
                Lh = torch.matmul(V.T, self.L).reshape(self.G * n, self.M)
                part = []
                for w0 in range(0, th.shape[0], 64):
                    x = th[w0:w0 + 64]
                    T = _cmul(x, Lh).reshape(x.shape[0], self.G, n, n)
                    part.append((T * T.transpose(2, 3)).sum((1, 2, 3)))
                ex = ex + mult * torch.cat(part)
            e = e + st[1][:, d] * (e1 + 0.5 * (tr * tr).sum(1) - 0.5 * ex)
        return e

    def apply_b(self, x, phi):
        y = torch.cat([x.real, x.imag]) @ self.Lp
        s = math.sqrt(self.dt)
        V = torch.complex(-s * y[self.W:], s * y[:self.W])[:, self.unpack]
        term = _cmul(phi, self.Bh)
        acc = term
        for k in range(1, self.order + 1):
            term = torch.matmul(V, term) / k
            acc = acc + term
        return _cmul(acc, self.Bh)

    def sweep(self):
        starts = [self.columns(s) for s in range(2)] if self.split else [slice(0, self.phi.shape[2])]
        for sl in starts:
            f = self.phi[:, :, sl]
            q, r = torch.linalg.qr(f)
            d = torch.diagonal(r, dim1=1, dim2=2)
            q = q * (d / d.abs())[:, None, :]
            self.phi[:, :, sl] = torch.where((self.w != 0)[:, None, None], q, f)

    def advance(self, steps, qr, comb=0, energy=0):
        s = math.sqrt(self.dt)
        for _ in range(steps):
            alive = self.w != 0
            xi = _fields(self.seed, self.step, self.W, self.G)
            xbar = -1j * s * (self.force(self.state) - self.c)
            mag = xbar.abs()
            xbar = torch.where(mag > 1.0, xbar / mag.clamp_min(1e-300), xbar)
            x = xi - xbar
            new = self.apply_b(x, self.phi)
            st = self.overlap(new)
            logR = st[0] - self.state[0] - self.dt * (self.H0p - self.E_T) - 1j * s * (x @ self.c.to(x.dtype))
            logI = logR.real + (xi * xbar).sum(1).real - 0.5 * (xbar * xbar).sum(1).real
            cosd = torch.cos(_wrap(logR.imag))
            w = (self.w * torch.exp(logI) * cosd.clamp_min(0.0)).clamp_max(max(100.0, self.W / 10.0))
            w = torch.where(alive & torch.isfinite(w), w, torch.zeros_like(w))
            self.phi = torch.where(alive[:, None, None], new, self.phi)
            self.state = self.overlap(self.phi)
            self.w = w
            self.step += 1
            if self.bp is not None:
                f = torch.polar(torch.where(cosd > 0, 1.0 / cosd, torch.zeros_like(cosd)),
                                -self.dt * self.energies(self.state).imag)
                self.bp["factor"] = self.bp["factor"] * f
                self.bp["fields"].append(torch.where(alive[:, None], x, torch.zeros_like(x)))
            if qr and self.step % qr == 0:
                self.sweep()
                self.state = self.overlap(self.phi)
            if comb and self.step % comb == 0:
                self.comb()
            if energy and self.step % energy == 0:
                e = self.energies(self.state).real
                half = math.sqrt(2.0 / self.dt)
                e = e.clamp(self.E_T - half, self.E_T + half)
                tot = float(self.w.sum())
                self.log.append([self.step, float((self.w * e).sum()) / tot, tot, float((self.w != 0).sum())])

    def comb(self):
        one = [torch.tensor([v], device=DEV) for v in (0, _MASK, self.step - 1, 0)]
        r = _philox(tuple(one), self.seed)
        u = float(_uniform(r[0], r[1]))
        w = _np(self.w)
        cum = np.add.accumulate(w)
        teeth = ((np.arange(self.W) + u) * cum[-1]) / self.W
        parent = np.searchsorted(cum, teeth, side="right")
        parent = np.where(parent >= self.W, np.nonzero(w > 0)[0][-1], parent)
        self.phi = self.phi[torch.from_numpy(parent).to(DEV)].clone()
        self.state = self.overlap(self.phi)
        self.w = torch.full_like(self.w, cum[-1] / self.W)

    def window(self, steps, qr):
        psi = self.phi.clone()
        self.bp = {"fields": [], "factor": torch.ones(self.W, dtype=torch.complex128, device=DEV)}
        self.advance(steps, qr)
        bra = self.dets[0][0].to(torch.complex128)[None].expand(self.W, -1, -1)
        for x in reversed(self.bp["fields"]):
            bra = self.apply_b(-x.conj(), bra)
        bh = bra.conj().transpose(1, 2)
        rho = 2.0 * torch.matmul(psi, torch.linalg.solve(torch.matmul(bh, psi), bh)).transpose(1, 2)
        w, wf = self.w.to(torch.complex128), self.w * self.bp["factor"]
        return {"rho": torch.tensordot(wf, rho, 1) / wf.sum(), "rho_phl": torch.tensordot(w, rho, 1) / w.sum(),
                "sum_wf": wf.sum().reshape(1), "sum_w": w.sum().reshape(1)}

    def population(self):
        """The walkers as the state holds them: in the basis whose first columns are the (spin-up)
        trial, completed by its Householder QR, orbital by orbital, real parts first."""
        V = self.dets[0][0]
        Q = np.linalg.qr(_np(V), mode="complete")[0]
        Q[:, :V.shape[1]] = _np(V)
        QT = torch.from_numpy(np.ascontiguousarray(Q.T)).to(DEV)

        def rows(f):
            f = _cmul(f, QT).transpose(1, 2)
            return torch.stack([f.real, f.imag], 1).reshape(self.W, -1)

        return {"phi": rows(self.phi), "theta": rows(torch.cat(self.state[2][0], 2)),
                "logov": torch.view_as_real(self.state[0]), "weights": self.w}


def _exact_run(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "noci":
        dets, coef = [list(b) for b in zip(inp["ups"], inp["dns"])], inp["coef"]
    else:
        dets, coef = [[inp["up"]] + ([inp["dn"]] if case.get("Ndn") else [])], np.ones(1, np.complex128)
    return _Exact(inp["h1"], inp["L"], dets, coef, 2.0, case["walkers"], int(seed) + 1)


def _pair_matrix(L):
    """V over the pairs p <= r of the vectors L, symmetric to the last bit."""
    i, j = torch.triu_indices(L.shape[1], L.shape[1], device=DEV)
    Lp = L[:, i, j]
    V = Lp.T @ Lp
    return (V + V.T) * 0.5


def _exact_mcd(case, seed):
    M, room = case["M"], case["nchol"] + 16
    _, L = _hamiltonian(M, case["nchol"], _generator(seed))
    V = _pair_matrix(L)
    i, j = torch.triu_indices(M, M, device=DEV)
    diag = torch.diagonal(V).clone()
    zeroed = torch.zeros_like(diag, dtype=torch.bool)
    rows, piv = [], []
    X = torch.zeros(room, V.shape[0], dtype=torch.float64, device=DEV)
    for n in range(room):
        k = int(diag.argmax())
        top = float(diag[k])
        if top < case["delta"]:
            break
        zeroed |= torch.sqrt(diag.abs() * top) <= min(1e-9, case["delta"])
        v = (V[k] - X[:n, k] @ X[:n]) / math.sqrt(top)
        X[n] = torch.where(zeroed, torch.zeros_like(v), v)
        diag = torch.where(zeroed, torch.zeros_like(diag), diag - X[n] * X[n])
        piv.append(int(i[k]) * M + int(j[k]))
    out = torch.zeros(len(piv), M, M, dtype=torch.float64, device=DEV)
    out[:, i, j] = X[:len(piv)]
    out[:, j, i] = X[:len(piv)]
    return {"L": out, "pivots": torch.tensor(piv, dtype=torch.int32, device=DEV)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "mcd":
        return _exact_mcd(case, seed)
    if kind in ("group", "serve"):
        out = []
        for k, (M, N, G, W) in enumerate(_systems(case)):
            h1, L = _hamiltonian(M, G, _generator(seed, 1 + k))
            ex = _Exact(h1, L, [[_scf(h1, L, N)]], np.ones(1, np.complex128), 2.0, W, int(seed) + 1 + 100 * k)
            ex.advance(case["steps"], 5, energy=case["steps"] // (1 if kind == "group" else 2))
            out.append((dict(ex.population()) if kind == "group" else {}, np.array(ex.log)))
        if kind == "serve":
            return {str(k): log for k, (_, log) in enumerate(out)}
        return [dict(p, log=log) for p, log in out]
    ex = _exact_run(case, seed)
    if kind == "noci":
        ex.advance(case["steps"], case["qr_period"])
        return {"eloc": ex.energies(ex.state), "weights": ex.w.to(torch.complex128)}
    if kind == "bp":
        got = ex.window(case["steps"], case["qr_period"])
        return dict(ex.population(), **got)
    ex.advance(case["steps"], case["qr_period"], case["pc_period"], case["energy_period"])
    return dict(ex.population(), log=np.array(ex.log))
