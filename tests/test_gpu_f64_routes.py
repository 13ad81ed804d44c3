"""The float64 path's routes by size against the oracle (Secs. 3.2 - 3.4): small
systems run the Taylor series in one block per walker, the others every
contraction as exact integer products on the tensor cores.  Sizes at the edges
of the routes and of the tiles.  Walkers, weights,
overlaps and energies agree to the 1e-10 of the parity tests (sums of a few
thousand float64 terms and inverses of well-conditioned overlaps: about 1e-13
here)."""
import numpy as np
import pytest

import workloads
from oracle import afqmc, multidet, smw

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1711_02242_gb300 as p

    return p


def inputs(M, N, G, Ndn=0):
    """Hamiltonian and orthonormal trial orbitals (the lowest ones of h1; the
    spin-down ones of a two-block walker slightly rotated)."""
    h1, L, _ = workloads.hamiltonian(M, G, 9000 + M, l_scale=workloads.l_amplitude(M, G))
    C = np.linalg.eigh(h1)[1]
    if not Ndn:
        return h1, L, C[:, :N]
    rng = np.random.default_rng(M)
    dn = np.linalg.qr(C[:, :Ndn] + 0.03 * rng.standard_normal((M, Ndn)))[0]
    return h1, L, (C[:, :N], dn)


def check(pkg, M, N, G, W, steps, Ndn=0):
    h1, L, trial = inputs(M, N, G, Ndn)
    up, dn = trial if Ndn else (trial, None)
    orc = afqmc.Oracle(h1, L, up, W, afqmc.Params(qr_period=2, energy_period=1), trial_dn=dn)
    p = pkg.default_params(M, N, G, W, qr_period=2, energy_period=1, Ndn=Ndn)
    run = pkg.AfqmcRun(h1, L, trial, p)
    run.propagate(steps)
    orc.run(steps)
    phi, wt, lo = run.get_walkers()
    assert np.all(orc.weight > 0)
    err = np.linalg.norm((phi - orc.phi).reshape(W, -1), axis=1) / np.linalg.norm(orc.phi.reshape(W, -1), axis=1)
    assert err.max() < TOL
    assert np.max(np.abs(wt - orc.weight) / orc.weight) < TOL
    assert np.max(np.abs(lo - orc.logdet)) < TOL * (1 + np.abs(orc.logdet).max())
    E = np.array([r[1] / r[2] for r in orc.records])
    assert np.max(np.abs(run.energy_log()[:, 1] - E) / np.abs(E)) < TOL
    el = orc.local_energies()
    assert np.max(np.abs(run.local_energies() - el) / np.abs(el)) < TOL
    assert run.info().status == 0
    run.close()


@pytest.mark.parametrize("M,N,G,W,Ndn", [
    # float64 kernels, the series in one block per walker
    (5, 5, 7, 3, 0),       # every orbital occupied
    (33, 9, 40, 5, 0),     # more elements of a term than threads of a block
    (39, 20, 30, 3, 19),   # two spin blocks
    (35, 2, 30, 3, 0),     # the most orbitals
    (28, 2, 33, 512, 0),   # with many walkers
    (27, 20, 30, 3, 0),    # Gram-Schmidt alone from the Gram matrix
    # tensor cores
    (28, 4, 57, 4, 0),     # the fewest orbitals
    (36, 1, 30, 3, 0),     # the fewest for a single column
    (40, 5, 57, 4, 0),     # columns of a term: one 16-wide tile
    (64, 32, 90, 3, 0),    # a walker fills the exchange's column tile
    (64, 64, 20, 2, 0),    # every orbital occupied, two column tiles, float64 exchange kernel
    (70, 1, 30, 130, 0),   # 32 walkers per column tile of the exchange, 128 vectors per row tile
    (129, 17, 401, 3, 0),  # two row tiles of V; one vector more than a segment of the sum
    (130, 33, 150, 3, 0),  # the fewest orbitals with two column tiles
    (150, 13, 300, 3, 10),  # two spin blocks
])
def test_sizes(pkg, M, N, G, W, Ndn):
    check(pkg, M, N, G, W, 3, Ndn)


@pytest.mark.parametrize("M,N,W,Ndn,nd,precision", [
    (40, 5, 6, 0, 0, 0), (60, 17, 6, 15, 0, 0), (70, 6, 6, 0, 2, 0), (100, 10, 200, 0, 0, 2), (70, 6, 6, 0, 2, 2)])
def test_least_workspace(pkg, M, N, W, Ndn, nd, precision):
    """A state in the least workspace it can do with walks the same walk to rounding
    (float64: a few hundred products a sum, 1e-10; mixed: the float64 overlaps and
    Gram-Schmidt differ by 1e-14, which a BF16 operand may round to another
    neighbour, 2^-8 of its size), and a byte less is refused."""
    import torch

    G = 60
    h1, L, trial = inputs(M, N, G, Ndn)
    if nd:
        rng = np.random.default_rng(M)
        dets = np.array([trial] + [np.linalg.qr(trial + 0.05 * rng.standard_normal((M, N)))[0] for _ in range(1, nd)])
        trial = (np.array([1.0] + [0.3] * (nd - 1), complex), dets, dets)
    p = pkg.default_params(M, N, G, W, qr_period=2, energy_period=0, Ndn=Ndn, ndet=nd, precision=precision,
                           bp_steps=0 if Ndn or nd else 2)
    size, least = pkg.afqmc_workspace_size(p), pkg.afqmc_workspace_size_min(p)
    assert least < size
    out = []
    for n in (size, size - 256, least):
        run = pkg.AfqmcRun(h1, L, trial, p, workspace=torch.empty(n, dtype=torch.uint8, device="cuda"))
        assert bool(run.sliced_routes()) == (n == size)
        run.propagate(3)
        phi, wt, lo = run.get_walkers()
        out.append([phi, wt, lo, run.local_energies()])
        if p.bp_steps:
            run.bp_begin()
            run.propagate(2)
            out[-1] += list(run.bp_end()[:2])
        assert run.info().status == 0
        run.close()
    for a, b, c in zip(*out):
        assert np.array_equal(b, c)  # a little too small for the slices, or by all of them
        assert np.max(np.abs(a - c)) < (TOL if precision == 0 else 2.0 ** -8) * (1 + np.abs(a).max())
    with pytest.raises(pkg.AfqmcError, match="ENOSPC"):
        pkg.AfqmcRun(h1, L, trial, p, workspace=torch.empty(least - 1, dtype=torch.uint8, device="cuda"))


def test_allocation_that_fails(pkg, monkeypatch):
    """Where the workspace a state uses cannot be allocated, one it can do with is."""
    import torch

    h1, L, C = inputs(40, 5, 60)
    p = pkg.default_params(40, 5, 60, 6, energy_period=0)
    size, least, empty = pkg.afqmc_workspace_size(p), pkg.afqmc_workspace_size_min(p), torch.empty

    def bounded(n, *a, **kw):
        if isinstance(n, int) and n >= size:
            raise torch.cuda.OutOfMemoryError("no room")
        return empty(n, *a, **kw)

    monkeypatch.setattr(torch, "empty", bounded)
    run = pkg.AfqmcRun(h1, L, C, p)
    assert run.ws.numel() == least + 256 and run.sliced_routes() == 0
    run.propagate(2)
    assert run.info().status == 0
    run.close()


@pytest.mark.parametrize("M,N,precision,qr", [(32, 2, 0, 5), (32, 4, 0, 2), (36, 2, 0, 5), (32, 4, 2, 2), (100, 10, 2, 2)])
def test_population_whole_or_split(pkg, M, N, precision, qr):
    """The arithmetic does not depend on the number of walkers: a state of 520 and
    two of 460 and 60 that draw its fields walk the same walk, bit for bit."""
    G = 40
    h1, L, C = inputs(M, N, G)
    out = []
    for n, w0 in ((520, 0), (460, 0), (60, 460)):
        p = pkg.default_params(M, N, G, n, qr_period=qr, energy_period=0, walker0=w0, precision=precision)
        run = pkg.AfqmcRun(h1, L, C, p)
        run.propagate(5)
        out.append((*run.get_walkers(), run.local_energies()))
        run.close()
    for whole, a, b in zip(*out):
        assert np.array_equal(whole, np.concatenate([a, b]))


def test_chunks_of_walkers(pkg):
    """Populations whose sliced operands exceed the scratch area are taken in
    chunks: the last walkers of 40000 are those of a small population that
    draws the same fields."""
    M, N, G, W, n = 40, 2, 50, 40000, 70
    h1, L, C = inputs(M, N, G)
    big = pkg.AfqmcRun(h1, L, C, pkg.default_params(M, N, G, W, qr_period=2, energy_period=0))
    small = pkg.AfqmcRun(h1, L, C, pkg.default_params(M, N, G, n, qr_period=2, energy_period=0, walker0=W - n))
    for r in (big, small):
        r.propagate(3)
    el = big.local_energies()
    assert np.array_equal(el[-n:], small.local_energies())
    assert np.array_equal(big.weights()[-n:], small.weights())
    assert np.all(np.isfinite(el)) and np.unique(el).size == W
    big.close()
    small.close()


@pytest.mark.parametrize("M,N,nd,kind,precision", [
    (40, 5, 3, "noci", 0),    # one 16-wide column tile
    (70, 33, 2, "noci", 0),   # two column tiles of Theta, 132 rows of the trial's orbitals
    (130, 6, 2, "noci", 0),   # two row tiles of Phi
    (40, 3, 33, "noci", 0),   # one determinant more than the lanes of a warp
    (44, 6, 4, "ci", 0),      # relative to determinant 0: its overlap alone
    (44, 6, 3, "noci", 2),    # the mixed path keeps these float64
])
def test_determinants(pkg, M, N, nd, kind, precision):
    """Overlaps and Theta of every determinant, against the oracles' walks.  The
    mixed path against the float64 one from the same perturbed walkers: overlaps to
    the 1e-10 of float64, local energies (BF16 exchange and traces) to 2^-8 of their
    terms, three steps' walkers to a few 2^-9 and weights to some more (sums of
    products of rounded fields and vectors)."""
    G, W = 50, 5
    h1, L, C = inputs(M, N, G)
    rng = np.random.default_rng(M + nd)
    full = np.linalg.qr(np.hstack([C, rng.standard_normal((M, M - N))]))[0]
    ups, dns = [C], [C]
    for d in range(1, nd):
        if kind == "ci":
            u, v = C.copy(), C.copy()
            u[:, d] = full[:, N + d]
            v[:, 0] = full[:, N + 2 * d]
        else:
            u, v = (np.linalg.qr(C + 0.05 * rng.standard_normal((M, N)))[0] for _ in range(2))
        ups.append(u)
        dns.append(v)
    ups, dns = np.array(ups), np.array(dns)
    coef = np.array([1.0] + [0.2 / d + 0.1j for d in range(1, nd)])
    Orc = smw.SMWOracle if kind == "ci" else multidet.MultiDetOracle
    orc = Orc(h1, L, coef, ups, dns, W, afqmc.Params(qr_period=2, energy_period=1))
    p = pkg.default_params(M, N, G, W, qr_period=2, energy_period=1, ndet=nd, precision=precision)
    run = pkg.AfqmcRun(h1, L, (coef, ups, dns), p)
    if precision:
        ref = pkg.AfqmcRun(h1, L, (coef, ups, dns), pkg.default_params(M, N, G, W, qr_period=2, energy_period=1, ndet=nd))
        phi = orc.phi + 0.02 * (rng.standard_normal(orc.phi.shape) + 1j * rng.standard_normal(orc.phi.shape))
        for steps in (0, 3):
            for r in (run, ref):
                r.set_walkers(phi, np.ones(W))
                r.propagate(steps)
            (p1, w1, l1), (p2, w2, l2) = run.get_walkers(), ref.get_walkers()
            e1, e2 = run.local_energies(), ref.local_energies()
            assert np.max(np.abs(e1 - e2) / np.abs(e2)) < 2.0 ** -8
            if steps == 0:
                assert np.max(np.abs(l1 - l2)) < TOL * (1 + np.abs(l2).max())
            else:
                assert np.max(np.abs(p1 - p2)) < 2.0 ** -6 * np.abs(p2).max()
                assert np.max(np.abs(w1 - w2) / np.abs(w2)) < 2.0 ** -5
        assert run.info().status == 0
        run.close()
        ref.close()
        return
    run.propagate(3)
    orc.run(3)
    phi, wt, lo = run.get_walkers()
    assert np.max(np.abs(phi - orc.phi)) < TOL * np.abs(orc.phi).max()
    assert np.max(np.abs(wt - orc.weight) / orc.weight) < TOL
    assert np.max(np.abs(lo - orc.logdet)) < TOL * (1 + np.abs(orc.logdet).max())
    el = orc.local_energies()
    assert np.max(np.abs(run.local_energies() - el) / np.abs(el)) < TOL
    assert run.info().status == 0
    run.close()


@pytest.mark.parametrize("M,N,Ndn", [(48, 6, 0), (60, 13, 0), (130, 25, 0), (60, 17, 15)])
def test_gram_schmidt_routes(pkg, M, N, Ndn):
    """Gram-Schmidt of well-conditioned walkers (from the Gram matrix) and of
    walkers with nearly parallel columns (the sweep) in one population, and the sweep
    alone for few columns: Q is
    orthonormal to rounding, and walkers, overlaps and weights follow the
    oracle's modified Gram-Schmidt.  The nearly parallel columns' condition
    number is about 1e3, so 1e-10 leaves their 1e-13 room."""
    G, W = 60, 5
    h1, L, trial = inputs(M, N, G, Ndn)
    up, dn = trial if Ndn else (trial, None)
    both = np.hstack([up, dn]) if Ndn else up
    rng = np.random.default_rng(3 * M)
    Nt = N + Ndn
    phi = np.repeat(both[None], W, 0).astype(complex)
    phi += 0.02 * (rng.standard_normal(phi.shape) + 1j * rng.standard_normal(phi.shape))
    for w in (1, 4):
        phi[w, :, N - 1] = phi[w, :, 0] + 1e-3 * phi[w, :, N - 1]
    orc = afqmc.Oracle(h1, L, up, W, afqmc.Params(qr_period=1, energy_period=0, fb_cap=1.0), trial_dn=dn, phi0=phi)
    p = pkg.default_params(M, N, G, W, qr_period=1, energy_period=0, Ndn=Ndn)
    run = pkg.AfqmcRun(h1, L, trial, p)
    run.set_walkers(phi, np.ones(W))
    run.propagate(1)
    orc.run(1)
    got, wt, lo = run.get_walkers()
    assert np.all(orc.weight > 0)
    for a, b in ((0, N), (N, Nt))[:2 if Ndn else 1]:
        S = np.einsum("wpi,wpj->wij", got[:, :, a:b].conj(), got[:, :, a:b])
        assert np.abs(S - np.eye(b - a)).max() < 1e-12
        assert np.abs(S[[0, 2, 3]] - np.eye(b - a)).max() < 1e-14
    assert np.abs(got - orc.phi).max() < TOL
    assert np.max(np.abs(wt - orc.weight) / orc.weight) < TOL
    assert np.max(np.abs(lo - orc.logdet)) < TOL * (1 + np.abs(orc.logdet).max())
    run.close()


@pytest.mark.parametrize("M,N,Ndn,nd,precision", [
    (48, 12, 0, 0, 0),    # Gram-Schmidt by the sweep
    (70, 16, 0, 0, 0),    # and from the Gram matrix
    (60, 17, 15, 0, 0),   # two spin blocks
    (70, 6, 0, 3, 0),     # three determinants
    (130, 25, 0, 0, 2),   # the mixed path's Gram-Schmidt
    (130, 25, 0, 2, 2),   # and its overlaps of several determinants
])
def test_orbitals_of_unequal_norm(pkg, M, N, Ndn, nd, precision):
    """Multiplying a walker's orbitals by powers of two (2^-30 .. 2^30, different for
    each) scales every product of a step by powers of two and changes nothing else:
    the same local energies, and after a step and Gram-Schmidt the same walkers,
    weights and overlaps, to the rounding of the overlaps' logarithms (|log| up to
    20 N: 1e-13); Q orthonormal to rounding."""
    G, W = 60, 6
    h1, L, trial = inputs(M, N, G, Ndn)
    up, dn = trial if Ndn else (trial, None)
    both = np.hstack([up, dn]) if Ndn else up
    Nt = N + Ndn
    rng = np.random.default_rng(5 * M)
    if nd:
        dets = np.array([up] + [np.linalg.qr(up + 0.05 * rng.standard_normal((M, N)))[0] for _ in range(1, nd)])
        trial = (np.array([1.0] + [0.3] * (nd - 1), complex), dets, dets)
    phi = np.repeat(both[None], W, 0).astype(complex)
    phi += 0.02 * (rng.standard_normal(phi.shape) + 1j * rng.standard_normal(phi.shape))
    scale = 2.0 ** rng.integers(-30, 31, (W, 1, Nt))
    scale[:, :, 0], scale[:, :, N - 1] = 2.0 ** -30, 2.0 ** 30
    out = []
    for ph in (phi, phi * scale):
        p = pkg.default_params(M, N, G, W, qr_period=1, energy_period=0, Ndn=Ndn, ndet=nd, precision=precision)
        run = pkg.AfqmcRun(h1, L, trial, p)
        run.set_walkers(ph, np.ones(W))
        el = run.local_energies()
        run.propagate(1)
        got, wt, lo = run.get_walkers()
        assert run.info().status == 0 and np.all(np.abs(wt) > 0)
        for a, b in ((0, N), (N, Nt)):
            S = np.einsum("wpi,wpj->wij", got[:, :, a:b].conj(), got[:, :, a:b])
            assert b == a or np.abs(S - np.eye(b - a)).max() < 1e-14
        out.append((el, got, wt, lo))
        run.close()
    (el, got, wt, lo), (el2, got2, wt2, lo2) = out
    assert np.max(np.abs(el2 - el) / np.abs(el)) < 1e-13
    assert np.max(np.abs(got2 - got)) < 1e-13
    assert np.max(np.abs(wt2 - wt) / np.abs(wt)) < 1e-11
    assert np.max(np.abs(lo2 - lo)) < 1e-11


@pytest.mark.parametrize("M,N,G,W,m,qr", [
    (40, 5, 57, 41, 3, 2),    # a group of 40 walkers and one of a single walker
    (65, 13, 70, 15, 2, 0),   # two row tiles of A, the last group full
    (100, 33, 60, 13, 2, 1),  # rows of the last tile short; K not a multiple of 16, QR by the sweep
    (44, 5, 50, 6, 0, 5),     # an empty window, fewer walkers than a group
])
def test_densities(pkg, M, N, G, W, m, qr):
    """The back-propagated densities from groups of walkers, against the oracle's window."""
    h1, L, C = inputs(M, N, G)
    orc = afqmc.Oracle(h1, L, C, W, afqmc.Params(qr_period=qr, energy_period=0))
    p = pkg.default_params(M, N, G, W, qr_period=qr, energy_period=0, bp_steps=4)
    run = pkg.AfqmcRun(h1, L, C, p)
    orc.run(2)
    run.propagate(2)
    orc.bp_begin()
    run.bp_begin()
    orc.run(m)
    run.propagate(m)
    want, got = orc.bp_end(), run.bp_end()
    scale = max(1.0, np.abs(want[0]).max(), np.abs(want[1]).max())
    for a, b in zip(got[:4], want[:4]):
        assert np.max(np.abs(a - b)) < TOL * max(scale, np.max(np.abs(b)))
    assert np.count_nonzero(orc.weight) > W // 2
    run.close()


def test_densities_of_chunks(pkg):
    """More groups than one launch takes: the sums of a population are those of
    its two halves (which draw the same fields), and bit for bit repeatable."""
    M, N, G, W = 40, 2, 50, 12000
    h1, L, C = inputs(M, N, G)

    def densities(n, walker0):
        p = pkg.default_params(M, N, G, n, qr_period=2, energy_period=0, bp_steps=2, walker0=walker0)
        run = pkg.AfqmcRun(h1, L, C, p)
        run.bp_begin()
        run.propagate(2)
        out = run.bp_end()
        run.close()
        return out

    whole, again, a, b = densities(W, 0), densities(W, 0), densities(7000, 0), densities(5000, 7000)
    assert np.array_equal(whole[0], again[0]) and np.array_equal(whole[1], again[1])
    for k in (0, 1):
        ref = (a[k] * a[2 + k] + b[k] * b[2 + k]) / (a[2 + k] + b[2 + k])
        assert np.max(np.abs(whole[k] - ref)) < TOL * max(1.0, np.abs(ref).max())
