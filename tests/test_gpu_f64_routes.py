"""The float64 path's routes by size against the oracle (Secs. 3.2 - 3.4): up to
64 orbitals the Taylor series runs in one block per walker, above that one
launch per term.  Sizes at the edges of the routes.  Walkers, weights,
overlaps and energies agree to the 1e-10 of the parity tests (sums of a few
thousand float64 terms and inverses of well-conditioned overlaps: about 1e-13
here)."""
import numpy as np
import pytest

import workloads
from oracle import afqmc

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
    (5, 5, 7, 3, 0),      # every orbital occupied
    (33, 9, 40, 5, 0),    # more elements of a term than threads of a block
    (64, 7, 70, 4, 0),    # the largest one-block series
    (64, 20, 30, 3, 19),  # two spin blocks, 39 columns: 144 KB of shared memory
    (64, 64, 20, 2, 0),   # the most orbitals: 192 KB
    (65, 7, 70, 4, 0),    # the smallest of the other route
])
def test_sizes(pkg, M, N, G, W, Ndn):
    check(pkg, M, N, G, W, 3, Ndn)
