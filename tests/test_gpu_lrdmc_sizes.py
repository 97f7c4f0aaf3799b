"""Hop ratios where the walker's positions and the atoms take about 48 KB of shared memory, more, and more than there is:
against ratios of log|Psi| and its sign at the hopped positions.  log|Psi| sums half a million one-body terms in FP64, so
that its rounding is within 1e-12 of its size (5e5), and the ratios agree to that."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _system(n_atoms, n_up):
    """Atoms on a cubic grid, one s Gaussian each, a pairing matrix near the identity."""
    rng = np.random.default_rng(n_atoms)
    side = int(np.ceil(n_atoms ** (1 / 3)))
    R = 3.0 * np.array([(i // side ** 2, i // side % side, i % side) for i in range(n_atoms)], dtype=np.float64)
    lam = rng.normal(0.0, 0.02, size=(n_atoms, n_atoms))
    lam = np.eye(n_atoms) + 0.5 * (lam + lam.T)
    z = np.zeros(n_atoms, np.int32)
    return synth.System(f"grid({n_atoms})", R, np.ones(n_atoms), np.arange(n_atoms, dtype=np.int32), z, z,
                        rng.uniform(0.1, 0.4, n_atoms), lam, n_up, n_up, unpaired=None, b_ea=0.8, b_para=1.3,
                        b_anti=0.7, delta=0.5, seed=1).check()


@pytest.mark.parametrize("n_atoms,n_up", [(760, 380), (764, 382), (768, 384), (900, 450), (5300, 1)])
def test_ratios_of_many_atoms(n_atoms, n_up):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm, a, W = _system(n_atoms, n_up), 0.2, 1
    x = synth.init_walkers(sysm, W, seed=3, spread=0.7)
    g = pg.JAGP(sysm, 24)
    r = g.positions(x)
    work = torch.zeros(pg.jagp_lrdmc_workspace_bytes(g.h, W), dtype=torch.uint8, device="cuda")
    w = torch.ones(W, dtype=torch.float64, device="cuda")
    pg.jagp_lrdmc_project(g.h, r, g.state, W, work, w, a=a, tau=1.0, max_hops=0)
    N = 2 * n_up
    rho = work[768:768 + 8 * 6 * N].view(torch.float64).cpu().numpy()  # after three padded arrays of W numbers
    ks = sorted(set(np.linspace(0, 6 * N - 1, 23).astype(int)))
    y = np.repeat(x, len(ks) + 1, axis=0)
    for j, k in enumerate(ks):
        y[j + 1, k // 6, k % 6 // 2] += -a if k & 1 else a
    la, sg = (t.cpu().numpy() for t in g.eval(g.positions(y)))
    g.close()
    ref = sg[1:] * sg[0] * np.exp(la[1:] - la[0])
    assert np.isfinite(ref).all()
    tol = 1e-12 * max(1.0, np.abs(la).max()) * np.maximum(1.0, np.abs(ref))
    assert np.all(np.abs(rho[ks] - ref) <= tol), np.abs(rho[ks] - ref).max()
