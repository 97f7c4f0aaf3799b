"""Hop ratios where a hop lands close to a nucleus or to another electron (down to on top of it), against the oracle's
determinants: 1e-10 of the ratio (or of 1), as for the generations.  Jastrow terms and Slater shells change with the
distance itself there, so an error of 2^-46 (r^2 + a^2) in its square would show as up to 1e-8."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _ratios(pg, torch, g, r, a):
    """rho [W][6 N] of the configurations: a projection without hops, then the workspace's fourth array (after three of
    W numbers, each padded to 256 bytes)."""
    W, N = r.shape[0], r.shape[1]
    work = torch.zeros(pg.jagp_lrdmc_workspace_bytes(g.h, W), dtype=torch.uint8, device="cuda")
    w = torch.ones(W, dtype=torch.float64, device="cuda")
    pg.jagp_lrdmc_project(g.h, r, g.state, W, work, w, a=a, tau=1.0, max_hops=0)
    off = 3 * ((8 * W + 255) // 256 * 256)
    return work[off:off + 8 * W * 6 * N].view(torch.float64).reshape(W, 6 * N).cpu().numpy()


@pytest.mark.parametrize("slater", [0.0, 0.5])
@pytest.mark.parametrize("a", [0.05, 0.2])
@pytest.mark.parametrize("eps", [0.0, 1e-7, 1e-4, 0.1, 0.4])
def test_hops_onto_a_centre(a, slater, eps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=3, n_up=3, n_dn=2, per_atom=20, seed=41, slater_fraction=slater, Z=2.0)
    tight = np.flatnonzero(sysm.shell_radial == 0)[::3]  # exponents whose zeta a^2 is up to 60
    sysm.shell_zeta[tight] = np.geomspace(5.0, 60.0 / a ** 2, len(tight))
    rng = np.random.default_rng(5)
    cases = []
    for k in range(6):
        for target in ("atom", "electron"):
            x = synth.jitter_walkers(synth.init_walkers(sysm, 1, seed=k), k, 0.3)[0]
            e = k % 5
            c = sysm.R[k % 3] if target == "atom" else x[(e + 2) % 5]
            u = rng.normal(size=3)
            x[e] = c + eps * a * u / np.linalg.norm(u)  # where the hop is to land
            x[e, k // 2] -= -a if k & 1 else a
            cases.append(x)
    x = np.ascontiguousarray(cases)
    g = pg.JAGP(sysm, len(cases))
    rho = _ratios(pg, torch, g, g.positions(x), a)
    g.close()
    o = oracle.Oracle(sysm)
    for w in range(len(cases)):
        ref = o.lrdmc_hops(x[w], a)[0]
        assert np.all(np.abs(rho[w] - ref) <= 1e-10 * np.maximum(1.0, np.abs(ref))), (w, np.abs(rho[w] - ref).max())
