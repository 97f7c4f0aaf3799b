"""Three-body Jastrow at the size where the acceptance kernel's shared memory holds G~^{-1} only without its padded rows
(even N_up: 154 with 39 to 55 Jastrow functions in FP64): a sweep follows the oracle's move by move.  Energies at 1e-8:
G~ has a condition number of 3e6 here.  Below the limit (38) nothing changes."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_atoms", [38, 39, 55])
def test_sweep_at_the_limit(n_atoms):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=n_atoms, n_up=154, n_dn=154, per_atom=16, seed=77, side=12.0, Z=2.0)
    sysm = synth.with_j3(sysm, seed=5, per_atom=(1, 0), sd=0.02)
    W = 2
    x0 = synth.jitter_walkers(synth.init_walkers(sysm, W, seed=3), 4, 0.3)
    xo = x0.copy()
    eL_ref, lp_ref, _ = oracle.Oracle(sysm).vmc(xo, 1, seed=5)
    g = pg.JAGP(sysm, W, seed=5)
    r = g.positions(x0)
    g.eval(r)
    eL, _ = g.sweep(r, 1)
    assert np.array_equal(r.cpu().numpy(), xo)
    e, la = eL.cpu().numpy(), g.info()["logabs"].cpu().numpy()
    assert np.all(np.abs(e - eL_ref) <= 1e-8 * np.maximum(1.0, np.abs(eL_ref)))
    assert np.all(np.abs(la - lp_ref) <= 1e-9 * np.maximum(1.0, np.abs(lp_ref)))
    g.close()
