"""The FP64 products on their small tiles (lambda rows on 16, 32 and 64 wide
tiles as the row count asks, per-walker products of two, four or eight rows
with many walkers per CTA) and the mixed path's M vectors with electron counts
off the groups of four: log|Psi| and e_L against the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("n_up,n_dn,W", [(2, 2, 1), (2, 1, 65), (3, 3, 17), (4, 2, 1000), (5, 4, 3), (7, 7, 700),
                                         (8, 8, 33), (5, 4, 20000)])
@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_small_products_match_oracle(torch_cuda, n_up, n_dn, W, mode):
    """FP64 at 1e-10; mixed at its 1e-6 (log|Psi|) and 1e-5 Ha (e_L).  W = 20000
    rows of L = 54 take the 32-wide lambda tiles, the others 16-wide ones."""
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=9, n_up=n_up, n_dn=n_dn, per_atom=6, seed=90 + n_up, side=4.5, Z=2.0)
    x = synth.init_walkers(sysm, W, seed=8)
    fp64 = mode == "fp64"
    g = pg.JAGP(sysm, W, precision=pg.JAGP_PREC_FP64 if fp64 else pg.JAGP_PREC_MIXED)
    r = g.positions(x)
    la, sg = g.eval(r)
    eL = g.local_energy(r)
    pick = np.unique(np.linspace(0, W - 1, 400).astype(int))
    o = oracle.Oracle(sysm)
    la_ref, sg_ref = o.logpsi_batch(x[pick])
    e_ref = o.local_energy_batch(x[pick])
    assert g.status() == 0
    assert np.array_equal(sg.cpu().numpy()[pick], sg_ref)
    assert np.allclose(la.cpu().numpy()[pick], la_ref, rtol=1e-10 if fp64 else 0.0, atol=1e-10 if fp64 else 1e-6)
    assert np.allclose(eL.cpu().numpy()[pick], e_ref, rtol=1e-9 if fp64 else 0.0, atol=1e-9 if fp64 else 1e-5)
    g.close()
