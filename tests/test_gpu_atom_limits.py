"""More atoms than the orbital kernels can hold in shared memory (9800; few of them have shells), against the oracle at the
parity bars of the two paths: 1e-10 relative in FP64; 1e-6 in log|Psi| and 1e-5 in e_L in mixed precision."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _case(na):
    """A grid of weak charges, two s shells on each of eight atoms in its middle; three walkers near those."""
    g = np.random.default_rng(na)
    side = int(np.ceil(na ** (1 / 3)))
    R = 2.0 * np.stack(np.unravel_index(np.arange(na), (side,) * 3), axis=1).astype(np.float64)
    mid = na // 2 + np.arange(8)
    lam = np.eye(16) + 0.05 * g.normal(size=(16, 16))
    sysm = synth.System(f"grid({na})", R, np.full(na, 0.01), np.repeat(mid, 2).astype(np.int32), np.zeros(16, np.int32),
                        np.arange(16, dtype=np.int32) % 2, 0.3 + 0.5 * g.random(16), 0.5 * (lam + lam.T), 2, 2,
                        unpaired=None, b_ea=0.8, b_para=1.3, b_anti=0.7, use_j1=True, use_j2=True,
                        j2_spin_independent=False, delta=0.5, seed=na).check()
    x = R[mid[[0, 2, 4, 6]]] + g.uniform(-1.0, 1.0, size=(3, 4, 3))
    return sysm, x


def _handle(sysm, prec, W):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    return pg.JAGP(sysm, W, precision=pg.JAGP_PREC_MIXED if prec == "mixed" else pg.JAGP_PREC_FP64)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_orbitals(prec):
    sysm, x = _case(9800)
    la_ref, sg_ref = oracle.Oracle(sysm).logpsi_batch(x)
    h = _handle(sysm, prec, len(x))
    la, sg = h.eval(h.positions(x))
    tol = 1e-6 if prec == "mixed" else 1e-10
    assert np.all(np.abs(la.cpu().numpy() - la_ref) <= tol * np.maximum(1.0, np.abs(la_ref)))
    assert np.array_equal(sg.cpu().numpy(), sg_ref)
    h.close()


# mixed precision: about as many atoms as shared memory holds the constants of (4100 and three walkers of four electrons
# are beside it with the electrons' sums), and far more
@pytest.mark.parametrize("prec,na", [("fp64", 9800), ("mixed", 3700), ("mixed", 4100), ("mixed", 9800)])
def test_local_energy(prec, na):
    sysm, x = _case(na)
    e_ref = oracle.Oracle(sysm).local_energy_batch(x)
    h = _handle(sysm, prec, len(x))
    r = h.positions(x)
    h.eval(r)
    e = h.local_energy(r).cpu().numpy()
    tol = 1e-5 if prec == "mixed" else 1e-10
    assert np.all(np.abs(e - e_ref) <= tol * np.maximum(1.0, np.abs(e_ref)))
    h.close()
