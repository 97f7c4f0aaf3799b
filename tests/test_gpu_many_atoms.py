"""Orbitals and kinetic terms with so many atoms that a warp's table of displacements takes most of shared memory (600
atoms: four warps per CTA) or does not fit (3000: the displacement is formed per shell), against the oracle at the
parity bars of the two paths: 1e-10 relative in FP64; 1e-6 in log|Psi| and 1e-5 in e_L in mixed precision."""
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


def _system(na):
    g = np.random.default_rng(na)
    side = int(np.ceil(na ** (1 / 3)))
    R = 2.0 * np.stack(np.unravel_index(np.arange(na), (side,) * 3), axis=1).astype(np.float64)
    lam = np.eye(na) + 0.01 * g.normal(size=(na, na))
    return synth.System(f"grid({na})", R, np.full(na, 0.01), np.arange(na, dtype=np.int32), np.zeros(na, np.int32),
                        np.zeros(na, np.int32), 0.3 + 0.5 * g.random(na), 0.5 * (lam + lam.T), 2, 2, unpaired=None,
                        b_ea=0.8, b_para=1.3, b_anti=0.7, use_j1=True, use_j2=True, j2_spin_independent=False, delta=0.5,
                        seed=na).check()


@pytest.mark.parametrize("na", [600, 3000])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_many_atoms(torch_cuda, na, prec):
    import paper_2002_07401_gb300 as pg
    sysm = _system(na)
    W = 3
    g = np.random.default_rng(1)
    x = sysm.R[g.integers(0, na, size=(W, 4))] + g.uniform(-1.0, 1.0, size=(W, 4, 3))
    o = oracle.Oracle(sysm)
    la_ref, sg_ref = o.logpsi_batch(x)
    e_ref = o.local_energy_batch(x)
    h = pg.JAGP(sysm, W, precision=pg.JAGP_PREC_MIXED if prec == "mixed" else pg.JAGP_PREC_FP64)
    r = h.positions(x)
    la, sg = h.eval(r)
    e = h.local_energy(r).cpu().numpy()
    tl, te = (1e-6, 1e-5) if prec == "mixed" else (1e-10, 1e-10)
    assert np.all(np.abs(la.cpu().numpy() - la_ref) <= tl * np.maximum(1.0, np.abs(la_ref)))
    assert np.array_equal(sg.cpu().numpy(), sg_ref)
    assert np.all(np.abs(e - e_ref) <= te * np.maximum(1.0, np.abs(e_ref)))
    h.close()
