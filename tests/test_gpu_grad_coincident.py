"""Derivatives of log|Psi| with respect to the Jastrow's parameters are finite where an electron sits on a nucleus or on an
electron of the other spin (the positions' derivatives are not): against the oracle, 1e-9 of the largest component."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b_ea", [0.8, 0.0])
@pytest.mark.parametrize("where", ["nucleus", "electron", "both"])
def test_jastrow_parameters_at_coincidences(b_ea, where):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=4, n_up=4, n_dn=3, per_atom=6, seed=41)
    sysm.b_ea = b_ea
    W = 2
    x = synth.jitter_walkers(synth.init_walkers(sysm, W, seed=3), 4, 0.3)
    if where != "electron":
        x[0, 1] = sysm.R[2]
        x[1, 5] = sysm.R[0]
    if where != "nucleus":
        x[0, 6] = x[0, 3]
    seeds = np.array([0.7, -1.3])
    o = oracle.Oracle(sysm)
    ref = sum(s * o.grad_logpsi(x[w])["jas"] for w, s in enumerate(seeds))
    assert np.isfinite(ref).all()
    g = pg.JAGP(sysm, W)
    r = g.positions(x)
    g.eval(r)
    jas = g.grad(r, seed_logpsi=torch.tensor(seeds, device="cuda"))["jas"].cpu().numpy()
    g.close()
    assert np.all(np.abs(jas - ref) <= 1e-9 * max(1.0, np.abs(ref).max())), (jas, ref)
