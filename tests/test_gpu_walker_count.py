"""log|Psi|, its sign and e_L of a walker do not depend on how many other walkers there are, bit for bit: walkers may be
spread over processes.  The sizes are those at which kernels share a walker's work between threads or CTAs differently."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_up,n_dn,n_atoms,W", [(1, 1, 2, 2048), (5, 4, 4, 2048), (16, 16, 16, 2048), (23, 23, 12, 2048),
                                                 (33, 32, 8, 1500), (70, 70, 12, 400), (140, 140, 12, 400)])
@pytest.mark.parametrize("prec", ["fp64", "fp64_tc", "mixed"])
def test_values_of_few_among_many(prec, n_up, n_dn, n_atoms, W):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=n_atoms, n_up=n_up, n_dn=n_dn, per_atom=20, seed=51, side=2.5 * n_atoms ** (1 / 3),
                              Z=2.0)
    x = synth.jitter_walkers(synth.init_walkers(sysm, W, seed=3), 4, 0.3)
    out = []
    for count in (W, 16, 1):
        g = pg.JAGP(sysm, count, precision=pg.JAGP_PREC_MIXED if prec == "mixed" else pg.JAGP_PREC_FP64,
                    fp64_tc=prec == "fp64_tc")
        r = g.positions(x[:count])
        la, sg = g.eval(r)
        out.append([t.cpu().numpy() for t in (la, sg, g.local_energy(r))])
        g.close()
    for few in out[1:]:
        for a, b in zip(out[0], few):
            assert np.array_equal(a[:len(b)], b, equal_nan=True)
