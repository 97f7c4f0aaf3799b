"""State and workspace sizes never fall as the walker count grows: a buffer for the most walkers serves fewer."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_up,n_dn,atoms,per_atom", [(2, 2, 4, 6), (16, 16, 16, 20), (17, 14, 16, 20),
                                                      (64, 64, 64, 24)])
@pytest.mark.parametrize("mode", ["fp64", "fp64tc", "mixed"])
def test_sizes_grow_with_walkers(n_up, n_dn, atoms, per_atom, mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=atoms, n_up=n_up, n_dn=n_dn, per_atom=per_atom, seed=61, side=9.0, Z=2.0)
    W = 4096
    h = pg.jagp_create(sysm, pg.JAGP_PREC_MIXED if mode == "mixed" else pg.JAGP_PREC_FP64, W, None, 0, 0.0, 0,
                       mode == "fp64tc")
    sizes = [pg.jagp_state_bytes]
    if mode != "mixed":
        sizes += [pg.jagp_grad_workspace_bytes, pg.jagp_lrdmc_workspace_bytes, pg.jagp_logpsi_derivs_workspace_bytes]
    for f in sizes:
        b = [f(h, w) for w in range(1, W + 1)]
        assert b[0] > 0 and all(x <= y for x, y in zip(b, b[1:])), f.__name__
    pg.jagp_destroy(h)
