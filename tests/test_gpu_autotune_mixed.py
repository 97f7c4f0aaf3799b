"""The mixed path's per-walker products have one kernel per size, so the tuner times each once and reports tile 0, at N_up
below, at and above the refresh's change to the tensor cores (32)."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_up", [4, 16, 31, 32, 40])
def test_tiles_without_effect_are_not_chosen_between(n_up):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=20, n_up=n_up, n_dn=n_up, per_atom=6, seed=33, side=7.0, Z=2.0)
    g = pg.JAGP(sysm, 64, precision=pg.JAGP_PREC_MIXED)
    for _ in range(4):
        t = g.autotune()
        assert t["tile_proposals"] == 0 and t["tile_refresh"] == 0 and all(m > 0 for m in t["ms"])
    g.close()
