"""The refresh's elimination at the edges of its forms (a warp's lanes up to N_up
= 32, four warps per walker up to 48 and 64, shared memory above): log|Psi| and
its sign against the oracle at 1e-10, with an odd walker count, and a
singular geminal matrix flagged."""
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


@pytest.mark.parametrize("n_up", [1, 8, 9, 17, 32, 33, 47, 48, 49, 63, 64, 65, 111, 157, 200])
@pytest.mark.parametrize("unpaired", [0, 1])
def test_log_det_and_sign(torch_cuda, n_up, unpaired):
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=max(2, (n_up + 1) // 2), n_up=n_up, n_dn=n_up - unpaired, per_atom=6,
                              seed=40 + n_up, side=2.5 * max(2, (n_up + 1) // 2) ** (1 / 3), Z=2.0)
    W = 7
    x = synth.init_walkers(sysm, W, seed=5)
    g = pg.JAGP(sysm, W)
    la, sg = g.eval(g.positions(x))
    la_ref, sg_ref = oracle.Oracle(sysm).logpsi_batch(x)
    assert g.status() == 0
    assert np.array_equal(sg.cpu().numpy(), sg_ref)
    assert np.allclose(la.cpu().numpy(), la_ref, rtol=1e-10, atol=1e-10)
    g.close()


@pytest.mark.parametrize("n_up", [33, 48, 49, 64, 65, 160])
def test_singular_matrix_is_flagged(torch_cuda, n_up):
    """A walker with a NaN coordinate among sound ones: its bits, and only its, are set."""
    import paper_2002_07401_gb300 as pg
    na = (n_up + 1) // 2
    sysm = synth.small_random(n_atoms=na, n_up=n_up, n_dn=n_up, per_atom=6, seed=70, side=2.5 * na ** (1 / 3), Z=2.0)
    W = 5
    x = synth.init_walkers(sysm, W, seed=5)
    x[3, n_up // 2, 1] = np.nan
    g = pg.JAGP(sysm, W)
    la, sg = g.eval(g.positions(x))
    bits = g.info()["status"].cpu().numpy()
    assert bits[3] == pg.WS_NONFINITE | pg.WS_SINGULAR
    assert np.all(bits[[0, 1, 2, 4]] == 0)
    assert sg.cpu().numpy()[3] == 0.0 and not np.isfinite(la.cpu().numpy()[3])
    g.close()
