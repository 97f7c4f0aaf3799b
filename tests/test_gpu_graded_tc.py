"""FP64-equivalent handles where the geminal matrix is graded: an electron of each spin far from every atom, whose row or
column of G~ is down to 1e-18 of the others' and whose entries of G~^{-1} are as much larger.  Local energies, and gradients
by electrons and nuclei, against the handle that uses FP64 instructions: 1e-9 of a walker's largest entry, as for gradients
elsewhere (the scaling of rows and columns leaves both forms' condition as it is)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("size", [1e-6, 1e-12, 1e-18])
@pytest.mark.parametrize("n_up", [34, 66])
def test_electrons_far_from_the_atoms(torch_cuda, n_up, size):
    torch = torch_cuda
    import paper_2002_07401_gb300 as pg
    na = n_up // 2
    sysm = synth.small_random(n_atoms=na, n_up=n_up, n_dn=n_up - 1, per_atom=16, seed=71, side=3.0 * na ** (1 / 3), Z=2.0)
    W = 4
    x = synth.jitter_walkers(synth.init_walkers(sysm, W, seed=5), 6, 0.3)
    # beyond the atoms by the distance at which the widest Gaussian has that size
    d = np.sqrt(-np.log(size) / sysm.shell_zeta.min())
    x[:, 5] = sysm.R[sysm.R[:, 2].argmax()] + np.array([0.1, 0.2, 1.0]) * d
    x[:, n_up + 7] = sysm.R[sysm.R[:, 0].argmin()] - np.array([1.0, 0.1, 0.2]) * d
    se = torch.ones(W, dtype=torch.float64, device="cuda")
    res = []
    for tc in (False, True):
        g = pg.JAGP(sysm, W, fp64_tc=tc)
        r = g.positions(x)
        g.eval(r)
        e = g.local_energy(r).cpu().numpy()
        out = g.grad(r, seed_eL=se)
        assert g.status() == 0
        res.append([e[:, None], out["r"].cpu().numpy().reshape(W, -1), out["R_walker"].cpu().numpy().reshape(W, -1)])
        g.close()
    for a, b in zip(*res):
        rel = np.abs(b - a).max(axis=1) / np.maximum(1.0, np.abs(a).max(axis=1))
        assert np.all(rel <= 1e-9), rel
