"""Reconfiguration where a comb tooth falls within rounding of the running weight at the edge of a block of walkers
without weight: none of those becomes a parent, and every walker has its share of children to the next integer.  (The
device adds the weights in another order than one after another, so a tooth may fall to either neighbour.)"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1024, 4096, 5000])
def test_walkers_without_weight_have_no_children(W):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_07401_gb300 as pg
    sysm = synth.one_electron_gauss(0.5)
    seed = 9
    g = pg.JAGP(sysm, W, seed=seed)
    r = g.positions(synth.init_walkers(sysm, W, seed=1))
    work = torch.zeros(pg.jagp_lrdmc_workspace_bytes(g.h, W), dtype=torch.uint8, device="cuda")
    eL = torch.zeros(W, dtype=torch.float64, device="cuda")
    rng = np.random.default_rng(W)
    per = -(-W // 1024)
    for case in range(300):
        w = rng.uniform(0.5, 1.5, W)
        z = (float(oracle.philox4x32_10((0, case, 0, 3), (seed, 0))[0]) + 0.5) * 2.0 ** -32
        b = per * int(rng.integers(W // per // 8, W // per // 2))  # walkers b .. b + per - 1 without weight
        w[b:b + per] = 0.0
        X, rest = np.cumsum(w)[b - 1], w[b + per:-1].sum()
        j = round(X * W / w.sum() - z)
        w[b + per:-1] *= (X * W / (j + z) - X - w[-1]) / rest  # (j + z) S / W = X to rounding
        w[-1] = X * W / (j + z) - X - w[b + per:-1].sum()
        assert w[-1] > 0.0
        wd = torch.tensor(w, device="cuda")
        parent, stats = pg.jagp_lrdmc_branch(g.h, r, W, work, wd, eL, generation=case)
        p = parent.cpu().numpy()
        assert np.all(w[p] > 0.0) and np.all(np.diff(p) >= 0)
        share = w * W / w.sum()
        assert np.all(np.abs(np.bincount(p, minlength=W) - share) < 1.0 + 1e-9)
        assert np.array_equal(wd.cpu().numpy(), np.ones(W))
    g.close()
