"""Products with G~^{-1} and of kinetic rows on the tensor cores (FP64-equivalent handles from N_up = 32 on): local
energies and gradients against the handle that uses FP64 instructions.

Tolerance: a product's error is at most K 2^-54 of its largest operands, below FP64's own rounding of such a sum, and the
gradients hold both to the conditioning of G~: 1e-9 of the largest entry, as for gradients against the oracle."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

TOL = 1e-9


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _walkers(sysm, W, seed=5):
    return synth.jitter_walkers(synth.init_walkers(sysm, W, seed=seed), seed + 1, 0.3)


def _close(a, b):
    a, b = a.cpu().numpy(), b.cpu().numpy()
    return np.abs(a - b).max() <= TOL * max(1.0, np.abs(b).max())


# below the rule, at it, odd sizes with unpaired and without down electrons, N_up > 64 (per-walker GEMMs for Gbar),
# L > 512 (7-bit slices of rows), and walkers beyond one chunk of packed operands (L = 320: 351 of columns, 702 of rows)
@pytest.mark.parametrize("n_up,n_dn,atoms,per_atom,W", [(31, 31, 16, 20, 3), (32, 32, 16, 20, 720), (33, 30, 17, 16, 5),
                                                        (40, 0, 20, 6, 3), (64, 64, 32, 20, 4), (67, 65, 34, 6, 3)])
def test_energy_and_gradients(torch_cuda, n_up, n_dn, atoms, per_atom, W):
    torch = torch_cuda
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=atoms, n_up=n_up, n_dn=n_dn, per_atom=per_atom, seed=61, side=8.0, Z=2.0)
    x = _walkers(sysm, W)
    rng = np.random.default_rng(2)
    sl, se = rng.normal(size=W), rng.normal(size=W)
    res = []
    for tc in (False, True):
        g = pg.JAGP(sysm, W, fp64_tc=tc)
        r = g.positions(x)
        g.eval(r)
        e = g.local_energy(r).clone()
        out = g.grad(r, seed_logpsi=torch.tensor(sl, device="cuda"), seed_eL=torch.tensor(se, device="cuda"))
        res.append((e, {k: out[k].clone() for k in ("lam", "jas", "R", "r")}))
        assert g.status() == 0
        g.close()
    assert _close(res[1][0], res[0][0])
    for k in res[0][1]:
        assert _close(res[1][1][k], res[0][1][k]), k


@pytest.mark.parametrize("prec", ["fp64tc", "mixed"])
@pytest.mark.parametrize("n_up", [16, 33])
def test_walker_with_nan_leaves_the_others(torch_cuda, prec, n_up):
    """Slices of numbers that are not finite stay in their walker: the others' bits do not change."""
    torch = torch_cuda
    import paper_2002_07401_gb300 as pg
    sysm = synth.small_random(n_atoms=17, n_up=n_up, n_dn=n_up - 1, per_atom=6, seed=62, side=7.0, Z=2.0)
    W, bad = 5, 2
    x = _walkers(sysm, W)
    y = x.copy()
    y[bad, 3, 1] = np.nan
    keep = [w for w in range(W) if w != bad]
    got = []
    for z in (x, y):
        g = pg.JAGP(sysm, W, precision=pg.JAGP_PREC_MIXED) if prec == "mixed" else pg.JAGP(sysm, W, fp64_tc=True)
        r = g.positions(z)
        la, _ = g.eval(r)
        row = [la.cpu().numpy(), g.local_energy(r).cpu().numpy()]
        if prec == "fp64tc":
            row.append(g.grad(r, seed_eL=torch.ones(W, dtype=torch.float64, device="cuda"))["r"].cpu().numpy())
        got.append(row)
        g.close()
    for a, b in zip(*got):
        assert np.array_equal(a[keep], b[keep])
        assert not np.isfinite(b[bad]).all()
