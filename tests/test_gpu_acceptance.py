"""The acceptance kernels with a CTA per walker (N_up > 32, or a three-body Jastrow at any size) where a walker's last
move of a half-sweep or chunk is rejected after an accepted one: the moves and energies of a sweep follow the oracle's
move by move.  (Positions are equal when every decision is; energies and log|Psi| at the 1e-10 and 1e-9 of the other
trajectory tests.)"""
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


def _close(a, b, tol):
    a, b = np.asarray(a), np.asarray(b)
    return np.all(np.abs(a - b) <= tol * np.maximum(1.0, np.abs(b)))


# G~^{-1} whole in shared memory (33 to 65, and 4 with a three-body Jastrow), partly in global memory (170)
@pytest.mark.parametrize("n_up,refresh,j3", [(33, 0, False), (64, 16, False), (65, 0, False), (65, 13, False),
                                             (170, 0, False), (170, 50, False), (4, 0, True), (40, 16, True)])
def test_last_move_rejected(torch_cuda, n_up, refresh, j3):
    import paper_2002_07401_gb300 as pg
    na = (n_up + 1) // 2 if n_up > 4 else 3
    sysm = synth.small_random(n_atoms=na, n_up=n_up, n_dn=n_up - 1, per_atom=6, seed=210 + n_up,
                              side=3.5 * na ** (1 / 3), Z=2.0)
    if j3:
        sysm = synth.with_j3(sysm, seed=3, sd=0.05)
    W, sweeps = 24 if n_up <= 65 else 6, 2
    x0 = synth.jitter_walkers(synth.init_walkers(sysm, W, seed=6), 7, 0.3)
    g = pg.JAGP(sysm, W, seed=12, refresh_moves=refresh)
    r = g.positions(x0)
    g.eval(r)
    xo, steps = x0.copy(), [x0.copy()]
    for t in range(sweeps):
        eL_ref, lp_ref, _ = oracle.Oracle(sysm).vmc(xo, 1, seed=12, sweep0=t)
        steps.append(xo.copy())
        eL, _ = g.sweep(r, 1, sweep0=t)
        assert np.array_equal(r.cpu().numpy(), xo)
        assert _close(eL.cpu().numpy(), eL_ref, 1e-10)
        assert _close(g.info()["logabs"].cpu().numpy(), lp_ref, 1e-9)
    # the case is there: a last up move rejected after an accepted one
    moved = [(b != a).any(axis=2)[:, :n_up] for a, b in zip(steps, steps[1:])]
    assert any((m[:, :-1].any(axis=1) & ~m[:, -1]).any() for m in moved)
    assert g.status() & (pg.WS_NONFINITE | pg.WS_SINGULAR) == 0
    g.close()
