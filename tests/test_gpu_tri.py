"""The tensor-core product over the full triangle of slice pairs at the edges of
its tiles (128 rows; 16 to 80 columns per CTA, one or two CTAs per cluster; K
chunks of 16 and 32), and a pairing matrix with zero blocks, whose K ranges
the product skips."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

PAIRS = [(a, d - a) for d in range(6) for a in range(d + 1)]


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("M,N,Kp,live", [(1, 1, 64, None), (127, 16, 64, None), (128, 17, 128, None),
                                         (129, 80, 64, None), (385, 81, 192, 257), (640, 160, 64, 0),
                                         (255, 161, 128, 128), (20000, 48, 64, None), (300, 333, 1024, 299)])
def test_triangle_of_integer_slices(torch_cuda, M, N, Kp, live):
    """Integer slices: every accumulator is exact, so the FP32 result is the
    exact sum to one rounding (the low part is dropped): 2^-23 relative."""
    torch = torch_cuda
    import paper_2002_07401_gb300 as pg
    g = torch.Generator(device="cuda").manual_seed(M + 7 * N + Kp)
    A = torch.randint(-128, 129, (M, 6 * Kp), device="cuda", generator=g)
    B = torch.randint(-128, 129, (N, 6 * Kp), device="cuda", generator=g)
    ea = torch.randint(-9, 10, (M,), device="cuda", generator=g, dtype=torch.int32)
    eb = torch.randint(-9, 10, (N,), device="cuda", generator=g, dtype=torch.int32)
    C = torch.full((M + 1, N), 7.0, dtype=torch.float32, device="cuda")
    count = None if live is None else torch.tensor([live], dtype=torch.int32, device="cuda")
    err = pg.jagp_gemm_bf16x(A.to(torch.bfloat16), 6, B.to(torch.bfloat16), 6, Kp, PAIRS, C, count=count, row_exp=ea,
                             col_exp=eb)
    # A has M rows, C one more: neither it nor rows past the live count are written
    rows = M if live is None else live
    ref = torch.zeros((M, N), dtype=torch.float64, device="cuda")
    for a, b in PAIRS:
        ref += (A[:, a * Kp:(a + 1) * Kp].double() @ B[:, b * Kp:(b + 1) * Kp].double().T) * 256.0 ** -(a + b)
    ref *= torch.pow(2.0, (ea[:, None] + eb[None] - 14).double())
    assert int(err.item()) == 0
    d = (C[:rows].double() - ref[:rows]).abs()
    assert torch.all(d <= 2.0 ** -23 * ref[:rows].abs()), float(d.max()) if rows else 0.0
    assert torch.all(C[rows:] == 7.0)


@pytest.mark.parametrize("mode", ["fp64tc", "mixed"])
@pytest.mark.parametrize("per_atom,n_atoms", [(6, 9), (24, 14)])
def test_zero_blocks_of_lambda(torch_cuda, mode, per_atom, n_atoms):
    """lambda with a band, an empty block of rows and columns and a far corner
    block: log|Psi| and e_L against the oracle (FP64-equivalent 1e-10, mixed
    1e-6 and 1e-5 Ha)."""
    import paper_2002_07401_gb300 as pg
    torch = torch_cuda
    sysm = synth.small_random(n_atoms=n_atoms, n_up=7, n_dn=6, per_atom=per_atom, seed=21, side=5.0, Z=2.0)
    L = sysm.L
    i, j = np.indices((L, L))
    lam = np.where(np.abs(i - j) <= L // 10, sysm.lam, 0.0)
    lam[L // 2:L // 2 + 33, :] = 0.0
    lam[:, L // 2:L // 2 + 33] = 0.0
    lam[:5, L - 7:] = 0.3
    lam[L - 7:, :5] = 0.3
    sysm.lam = lam
    W = 12
    x = synth.init_walkers(sysm, W, seed=3)
    fp64 = mode == "fp64tc"
    g = pg.JAGP(sysm, W, precision=pg.JAGP_PREC_FP64 if fp64 else pg.JAGP_PREC_MIXED, fp64_tc=fp64)
    r = g.positions(x)
    la, sg = g.eval(r)
    eL = g.local_energy(r)
    torch.cuda.synchronize()
    o = oracle.Oracle(sysm)
    la_ref, sg_ref = o.logpsi_batch(x)
    eL_ref = o.local_energy_batch(x)
    assert g.status() == 0
    assert np.array_equal(sg.cpu().numpy(), sg_ref)
    tol, etol = (1e-10, 1e-10) if fp64 else (1e-6, 0.0)
    assert np.allclose(la.cpu().numpy(), la_ref, rtol=tol if fp64 else 0.0, atol=tol)
    assert np.allclose(eL.cpu().numpy(), eL_ref, rtol=etol, atol=1e-10 if fp64 else 1e-5)
    g.close()
